"""Calls that follow one another on a stream without a wait between them: each reads what the one before it wrote and
overwrites what the one before it read, so that a kernel which touches memory before the previous one has ended would
show.  Eagerly, on a stream of its own and replayed from a captured graph, against the same calls with a
synchronisation after each."""
import pytest

from paper_2604_05250_b200 import synth
from tests._parity import takes_the_streaming_kernel, to_torch_bf16

pytestmark = pytest.mark.gpu
TRUST, KL, CONF = 0, 1, 2


@pytest.fixture(scope="module")
def dd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_05250_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def attention_chain(dd, B, H, N, D, Nq=None, ragged=False):
    """Output of one call = the values of the next, in two buffers taken in turn; of a block of queries, = the next one's
    queries."""
    import torch
    q, k, v = (to_torch_bf16(x, "cuda") for x in synth.attention_inputs(B, H, N, D, N + D))
    first = v.clone()
    other = torch.empty_like(v)
    block = part = None
    if Nq is not None:
        block, part = q[:, :, :Nq].contiguous(), torch.empty_like(q[:, :, :Nq].contiguous())
    lens = torch.tensor([max(1, N - 7 * b) for b in range(B)], dtype=torch.int32, device="cuda") if ragged else None

    def run(after):
        v.copy_(first)
        if Nq is not None:
            block.copy_(q[:, :, :Nq])
            other.copy_(first)
        a, b = v, other
        for _ in range(6):
            if Nq is None:
                dd.bidir_attention(q, k, a, out=b)
            else:
                dd.block_attention(block, k, a, kv_len=lens, out=part)
                dd.block_attention(part, k, a, kv_len=lens, out=block)
            after()
            a, b = b, a
        return [x.clone() for x in ((a, b) if Nq is None else (block, part))]
    return run


def verify_chain(dd, B, P, V, mode, K=None):
    """The tokens and flags of one call are the next one's, in two sets of buffers taken in turn."""
    import torch
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, "all", 0.2, P + V)
    dra, ver = (to_torch_bf16(x, "cuda") for x in (dra, ver))
    dh = dw = vh = vw = None
    if K:
        dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(B, P, K, V, "all", 0.2, seed=P + V)
        dh, dw, vh, vw = (to_torch_bf16(x, "cuda") for x in (dh, dw, vh, vw))
        if mode != KL:
            dh = dw = None
    start = [torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()]
    sets = [[torch.empty_like(x) for x in start] for _ in range(2)]
    score = torch.empty(B, P, device="cuda")

    def run(after):
        for x, y in zip(sets[0], start):
            x.copy_(y)
        a, b = sets
        for i in range(6):
            if K:
                dd.lm_head_verify(dh, dw, vh, vw, a[0], a[1], mode, 0.3, P // 8, i, b[0], b[1], score)
            else:
                dd.verify(dra if mode == KL else None, ver, a[0], a[1], mode, 0.3, P // 8, i, b[0], b[1], score)
            after()
            a, b = b, a
        return [x.clone() for x in a + b] + [score.clone()]
    return run


def mixed_chain(dd):
    """Every kind of kernel behind every other: the flags that one call leaves are the next one's, the hidden states of a fused head
    are what attention has just written.  fork: attention on a stream of its own beside the verification, joined before the head."""
    import torch
    B, P, H, D = 3, 300, 16, 128
    gen = torch.Generator(device="cuda").manual_seed(1)
    bf16 = lambda *shape, scale=1.0: torch.randn(shape, device="cuda", generator=gen).mul_(scale).to(torch.bfloat16)
    off = torch.zeros(2, B * P * 1003 + 8, dtype=torch.bfloat16, device="cuda")
    off.copy_(bf16(*off.shape, scale=2.0))
    off = [x[3:3 + B * P * 1003].view(B, P, 1003) for x in off]                    # not on 16-byte boundaries
    mapped, streamed, deep = [bf16(B, P, 24576, scale=2.0) for _ in "dv"], bf16(B, P, 65000, scale=2.0), [bf16(1, P, 126464, scale=2.0) for _ in "dv"]
    assert takes_the_streaming_kernel(B, P, 65000, False) and not takes_the_streaming_kernel(B, P, 24576, True)
    q0, k, v = (bf16(B, H, P, D) for _ in "qkv")
    q, out = torch.empty_like(q0), torch.empty_like(q0)
    hidden, w_wide = out.view(B, P, H * D), bf16(6500, H * D, scale=0.1)           # pairs of CTAs
    dh, vh, dw, vw = bf16(B, P, 64), bf16(B, P, 64), bf16(40000, 64, scale=0.2), bf16(40000, 64, scale=0.2)
    tok = torch.zeros(B, P, dtype=torch.int32, device="cuda")
    x = [torch.empty(B, P, dtype=torch.uint8, device="cuda") for _ in range(6)]
    t = [torch.empty_like(tok) for _ in range(6)]
    score = torch.empty(B, P, device="cuda")
    side = torch.cuda.Stream()

    def run(after, fork=False):
        q.copy_(q0)
        x[0].fill_(1)
        kept = []
        for i in range(3):
            def attend():
                dd.bidir_attention(q, k, v, out=out)
                after()
                dd.block_attention(out[:, :, :32].contiguous(), k, v, out=q[:, :, :32].contiguous())
            main = torch.cuda.current_stream()
            if fork:
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    attend()
            else:
                attend()
                after()
            dd.verify(*mapped, tok, x[0], KL, 0.3, 20, i, t[1], x[1], score)
            after()
            dd.verify(None, streamed, t[1], x[1], CONF | 0x100, 0.3, 20, i, t[2], x[2], score)
            after()
            if fork:
                main.wait_stream(side)
            dd.lm_head_verify(None, None, hidden, w_wide, t[2], x[2], CONF, 0.5, 30, i, t[3], x[3], score)
            after()
            dd.verify(*off, t[3], x[3], KL, 0.3, 30, i, t[4], x[4], score)
            after()
            dd.lm_head_verify(dh, dw, vh, vw, t[4], x[4], KL, 0.01, 30 + 60 * i, i, t[5], x[5], score)
            after()
            dd.verify(*deep, t[5][:1], x[5][:1], KL, 0.3, 20, i, t[0][:1], x[0][:1], score[:1])
            after()
            q.copy_(out)
            kept += [y.clone() for y in (*x, *t[1:], score, out)]
        return kept
    return run


@pytest.mark.parametrize("chain,args", [
    (attention_chain, (1, 4, 128, 64)), (attention_chain, (1, 32, 1024, 128)), (attention_chain, (4, 32, 512, 64)),
    (attention_chain, (2, 4, 1000, 128, 32, True)), (attention_chain, (2, 2, 300, 64, 200)),
    (verify_chain, (1, 128, 1024, KL)), (verify_chain, (4, 256, 8000, KL)), (verify_chain, (4, 300, 4001, CONF)),
    (verify_chain, (2, 100, 1000, KL, 256)), (verify_chain, (1, 256, 4000, CONF, 512)),
    # persistent attention, D = 128; long rows: clusters, deep, flagged rows first; heads: rows listed and gathered, the kernel chosen on the
    # device, pairs without the drafter
    (attention_chain, (2, 80, 300, 128)), (verify_chain, (1, 40, 65003, KL)), (verify_chain, (2, 140, 126464, KL)),
    (verify_chain, (1, 700, 40000, KL, 128)), (verify_chain, (1, 600, 6500, CONF, 2048)), (mixed_chain, ()),
])
def test_back_to_back(dd, chain, args):
    import torch
    run = chain(dd, *args)
    want = run(torch.cuda.synchronize)

    def check(got):
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        assert dd.attention_status() == 0 and dd.verify_status() == 0
    check(run(lambda: None))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        got = run(lambda: None)
    check(got)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = run(lambda: None)
    for _ in range(3):
        graph.replay()
    check(got)
    if chain is mixed_chain:
        forked = torch.cuda.CUDAGraph()
        with torch.cuda.graph(forked):
            got = run(lambda: None, fork=True)
        for _ in range(3):
            forked.replay()
        check(got)

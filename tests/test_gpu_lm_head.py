"""dd_lm_head_verify on the GPU against the CPU oracle (fp64 head, then the verification algorithm
on the unrounded logits), through the C ABI."""
import numpy as np
import pytest

from paper_2604_05250_b200 import synth
from tests._parity import Guarded, check_verify, to_torch_bf16

pytestmark = pytest.mark.gpu

TRUST, KL, CONF, PROB, EMIT = 0, 1, 2, 0x100, 0x200
# The kernel accumulates the bf16 products in fp32 where the oracle uses fp64: a verifier token is
# only comparable where the two largest logits are further apart than that can blur.
TOP2_GAP = 1e-3
# KL scores (Eq. 4-5) are differences of quantities of size |logit| ~ 10: the fp32 accumulation of
# K bf16 products leaves each logit within about sqrt(K) * 2^-24 * |logit| ~ 4e-5 (K = 4096) of the
# oracle's fp64 value, and the score inherits an error of that size whatever its own magnitude.
KL_SCORE_ABS = 1e-4


@pytest.fixture(scope="module")
def dd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_05250_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def compare(dd, oracle_mod, hidden, weight, tokens, flags, mode, tau, k, seed, drafter=(None, None)):
    import torch
    B, P, K = hidden.shape
    ref = oracle_mod.lm_head_verify(drafter[0], drafter[1], hidden, weight, tokens, flags, mode, tau, k, seed)
    g_tok, g_mask, g_score = (Guarded((B, P), dt) for dt in (torch.int32, torch.uint8, torch.float32))
    t_dra = [None if x is None else to_torch_bf16(x, "cuda") for x in drafter]
    ot, om, osc = dd.lm_head_verify(t_dra[0], t_dra[1], to_torch_bf16(hidden, "cuda"), to_torch_bf16(weight, "cuda"),
                                    torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda(),
                                    mode, tau, k, seed, out_tokens=g_tok.view, out_mask=g_mask.view, out_score=g_score.view)
    torch.cuda.synchronize()
    assert dd.verify_status() == 0
    g_tok.check("out_tokens"); g_mask.check("out_mask"); g_score.check("out_score")
    ot, om, osc = ot.cpu().numpy(), om.cpu().numpy(), osc.cpu().numpy()
    # where the verifier's two best tokens are closer than fp32 accumulation resolves, either is right
    close = (ref["top2_gap"] <= TOP2_GAP) & flags.astype(bool) & (om == 0) & (ref["out_mask"] == 0)
    ref = dict(ref)
    ref["out_tokens"] = np.where(close, ot, ref["out_tokens"])
    n_exempt = check_verify(ot, om, osc, ref, flags, tokens,
                            **(dict(score_abs=KL_SCORE_ABS) if (mode & 0xFF) == KL else {}))
    return ref, (ot, om, osc), int(close.sum()), n_exempt


@pytest.mark.parametrize("B,P,K,V,flagged", [
    (1, 40, 128, 1000, 25),            # one row block, rows and vocabulary both ragged
    (2, 70, 256, 4100, 51),            # rows of two sequences share a 128-row tile
    (1, 300, 64, 8232, 300),           # two row blocks, a single k-step
    (3, 128, 512, 2048, "uniform_25_100"),
    (1, 1, 64, 8, 1),
])
@pytest.mark.parametrize("mode", [TRUST, CONF, CONF | PROB])
def test_small_shapes(dd, oracle_mod, B, P, K, V, flagged, mode):
    hidden, weight, tokens, flags = synth.lm_head_inputs(B, P, K, V, flagged, seed=B * 1000 + P)
    compare(dd, oracle_mod, hidden, weight, tokens, flags, mode, 0.05, 3, 7)


@pytest.mark.parametrize("B,P,K,V,flagged", [
    (1, 40, 128, 1000, 25),
    (2, 70, 256, 4100, 51),
    (1, 300, 64, 8232, 300),
    (3, 128, 512, 2048, "uniform_25_100"),
    (1, 1, 64, 8, 1),
])
@pytest.mark.parametrize("mode", [KL, KL | PROB, KL | EMIT])
def test_small_shapes_kl(dd, oracle_mod, B, P, K, V, flagged, mode):
    """Eq. 4-5 from both models' hidden states: two products per work item, one epilogue."""
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(B, P, K, V, flagged, 0.2, seed=B * 1000 + P)
    ref, got, _, _ = compare(dd, oracle_mod, vh, vw, tokens, flags, mode, 0.5, 3, 7, drafter=(dh, dw))
    if P >= 40:        # the scores are those of two different distributions, and both outcomes occur
        fl = flags.astype(bool)
        assert (ref["out_score"][fl] > 1e-3).all()
        if not mode & PROB:
            assert ref["out_mask"][fl].any() and not ref["out_mask"][fl].all()


@pytest.mark.parametrize("P,K,V,flagged", [
    (129, 64, 8, 129),                 # one row in the second CTA of a pair; one tile, its neighbour beyond the vocabulary
    (256, 128, 321, 256),              # whole blocks of rows; an odd number of tiles
    (257, 192, 256, 257),              # a second block of one row
    (600, 256, 20011, 130),            # the flagged rows gathered, in one block
    (700, 128, 40000, 390),            # and in two
])
def test_pairs_of_ctas(dd, oracle_mod, P, K, V, flagged):
    """The KL mode beyond 128 rows: 256 rows by two tiles of the vocabulary per pair of CTAs."""
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(1, P, K, V, flagged, 0.2, seed=P)
    compare(dd, oracle_mod, vh, vw, tokens, flags, KL, 0.5, 9, 3, drafter=(dh, dw))


@pytest.mark.parametrize("P,K,V,flagged", [
    (129, 2048, 19000, 129),           # one block of rows, two tiles of the vocabulary at a time; an odd number of tiles
    (513, 2048, 6500, 513),            # 512 rows a tile at a time, one row two tiles at a time
    (300, 2112, 9500, 300),            # 512 rows that are not all there
    (1000, 2048, 6500, 200),           # the flagged rows gathered
    (70, 1088, 1100, 70),              # not in pairs: tiles narrower than 128, to have more of them
])
def test_pairs_of_ctas_verifier_only(dd, oracle_mod, P, K, V, flagged):
    """The other modes in pairs, and the narrow tiles of problems with few items."""
    hidden, weight, tokens, flags = synth.lm_head_inputs(1, P, K, V, flagged, seed=P)
    compare(dd, oracle_mod, hidden, weight, tokens, flags, CONF | PROB, 0.05, 9, 11)


@pytest.mark.parametrize("mode,K", [(KL, 64), (CONF, 2048)])
@pytest.mark.parametrize("P,flagged", [(300, [128]), (300, [129]), (129, [0, 1, 129]), (520, [520, 1])])
def test_kernel_chosen_on_the_device(dd, mode, K, P, flagged):
    """Vocabularies of more than 37888 entries (148 SMs): up to 128 flagged rows by single CTAs, more in pairs, one call after the other.  A row's result does
    not depend on the other rows' flags, nor on which kernel multiplied it."""
    import torch
    V = 38000
    gen = torch.Generator(device="cuda").manual_seed(P)
    vh, vw, dh, dw = (torch.randn(n, K, device="cuda", generator=gen).mul_(s).to(torch.bfloat16)
                      for n, s in ((P, 1.0), (V, 2.0 / K ** 0.5), (P, 1.0), (V, 2.0 / K ** 0.5)))
    vh, dh = vh[None], dh[None]
    d = (dh, dw) if mode == KL else (None, None)
    tok = torch.zeros(1, P, dtype=torch.int32, device="cuda")
    logits = vh[0].double() @ vw.double().T
    lv = torch.log_softmax(logits, -1)
    if mode == KL:
        ld = torch.log_softmax(dh[0].double() @ dw.double().T, -1)
        want = (ld.exp() * (ld - lv)).sum(-1)
    else:
        want = lv.max(-1).values.exp()
    top = logits.topk(2, -1)
    clear = top.values[:, 0] - top.values[:, 1] > TOP2_GAP
    for n in flagged:
        on = torch.randperm(P, device="cuda", generator=gen) < n
        got = dd.lm_head_verify(*d, vh, vw, tok, on[None].to(torch.uint8), mode, 1e9 if mode == KL else 0.0, 0, 0)
        assert dd.verify_status() == 0
        tol = KL_SCORE_ABS if mode == KL else 1e-4 * want.max().item()
        assert (got[2][0].double() - want)[on].abs().max().item() <= tol if n else not got[2].any()
        assert torch.equal(got[0][0][on & clear], top.indices[:, 0].int()[on & clear]) and not got[0][0][~on].any() and not got[1].any()


@pytest.mark.parametrize("P", [700, 1100, 2100])
def test_long_sequences(dd, oracle_mod, P):
    """Sequences longer than the register-resident decision stage holds (512 positions), longer
    than the general form keeps in registers (1024), and longer than the fold kernel's key area in
    shared memory (2048)."""
    hidden, weight, tokens, flags = synth.lm_head_inputs(2, P, 64, 520, "uniform_25_100", seed=P)
    compare(dd, oracle_mod, hidden, weight, tokens, flags, CONF | PROB, 0.05, 9, 11)
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(2, P, 64, 520, "uniform_25_100", 0.2, seed=P + 1)
    compare(dd, oracle_mod, vh, vw, tokens, flags, KL, 0.5, 9, 11, drafter=(dh, dw))


def test_kl_tells_the_two_models_apart(dd, oracle_mod):
    """The drafter's pair and the verifier's pair swapped: D_KL(p_V || p_D) is another number."""
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(1, 64, 128, 2000, 64, 0.2, seed=5)
    a, _, _, _ = compare(dd, oracle_mod, vh, vw, tokens, flags, KL, 0.5, 0, 0, drafter=(dh, dw))
    b, _, _, _ = compare(dd, oracle_mod, dh, dw, tokens, flags, KL, 0.5, 0, 0, drafter=(vh, vw))
    assert (np.abs(a["out_score"] - b["out_score"]) > 1e-3).sum() > 32
    # and a drafter equal to the verifier scores zero everywhere
    import torch
    t = [to_torch_bf16(x, "cuda") for x in (vh, vw)]
    out = dd.lm_head_verify(t[0], t[1], t[0], t[1], torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda(),
                            KL, 0.5, 0, 0)
    assert float(out[2].abs().max()) <= 1e-6 and int(out[1].sum()) == 0


def test_matches_the_unfused_path(dd, oracle_mod):
    """Logits by the oracle's head, rounded to bf16, through dd_verify: the same decisions wherever
    the confidence is far from the threshold (the two paths differ by the rounding of the logits)."""
    import torch
    B, P, K, V = 1, 64, 256, 4096
    hidden, weight, tokens, flags = synth.lm_head_inputs(B, P, K, V, 64, seed=9)
    logits = oracle_mod.lm_head(hidden.reshape(P, K), weight)
    bits = synth.f32_to_bf16_bits(logits.astype(np.float32)).reshape(B, P, V)
    a = dd.lm_head_verify(None, None, to_torch_bf16(hidden, "cuda"), to_torch_bf16(weight, "cuda"), torch.from_numpy(tokens).cuda(),
                          torch.from_numpy(flags).cuda(), CONF, 0.05, 0, 0)
    b = dd.verify(None, to_torch_bf16(bits, "cuda"), torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda(),
                  CONF, 0.05, 0, 0)
    torch.cuda.synchronize()
    sa, sb = a[2].cpu().numpy(), b[2].cpu().numpy()
    assert np.abs(sa - sb).max() <= 2e-2 * sb.max()
    far = np.abs(sb - 0.05) > 5e-3
    assert far.sum() > P // 2 and (a[1].cpu().numpy()[far] == b[1].cpu().numpy()[far]).all()


def test_llada_shaped_full_size(dd, oracle_mod):
    """cfg1's verification step from hidden states: 256 positions, K = 4096, V = 126464."""
    hidden, weight, tokens, flags = synth.lm_head_inputs(1, 256, 4096, 126464, "all", seed=1000)
    ref, got, n_close, _ = compare(dd, oracle_mod, hidden, weight, tokens, flags, CONF, 0.5, 32, 0)
    assert n_close <= 8
    kept = (flags.astype(bool) & ~ref["out_mask"].astype(bool)).sum()
    assert kept >= 32


def test_llada_shaped_full_size_kl(dd, oracle_mod):
    """The same step in the KL mode: both heads at K = 4096, V = 126464."""
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(1, 256, 4096, 126464, "all", 0.2, seed=1001)
    ref, got, _, _ = compare(dd, oracle_mod, vh, vw, tokens, flags, KL, 0.5, 32, 0, drafter=(dh, dw))
    rejected = int(ref["out_mask"].sum())
    assert 20 <= rejected <= 120


@pytest.mark.parametrize("n", [0, 1, 127, 128, 129, 256, 257, 384, 385])
def test_flagged_rows_at_the_edges_of_tiles(dd, oracle_mod, n):
    """Flagged rows gathered into fewer 128-row tiles (n <= 384 of 400 rows), or left where they are
    (385); the last item of a vocabulary tile with one or two tiles of rows, the first one with none.
    Every unflagged hidden state is NaN: none may reach a result."""
    rng = np.random.default_rng(n)
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(2, 200, 128, 1500, "all", 0.2, seed=77)
    flags[:] = 0
    flags.reshape(-1)[rng.choice(400, size=n, replace=False)] = 1
    clean_v, clean_d = vh.copy(), dh.copy()
    vh[flags == 0] = dh[flags == 0] = 0x7FC0
    for mode, drafter in ((CONF, False), (KL, True)):
        import torch
        ref = oracle_mod.lm_head_verify(clean_d if drafter else None, dw if drafter else None, clean_v, vw, tokens, flags, mode, 0.05, 5, 1)
        on = lambda x: to_torch_bf16(x, "cuda")
        got = dd.lm_head_verify(on(dh) if drafter else None, on(dw) if drafter else None, on(vh), on(vw),
                                torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda(), mode, 0.05, 5, 1)
        torch.cuda.synchronize()
        assert dd.verify_status() == 0
        ot, om, osc = (x.cpu().numpy() for x in got)
        close = (ref["top2_gap"] <= TOP2_GAP) & flags.astype(bool) & (om == 0) & (ref["out_mask"] == 0)
        ref = dict(ref, out_tokens=np.where(close, ot, ref["out_tokens"]))
        check_verify(ot, om, osc, ref, flags, tokens, **(dict(score_abs=KL_SCORE_ABS) if drafter else {}))


def test_results_do_not_depend_on_the_grid(dd, oracle_mod):
    import torch
    hidden, weight, tokens, flags = synth.lm_head_inputs(2, 150, 128, 3000, 97, seed=12)
    dh, dw, _, _, _, _ = synth.lm_head_pair_inputs(2, 150, 128, 3000, 97, 0.2, seed=12)
    tail = (to_torch_bf16(hidden, "cuda"), to_torch_bf16(weight, "cuda"), torch.from_numpy(tokens).cuda(),
            torch.from_numpy(flags).cuda())
    for args in ((None, None) + tail + (CONF | PROB, 0.05, 4, 3),
                 (to_torch_bf16(dh, "cuda"), to_torch_bf16(dw, "cuda")) + tail + (KL | PROB, 0.5, 4, 3)):
        try:
            ref = [x.cpu().numpy() for x in dd.lm_head_verify(*args)]
            for cap in (1, 5, 37):
                dd.debug_set_max_ctas(cap)
                got = [x.cpu().numpy() for x in dd.lm_head_verify(*args)]
                for a, b in zip(ref, got):
                    assert np.array_equal(a, b), f"cap {cap}"
        finally:
            dd.debug_set_max_ctas(0)


def test_argument_errors(dd):
    import torch
    h = torch.zeros(1, 4, 64, dtype=torch.bfloat16, device="cuda")
    w = torch.zeros(16, 64, dtype=torch.bfloat16, device="cuda")
    t = torch.zeros(1, 4, dtype=torch.int32, device="cuda")
    f = torch.ones(1, 4, dtype=torch.uint8, device="cuda")
    o = torch.zeros(1, 4, dtype=torch.float32, device="cuda")
    L, p = dd.lib(), (lambda x: x.data_ptr())
    call = lambda mode, K: L.dd_lm_head_verify(None, None, p(h), p(w), p(t), p(f), mode, 0.5, 0, 0, p(t), p(f), p(o), 1, 4, K, 16, None)
    assert call(KL, 64) == dd.DD_ERR_INVALID_ARG           # the KL mode needs the drafter's pair
    assert L.dd_lm_head_verify(p(h), None, p(h), p(w), p(t), p(f), KL, 0.5, 0, 0, p(t), p(f), p(o), 1, 4, 64, 16, None) == dd.DD_ERR_INVALID_ARG
    assert L.dd_lm_head_verify(p(h) + 2, p(w), p(h), p(w), p(t), p(f), KL, 0.5, 0, 0, p(t), p(f), p(o), 1, 4, 64, 16, None) == dd.DD_ERR_UNSUPPORTED
    assert call(CONF, 48) == dd.DD_ERR_UNSUPPORTED
    assert call(CONF, 0) == dd.DD_ERR_INVALID_ARG
    assert call(7, 64) == dd.DD_ERR_INVALID_ARG
    assert L.dd_lm_head_verify(None, None, None, p(w), p(t), p(f), CONF, 0.5, 0, 0, p(t), p(f), p(o), 1, 4, 64, 16, None) == dd.DD_ERR_INVALID_ARG


def test_without_room_for_the_gathered_rows(dd):
    """Little free memory: no copy of the hidden states is made, every row is multiplied, the results are the same, no
    call allocates or waits (one can be captured), and the copy is made again once there is room."""
    import torch
    dd.release()
    B, P, K, V = 24, 2048, 4096, 500
    g = torch.Generator(device="cuda").manual_seed(3)
    hidden = torch.randn(B, P, K, device="cuda", generator=g, dtype=torch.bfloat16)           # 403 MB
    weight = torch.randn(V, K, device="cuda", generator=g).mul_(K ** -0.5).to(torch.bfloat16)
    tok = torch.zeros(B, P, dtype=torch.int32, device="cuda")
    fl = (torch.rand(B, P, device="cuda", generator=g) < 0.3).to(torch.uint8)
    outs = dict(out_tokens=torch.empty_like(tok), out_mask=torch.empty_like(fl), out_score=torch.empty(B, P, device="cuda"))
    call = lambda: [x.clone() for x in dd.lm_head_verify(None, None, hidden, weight, tok, fl, CONF, 0.0, 0, 0, **outs)]
    free = lambda: torch.cuda.mem_get_info()[0]

    def same(a, b):
        # the products are the same numbers; sums over tiles of another width differ in their order only
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
        torch.testing.assert_close(a[2], b[2], rtol=1e-5, atol=0)
    roomy = call()
    torch.cuda.synchronize()
    dd.release()
    torch.cuda.empty_cache()
    filler = torch.empty(free() - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        first = call()
        torch.cuda.synchronize()
        before = free()
        same(call(), roomy)
        same(first, roomy)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            dd.lm_head_verify(None, None, hidden, weight, tok, fl, CONF, 0.0, 0, 0, **outs)
        outs["out_score"].fill_(-1.0)
        graph.replay()
        torch.cuda.synchronize()
        same([outs["out_tokens"], outs["out_mask"], outs["out_score"]], roomy)
        assert before - free() < hidden.numel()                  # (less than half of the copy)
    finally:
        del filler
        torch.cuda.empty_cache()
    before = free()
    same(call(), roomy)
    torch.cuda.synchronize()
    assert before - free() >= hidden.numel() * 2
    assert dd.verify_status() == 0


def test_captured_with_the_scratch_of_a_smaller_call(dd):
    """A call whose narrowest tiles need more scratch than there is, first seen under capture: wider tiles, as nothing may be allocated."""
    import torch
    P, V = 100, 2000
    gen = torch.Generator(device="cuda").manual_seed(4)
    tok, fl = torch.zeros(1, P, dtype=torch.int32, device="cuda"), torch.ones(1, P, dtype=torch.uint8, device="cuda")

    def arguments(K):
        h, w = (torch.randn(n, K, device="cuda", generator=gen).mul_(s).to(torch.bfloat16) for n, s in ((P, 1.0), (V, 2.0 / K ** 0.5)))
        return None, None, h[None], w, tok, fl, CONF, 0.0, 0, 0
    small, large = arguments(128), arguments(1024)
    outs = dict(out_tokens=torch.empty_like(tok), out_mask=torch.empty_like(fl), out_score=torch.empty(1, P, device="cuda"))
    dd.release()
    dd.lm_head_verify(*small)                    # 32 tiles of 64 entries; the larger one would like 63 of 32
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dd.lm_head_verify(*large, **outs)
    graph.replay()
    torch.cuda.synchronize()
    got = [outs[x].clone() for x in ("out_tokens", "out_mask", "out_score")]
    del graph
    want = dd.lm_head_verify(*large)             # now there is room
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    torch.testing.assert_close(got[2], want[2], rtol=1e-5, atol=0)
    assert dd.verify_status() == 0


# Rows gathered or not: nothing flagged where rows are not listed; many rows (more than one for a warp of the listing
# kernel) with two tiles of the vocabulary, where few and where most of them are flagged, and with three.
@pytest.mark.parametrize("B,P,K,V,share", [(1, 20, 128, 1000, 0.0), (2, 500, 64, 300, 0.0), (3, 8000, 64, 300, 0.15),
                                           (3, 8000, 64, 300, 0.8), (3, 8000, 64, 700, 0.3)])
@pytest.mark.parametrize("mode", [CONF, KL])
def test_rows_gathered_or_not(dd, oracle_mod, B, P, K, V, share, mode):
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(B, P, K, V, "all", 0.2, seed=P + V)
    flags[:] = np.random.default_rng(P).random((B, P)) < share
    compare(dd, oracle_mod, vh, vw, tokens, flags, mode, 0.3, 5, 1, drafter=(dh, dw) if mode == KL else (None, None))

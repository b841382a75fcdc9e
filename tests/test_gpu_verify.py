"""dd_verify on the GPU against the CPU oracle, through the C ABI."""
import numpy as np
import pytest

from paper_2604_05250_b200 import synth
from tests._parity import Guarded, check_verify, off_vector_boundary, takes_the_streaming_kernel, to_torch_bf16

pytestmark = pytest.mark.gpu

TRUST, KL, CONF = 0, 1, 2
PROB, EMIT = 0x100, 0x200


@pytest.fixture(scope="module")
def dd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_05250_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def run_gpu(dd, dra, ver, tokens, flags, mode, tau, k, seed, host=False, off=False):
    """off: logits off 16-byte boundaries, which take the element-wise kernel."""
    import torch
    dev = None if host else "cuda"
    logits = off_vector_boundary if off else (lambda bits: to_torch_bf16(bits, dev, pin=host))
    t_ver = logits(ver)
    t_dra = None if dra is None else logits(dra)
    t_tok = torch.from_numpy(tokens)
    t_fl = torch.from_numpy(flags)
    if host:
        t_tok, t_fl = t_tok.pin_memory(), t_fl.pin_memory()
    else:
        t_tok, t_fl = t_tok.cuda(), t_fl.cuda()
    # each output sits between two guard regions that the kernels must leave alone
    g_tok = Guarded(tokens.shape, torch.int32, device=dev, pin=host)
    g_mask = Guarded(tokens.shape, torch.uint8, device=dev, pin=host)
    g_score = Guarded(tokens.shape, torch.float32, device=dev, pin=host)
    ot, om, osc = dd.verify(t_dra, t_ver, t_tok, t_fl, mode, tau, k, seed, out_tokens=g_tok.view,
                            out_mask=g_mask.view, out_score=g_score.view, host=host)
    torch.cuda.synchronize()
    assert dd.verify_status() == 0
    g_tok.check("out_tokens"); g_mask.check("out_mask"); g_score.check("out_score")
    return ot.cpu().numpy(), om.cpu().numpy(), osc.cpu().numpy()


def compare(dd, oracle_mod, dra, ver, tokens, flags, mode, tau, k, seed, host=False, off=False):
    algo = mode & 0xFF
    d_in = dra if algo == KL else None
    ref = oracle_mod.verify(d_in, ver, tokens, flags, mode, tau, k, seed)
    ot, om, osc = run_gpu(dd, d_in, ver, tokens, flags, mode, tau, k, seed, host=host, off=off)
    return check_verify(ot, om, osc, ref, flags, tokens), ref, (ot, om, osc)


ALL_MODES = [TRUST, KL, CONF, KL | PROB, CONF | PROB, KL | EMIT, TRUST | EMIT, CONF | PROB | EMIT]


@pytest.mark.parametrize("mode", ALL_MODES)
def test_config0_tiny(dd, oracle_mod, mode):
    c = synth.VERIFY_CONFIGS[0]
    dra, ver, tokens, flags = synth.verify_config_inputs(0)
    assert flags.sum() == 32
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, c["tau"], c["k"], c["seed"])


@pytest.mark.parametrize("V", [8, 1000, 1003, 8192, 8200, 8201, 20000, 32000])
@pytest.mark.parametrize("mode", [KL, CONF])
def test_vocab_sizes_and_ragged_tails(dd, oracle_mod, V, mode):
    """Several pieces or chunks plus a ragged tail, in the row kernel and in the element-wise kernel."""
    dra, ver, tokens, flags = synth.verify_inputs(2, 24, V, 17, 0.2, seed=V)
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 4, 1)
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 4, 1, off=True)


def test_config1_llada_shaped_full_size(dd, oracle_mod):
    c = synth.VERIFY_CONFIGS[1]
    dra, ver, tokens, flags = synth.verify_config_inputs(1)
    n_ex, ref, _ = compare(dd, oracle_mod, dra, ver, tokens, flags, KL, c["tau"], c["k"], c["seed"])
    assert 5 <= ref["out_mask"].sum() <= 60           # ~10% drafter errors get remasked
    assert n_ex <= 4
    # probabilistic variant and the host-buffer entry point on the same data
    compare(dd, oracle_mod, dra, ver, tokens, flags, KL | PROB, c["tau"], c["k"], 3)
    compare(dd, oracle_mod, dra, ver, tokens, flags, KL, c["tau"], c["k"], c["seed"], host=True)


def test_config2_batched_full_size(dd, oracle_mod):
    c = synth.VERIFY_CONFIGS[2]
    dra, ver, tokens, flags = synth.verify_config_inputs(2)
    counts = flags.sum(axis=1)
    assert counts.min() >= 64 and counts.max() <= 256 and len(set(counts.tolist())) > 4
    _, ref, _ = compare(dd, oracle_mod, dra, ver, tokens, flags, CONF, c["tau"], c["k"], c["seed"])
    # every position fails c < 0.5 at this vocabulary size: the top-k rule decides
    kept = (flags.astype(bool) & ~ref["out_mask"].astype(bool)).sum(axis=1)
    assert (kept == c["k"]).all()
    compare(dd, oracle_mod, dra, ver, tokens, flags, CONF | PROB, c["tau"], c["k"], 5)


@pytest.mark.parametrize("mode", [TRUST, KL])
def test_config3_long_context(dd, oracle_mod, mode):
    c = synth.VERIFY_CONFIGS[3]
    dra, ver, tokens, flags = synth.verify_config_inputs(3)
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, c["tau"], c["k"], c["seed"])


@pytest.mark.parametrize("V,seeds", [(32000, (0, 1, 2, 3)), (126464, (0,))])
@pytest.mark.parametrize("err", [0.05, 0.20, 0.50])
def test_config4_sweep(dd, oracle_mod, V, seeds, err):
    sw = synth.VERIFY_SWEEP
    for seed in seeds:
        for nflag in sw["flagged"]:
            dra, ver, tokens, flags = synth.verify_inputs(1, sw["P"], V, nflag, err,
                                                          synth.config_seed(4, seed))
            k = 8 if nflag == 32 else 32
            for mode in (TRUST, KL, CONF) if seed == 0 else (KL,):
                compare(dd, oracle_mod, dra, ver, tokens, flags, mode, sw["tau"], k, seed)
            if seed == 0 and nflag == 128:
                compare(dd, oracle_mod, dra, ver, tokens, flags, KL | PROB, sw["tau"], k, seed)
                compare(dd, oracle_mod, dra, ver, tokens, flags, CONF | PROB, sw["tau"], k, seed)


def test_degenerate_cases(dd, oracle_mod):
    dra, ver, tokens, flags = synth.verify_inputs(3, 16, 256, 9, 0.3, seed=11)
    # nothing flagged anywhere: pure pass-through
    none = np.zeros_like(flags)
    compare(dd, oracle_mod, dra, ver, tokens, none, KL, 0.5, 4, 0)
    # one sequence empty, one full
    mixed = flags.copy(); mixed[0] = 0; mixed[1] = 1
    compare(dd, oracle_mod, dra, ver, tokens, mixed, KL, 0.5, 4, 0)
    # k = 0 (pure rule), k >= number flagged (keep all), unreachable thresholds
    compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.05, 0, 0)
    _, ref, got = compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.0, 1000, 0)
    assert not got[1].any()
    compare(dd, oracle_mod, dra, ver, tokens, flags, CONF, 2.0, 3, 0)
    compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 1e9, 3, 0)
    # identical drafter and verifier: KL = 0 everywhere, nothing exceeds tau = 0
    _, ref, got = compare(dd, oracle_mod, ver, ver, tokens, flags, KL, 0.0, 0, 0)
    assert not got[1].any() and np.abs(got[2]).max() <= 1e-6
    # P = 1, V = 8
    d1, v1, t1, f1 = synth.verify_inputs(1, 1, 8, 1, 0.0, seed=12)
    compare(dd, oracle_mod, d1, v1, t1, f1, CONF, 0.5, 0, 0)


def test_many_short_rows_and_long_sequences(dd, oracle_mod):
    # more (row, chunk) units than the CTAs' tables hold at once (several rounds per CTA), and
    # sequences that exactly fill the decision stage's key area in shared memory (8192 keys)
    dra, ver, tokens, flags = synth.verify_inputs(15, 8192, 64, 5700, 0.2, seed=31)
    compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.5, 40, 3)
    compare(dd, oracle_mod, dra, ver, tokens, flags, CONF | PROB, 0.5, 7, 3)
    # the row kernel's decision of sequences longer than 512 positions
    dra, ver, tokens, flags = synth.verify_inputs(2, 1500, 4104, 900, 0.2, seed=32)
    compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.5, 33, 1)
    # the element-wise kernel (logits off 16-byte boundaries): inside its key area (2048 keys) and beyond
    # it, where every pass of the decision stage re-reads the scores from memory (the streaming kernel's
    # area holds the longest sequence the library accepts)
    for P, nflag in ((1900, 1000), (2500, 1200)):
        dra, ver, tokens, flags = synth.verify_inputs(1, P, 203, nflag, 0.2, seed=P)
        compare(dd, oracle_mod, dra, ver, tokens, flags, KL | PROB, 0.5, 21, 5)
        compare(dd, oracle_mod, dra, ver, tokens, flags, KL | PROB, 0.5, 21, 5, off=True)


@pytest.mark.parametrize("B,P,V,flagged", [(60, 700, 64, 500), (24, 1500, 37, 900), (6, 6000, 64, 3000)])
@pytest.mark.parametrize("mode", [KL, CONF | PROB])
def test_long_sequences_in_the_streaming_kernel(dd, oracle_mod, B, P, V, flagged, mode):
    """Beyond the row kernel's line: the streaming kernel, its decision from registers (up to 1024 positions) and from its key area."""
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, flagged, 0.2, seed=P)
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 33, 1)


def test_exact_ties_in_verifier_row(dd, oracle_mod):
    dra, ver, tokens, flags = synth.verify_inputs(1, 8, 20000, 8, 0.0, seed=13)
    top = synth.f32_to_bf16_bits(np.array([30.0], dtype=np.float32))[0]
    ver[0, 0, [19999, 8191, 8192, 12345]] = top        # ties across chunk and warp boundaries
    ver[0, 1, [7, 3]] = top
    ver[0, 2, :] = top                                  # a constant row
    _, ref, got = compare(dd, oracle_mod, dra, ver, tokens, flags, TRUST, 0.5, 0, 0)
    assert got[0][0, 0] == 8191 and got[0][0, 1] == 3 and got[0][0, 2] == 0


def test_threshold_sweep_crosses_scores(dd, oracle_mod):
    """Thresholds placed on and next to actual scores exercise the exempt band."""
    dra, ver, tokens, flags = synth.verify_inputs(1, 32, 4096, 32, 0.3, seed=14)
    ref = oracle_mod.verify(dra, ver, tokens, flags, KL, 0.5, 0, 0)
    scores = np.sort(ref["out_score"][0])
    n_exempt = 0
    for s in scores[::4]:
        for tau in (s, s * (1 + 3e-6), s * (1 - 3e-6), s + 1e-3):
            n, _, _ = compare(dd, oracle_mod, dra, ver, tokens, flags, KL, float(tau), 0, 0)
            n_exempt += n
    assert n_exempt > 0


def test_out_tokens_may_alias_tokens_and_score_is_optional(dd, oracle_mod):
    import torch
    dra, ver, tokens, flags = synth.verify_inputs(2, 16, 1024, 10, 0.2, seed=15)
    ref = oracle_mod.verify(dra, ver, tokens, flags, KL, 0.5, 2, 0)
    t_tok = torch.from_numpy(tokens.copy()).cuda()
    ot, om, osc = dd.verify(to_torch_bf16(dra, "cuda"), to_torch_bf16(ver, "cuda"), t_tok,
                            torch.from_numpy(flags).cuda(), KL, 0.5, 2, 0,
                            out_tokens=t_tok, want_score=False)
    torch.cuda.synchronize()
    assert osc is None
    strict = ~ref["exempt"].astype(bool)
    assert (ot.cpu().numpy()[strict] == ref["out_tokens"][strict]).all()
    assert (om.cpu().numpy()[strict] == ref["out_mask"][strict]).all()


def test_bitwise_repeatability(dd, oracle_mod):
    dra, ver, tokens, flags = synth.verify_inputs(4, 64, 32000, "uniform_25_100", 0.2, seed=16)
    first = run_gpu(dd, dra, ver, tokens, flags, KL | PROB, 0.5, 8, 9)
    for _ in range(5):
        again = run_gpu(dd, dra, ver, tokens, flags, KL | PROB, 0.5, 8, 9)
        for a, b in zip(first, again):
            assert np.array_equal(a, b)


def test_philox_stream_matches_oracle(dd, oracle_mod):
    """With all verifier logits equal, c = 1/2 exactly at V = 2... use V = 8: c = 1/8, so
    CONF|PROB remasks iff u < 7/8: the GPU's uniforms must match the oracle's one by one."""
    B, P, V = 3, 200, 8
    ver = np.zeros((B, P, V), dtype=np.uint16)
    tokens = np.zeros((B, P), dtype=np.int32)
    flags = np.ones((B, P), dtype=np.uint8)
    for seed in (0, 1, 0xDEADBEEFCAFEF00D):
        ot, om, osc = run_gpu(dd, None, ver, tokens, flags, CONF | PROB, 0.5, 0, seed)
        expect = np.array([[oracle_mod.uniform(seed, b, i) < 0.875 for i in range(P)] for b in range(B)])
        assert np.array_equal(om.astype(bool), expect)


def test_scratch_survives_changing_shapes(dd, oracle_mod):
    """Calls of different (B, P, V) in a row reuse the library's scratch: the completion
    counters must not inherit stale data from a previous layout."""
    shapes = [(1, 8, 64), (4, 300, 1024), (2, 16, 20000), (6, 700, 256), (1, 8, 64), (3, 200, 8)]
    for n, (B, P, V) in enumerate(shapes):
        dra, ver, tokens, flags = synth.verify_inputs(B, P, V, max(1, P // 2), 0.2, seed=100 + n)
        compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.5, 3, n)


@pytest.fixture
def cta_cap(dd):
    """Caps the streaming kernel's grid for one test and lifts the cap afterwards."""
    yield dd.debug_set_max_ctas
    dd.debug_set_max_ctas(0)


def test_results_do_not_depend_on_the_grid(dd, oracle_mod, cta_cap):
    """Same inputs on 1, 7, 37 CTAs and on every SM: tokens, masks and scores bit-identical (which
    warp computes a unit, and in which order units finish, must not matter)."""
    cases = [
        # the row kernel's deep form, whose grid the cap leaves alone
        (synth.verify_inputs(2, 200, 65000, 150, 0.2, seed=43), KL | PROB, 0.5, 8, 0),
        (synth.verify_inputs(2, 200, 65003, 150, 0.2, seed=44), KL, 0.5, 4, 1),
        # the streaming kernel: rows on and off vector boundaries, long and short
        (synth.verify_inputs(4, 200, 65000, 150, 0.2, seed=47), KL | PROB, 0.5, 8, 0),
        (synth.verify_inputs(4, 200, 65003, 150, 0.2, seed=48), KL, 0.5, 4, 1),
        (synth.verify_inputs(4, 256, 65003, 40, 0.2, seed=45), CONF | PROB, 0.5, 4, 2),
        (synth.verify_inputs(6, 6000, 41, 3000, 0.2, seed=46), KL, 0.5, 40, 3),
        # the row kernel
        (synth.verify_config_inputs(0), KL | PROB, 0.5, 8, 0),
        (synth.verify_inputs(2, 40, 20000 + 8 * 37, 29, 0.2, seed=41), KL, 0.5, 4, 1),       # ragged last chunk
        (synth.verify_inputs(2, 40, 20000 + 8 * 37, 29, 0.2, seed=41), CONF | PROB, 0.5, 4, 2),
        (synth.verify_inputs(15, 8192, 64, 5700, 0.2, seed=31), KL, 0.5, 40, 3),              # many short rows: streamed
        (synth.verify_inputs(3, 96, 32000, 80, 0.3, seed=42), TRUST, 0.5, 0, 0),
    ]
    streamed = [takes_the_streaming_kernel(*c[0][1].shape, (c[1] & 0xFF) == KL) for c in cases]
    assert streamed == 2 * [False] + 4 * [True] + 3 * [False] + [True, False]
    for (dra, ver, tokens, flags), mode, tau, k, seed in cases:
        d_in = dra if (mode & 0xFF) == KL else None
        cta_cap(0)
        ref = run_gpu(dd, d_in, ver, tokens, flags, mode, tau, k, seed)
        for cap in (1, 7, 37):
            cta_cap(cap)
            got = run_gpu(dd, d_in, ver, tokens, flags, mode, tau, k, seed)
            for a, b in zip(ref, got):
                assert np.array_equal(a, b), f"cap {cap}"
        cta_cap(0)
        check_verify(*ref, oracle_mod.verify(d_in, ver, tokens, flags, mode, tau, k, seed), flags, tokens)


@pytest.mark.parametrize("V", [20000, 1003])
def test_token_excluded_by_the_verifier_alone(dd, oracle_mod, V):
    """p_V(x) = 0 where p_D(x) > 0: the divergence of Eq. 5 is infinite, in the oracle and in both
    kernels (the vector paths meet the token as a finite logit of -3.4e38 and must notice)."""
    ninf = np.uint16(0xFF80)
    dra, ver, tokens, flags = synth.verify_inputs(2, 12, V, 12, 0.25, seed=77 + V)
    rng = np.random.default_rng(V + 1)
    ver[0, 2, rng.choice(V, size=5, replace=False)] = ninf            # five ordinary tokens
    top = int(np.argmax(synth.bf16_bits_to_f32(dra[1, 3])))
    ver[1, 3, top] = ninf                                              # the drafter's most likely token
    both = rng.choice(V, size=40, replace=False)
    dra[1, 4, both] = ninf; ver[1, 4, both] = ninf                     # a row that stays finite
    tokens[:] = np.argmax(synth.bf16_bits_to_f32(dra), axis=2)
    for off in (False, True):
        _, ref, got = compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.5, 3, 7, off=off)
        inf_at = np.zeros((2, 12), dtype=bool)
        inf_at[0, 2] = inf_at[1, 3] = True
        assert np.isposinf(ref["out_score"][inf_at]).all() and np.isposinf(got[2][inf_at]).all()
        assert np.isfinite(ref["out_score"][~inf_at]).all() and np.isfinite(got[2][~inf_at]).all()


@pytest.mark.parametrize("V", [41000, 41003])
def test_excluded_tokens_in_the_streaming_kernel(dd, oracle_mod, V):
    """The same in rows of several chunks, cut by the ends of ranges."""
    assert takes_the_streaming_kernel(5, 130, V, True)
    ninf = np.uint16(0xFF80)
    dra, ver, tokens, flags = synth.verify_inputs(5, 130, V, 20, 0.25, seed=V)
    rng = np.random.default_rng(V)
    rows = np.argwhere(flags)
    alone, both, drafter, run = rows[3::7], rows[4::7], rows[5::7], rows[6::7]
    for b, i in alone:
        ver[b, i, int(np.argmax(synth.bf16_bits_to_f32(dra[b, i])))] = ninf
    for b, i in both:
        at = rng.choice(V, size=V // 16, replace=False)
        dra[b, i, at] = ninf; ver[b, i, at] = ninf
    for b, i in drafter:
        dra[b, i, rng.choice(V, size=50, replace=False)] = ninf
    for b, i in run:                                          # a chunk and more, and all but the last logits
        dra[b, i, 8:30000] = ninf; ver[b, i, 8:30000] = ninf
    tokens[:] = np.argmax(synth.bf16_bits_to_f32(dra), axis=2)
    _, ref, got = compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 0.5, 3, 7)
    assert sorted(map(tuple, np.argwhere(np.isposinf(got[2])))) == sorted(map(tuple, alone))


@pytest.mark.parametrize("V", [4096, 20000, 1003])
def test_excluded_tokens(dd, oracle_mod, V):
    """Logits of -inf (banned or padded vocabulary entries) at shared and at drafter-only
    indices: probability zero, no term in Eq. 5; the other rows are untouched by the detour."""
    ninf = np.uint16(0xFF80)
    if True:
        dra, ver, tokens, flags = synth.verify_inputs(2, 12, V, 12, 0.25, seed=51 + V)
        rng = np.random.default_rng(V)
        both = rng.choice(V, size=V // 16, replace=False)
        dra[0, 1, both] = ninf; ver[0, 1, both] = ninf                 # excluded by both models
        dra[0, 3, both[:50]] = ninf                                    # excluded by the drafter only
        run_end = 4000 if V > 4096 else 1000
        dra[1, 5, 8:run_end] = ninf; ver[1, 5, 8:run_end] = ninf       # a whole run of the row
        dra[1, 7, :V - 3] = ninf; ver[1, 7, :V - 3] = ninf             # nearly everything
        tokens[:] = np.argmax(synth.bf16_bits_to_f32(dra), axis=2)
        for mode in (KL, CONF, KL | PROB):
            for off in (False, True):
                _, ref, got = compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 3, 7, off=off)
                assert np.isfinite(ref["out_score"]).all() and np.isfinite(got[2]).all()


# vocabularies that put rows anywhere between 16-byte boundaries: fewer logits than a vector, one vector more
# or less than a stage (1024 logits of both tensors, 2048 of one), a chunk's last stage of a few logits
@pytest.mark.parametrize("V", [1, 3, 7, 9, 15, 1017, 1023, 1025, 1031, 2041, 2047, 2050, 4089, 4095, 4097, 8190, 8193, 16385])
@pytest.mark.parametrize("mode", [KL, CONF])
def test_rows_off_vector_boundaries(dd, oracle_mod, V, mode):
    dra, ver, tokens, flags = synth.verify_inputs(2, 37, V, 23, 0.3, seed=V + 1)
    flags[1, -1] = 1                         # the tensor's last row, whose last vector is not whole
    flags[0, 0] = 1
    # the neighbours' logits share vectors with a flagged row's and must not reach it
    ver[flags == 0] = 0x7FC0
    dra[flags == 0] = 0x7F80
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 4, 1)


@pytest.mark.parametrize("V", [1000, 1003])
@pytest.mark.parametrize("mode", [KL, CONF])
def test_logits_off_16_byte_boundaries(dd, oracle_mod, V, mode):
    """Tensors that start in the middle of a vector take the element-wise kernel."""
    import torch
    dra, ver, tokens, flags = synth.verify_inputs(2, 24, V, 17, 0.2, seed=V)
    ref = oracle_mod.verify(dra if mode == KL else None, ver, tokens, flags, mode, 0.5, 4, 1)
    off = off_vector_boundary
    out = dd.verify(off(dra) if mode == KL else None, off(ver), torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda(),
                    mode, 0.5, 4, 1)
    torch.cuda.synchronize()
    assert dd.verify_status() == 0
    check_verify(*(x.cpu().numpy() for x in out), ref, flags, tokens)


# shapes on both sides of the line between the row kernel and the streaming kernel (23680 pieces of 1024 logits of
# both tensors or 2048 of one on 148 SMs), rows on and off vector boundaries; in the streaming kernel rows cut
# by range boundaries and grids of any size; in the row kernel clusters, CTAs, warps per row
@pytest.mark.parametrize("B,P,V,flagged,mode", [
    (2, 200, 65000, 150, KL), (2, 200, 65003, 150, KL),              # the deep form of the row kernel
    (4, 200, 65000, 150, KL | PROB), (4, 200, 65003, 150, KL),       # streaming
    (4, 256, 65000, 40, CONF), (4, 256, 65003, 40, CONF | PROB),     # streaming
    (1, 20, 126464, 20, KL | PROB), (1, 40, 65003, 33, KL), (2, 70, 40003, 60, CONF),   # clusters of eight, four and two
    (1, 300, 20003, 77, KL), (4, 200, 9001, 150, KL), (6, 512, 4100, 100, KL), (24, 300, 1001, 100, CONF),   # 8, 4, 2 and 1 warps
])
def test_row_and_streaming_kernels(dd, oracle_mod, B, P, V, flagged, mode):
    assert takes_the_streaming_kernel(B, P, V, (mode & 0xFF) == KL) == (B * P > 592 and V > 60000)
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, flagged, 0.2, seed=V + P)
    hot = np.argmax(synth.bf16_bits_to_f32(ver[0, :1]), axis=1)
    flags[0, 0] = 1
    for row in ver.reshape(-1, V)[::7]:      # a token excluded by the verifier, somewhere
        row[(int(hot[0]) + 5) % V] = 0xFF80
    for row in dra.reshape(-1, V)[::7]:      # and by the drafter
        row[(int(hot[0]) + 5) % V] = 0xFF80
    _, _, whole = compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 9, 3)
    try:
        for cap in (1, 61):
            dd.debug_set_max_ctas(cap)
            got = run_gpu(dd, dra if (mode & 0xFF) == KL else None, ver, tokens, flags, mode, 0.5, 9, 3)
            for a, b in zip(whole, got):
                np.testing.assert_array_equal(a, b)
    finally:
        dd.debug_set_max_ctas(0)


# the row kernel's deep form: two pieces to a warp and many, rows on and off vector boundaries (edges at both ends of a row), a last piece of
# a few logits, of all but one and none at all, clusters; flagged rows first: none, one, the last, more of them than a word of 32
@pytest.mark.parametrize("B,P,V,flagged,mode", [
    (1, 256, 24 * 1024, 256, KL), (1, 200, 25 * 1024 + 1, 1, KL | PROB), (1, 130, 51 * 1024 - 1, 130, CONF), (2, 148, 49155, 97, KL),
    (1, 40, 70001, 40, CONF), (2, 5, 126464, 3, KL), (1, 300, 25 * 1024 + 3, 33, KL), (2, 290, 26001, 580, KL), (3, 60, 50000, 0, KL)])
def test_row_kernel_with_long_rows(dd, oracle_mod, B, P, V, flagged, mode):
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, min(flagged, P), 0.2, seed=V + P)
    if flagged == 0:
        flags[:] = 0
        flags[1, P - 1] = 1                  # one sequence with its last row only, two without any
    every = ver.reshape(-1, V)
    for i, row in enumerate(every[::5]):     # excluded tokens: at the row's ends, a whole lane's vector, a whole piece
        row[[0, V - 1, 7 * i % V]] = 0xFF80
        row[1024:1032] = 0xFF80
        dra.reshape(-1, V)[5 * i, [0, V - 1, 7 * i % V]] = 0xFF80
        dra.reshape(-1, V)[5 * i, 1024:2048] = 0xFF80
    compare(dd, oracle_mod, dra, ver, tokens, flags, mode, 0.5, 9, 3)


# more long rows than the GPU holds CTAs of the row kernel at a time: the first sequences are decided before the last rows begin
@pytest.mark.parametrize("B,P,V,flagged,mode", [(2, 256, 126464, 256, KL), (4, 100, 126464, 60, CONF), (2, 290, 26001, 290, KL | PROB)])
def test_mask_in_place_of_the_flags(dd, B, P, V, flagged, mode):
    import torch
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, flagged, 0.2, seed=V + P)
    dra, ver = to_torch_bf16(dra, "cuda") if (mode & 0xFF) == KL else None, to_torch_bf16(ver, "cuda")
    tok, fl = torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()
    want = dd.verify(dra, ver, tok, fl, mode, 0.5, 9, 3)
    for _ in range(2):
        mask = fl.clone()
        got = dd.verify(dra, ver, tok, mask, mode, 0.5, 9, 3, out_mask=mask)
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    again = dd.verify(dra, ver, tok, fl, mode, 0.5, 9, 3)         # the counters are as they should be
    assert all(torch.equal(a, b) for a, b in zip(want, again))
    assert dd.verify_status() == 0


@pytest.mark.parametrize("B,P,V,mode", [(1, 256, 126464, KL), (1, 256, 126464, CONF), (2, 200, 126464, KL), (2, 200, 126464, CONF),
                                        (4, 200, 126464, KL), (4, 200, 126464, CONF)])
def test_long_sums_are_as_exact_as_short_ones(dd, B, P, V, mode):
    """Terms of 2^-8.8 added to sums that begin at 1: every addition rounds down.  A chain of 128 additions (a lane's half of a chunk of 8192
    logits) is out by no more than 128 * 2^-24; one over a warp's share of a row in the row kernel would be out by 9.6e-6."""
    import torch
    row = torch.full((V,), -6.09375, dtype=torch.float64)
    step = 1024 if mode == KL else 2048
    for piece in range(8):                       # each lane's first word, in each warp's first piece of the row kernel
        first = piece * step + 8 * torch.arange(32)
        row[first] = row[first + 1] = 0.0
    ver = row.to(torch.bfloat16).cuda().expand(B, P, V).contiguous()
    dra = torch.zeros_like(ver) if mode == KL else None          # all terms of its sums are exact
    tok, fl = torch.zeros(B, P, dtype=torch.int32, device="cuda"), torch.ones(B, P, dtype=torch.uint8, device="cuda")
    got = dd.verify(dra, ver, tok, fl, mode, 0.5, 0, 0)[2].double()
    bound = 128 * 2.0 ** -24
    lse = torch.logsumexp(row, 0).item()
    # the logarithm of the sum has the sum's relative error as its absolute one
    want, tol = (lse - np.log(V) - row.mean().item(), bound) if mode == KL else (np.exp(-lse), bound * np.exp(-lse))
    assert (got - want).abs().max().item() <= tol
    assert dd.verify_status() == 0


# lengths at the lines between the row kernel and the streaming kernel on 148 SMs (one row: 23680 pieces; 150 and 40 rows: 20 pieces for each of
# eight and thirty-two warps), and far beyond what a warp of the row kernel could count
@pytest.mark.parametrize("P,V,mode", [
    (1, 48_490_000, CONF), (1, 48_500_000, CONF), (1, 300_000_001, CONF), (1, 24_240_000, KL), (1, 24_250_000, KL), (1, 300_000_000, KL),
    (150, 327_000, CONF), (150, 328_000, CONF), (150, 163_000, KL), (150, 164_000, KL), (40, 654_000, KL), (40, 656_000, KL)])
def test_place_of_the_maximum_of_very_long_rows(dd, P, V, mode):
    import torch
    ver = torch.zeros(1, P, V, dtype=torch.bfloat16, device="cuda")
    places = [V - 5 if r == P - 1 else V * (r + 1) // P - 1 for r in range(P)]
    ver[0, torch.arange(P), torch.tensor(places)] = 8.0
    tok, fl = torch.zeros(1, P, dtype=torch.int32, device="cuda"), torch.ones(1, P, dtype=torch.uint8, device="cuda")
    # (KL: of the constant distribution from this one)
    dra = torch.zeros_like(ver) if mode == KL else None
    got = dd.verify(dra, ver, tok, fl, mode, 100.0 if mode == KL else 0.0, 0, 0)
    assert got[0].cpu().tolist() == [places] and not got[1].any()
    total = np.exp(8.0) + V - 1
    want = -8.0 / V - np.log(V) + np.log(total) if mode == KL else np.exp(8.0) / total
    # KL is a difference of numbers of the size of log V, which come from fp32 sums
    assert np.abs(got[2].cpu().numpy() - want).max() <= (1e-5 * np.log(V) if mode == KL else 1e-4 * want)
    assert dd.verify_status() == 0


@pytest.mark.parametrize("k", [1, 2, 31, 32, 33, 100, 299, 300, 301])
def test_minimum_keep_with_many_equal_scores(dd, oracle_mod, k):
    """300 rows of which many are the same: ties at every place of the order, kept lowest index first."""
    dra, ver, tokens, flags = synth.verify_inputs(1, 300, 256, 300, 0.5, seed=3)
    same = np.random.default_rng(k).integers(0, 12, size=300)
    dra, ver = dra[:, same], ver[:, same]
    for mode in (KL, CONF):
        ref = oracle_mod.verify(dra if mode == KL else None, ver, tokens, flags, mode, 0.0 if mode == KL else 1.0, k, 0)
        ot, om, osc = run_gpu(dd, dra if mode == KL else None, ver, tokens, flags, mode, 0.0 if mode == KL else 1.0, k, 0)
        # equal rows have equal scores on either side, so the order is the same and so is the kept set
        np.testing.assert_array_equal(om, ref["out_mask"])
        np.testing.assert_array_equal(ot, ref["out_tokens"])


@pytest.mark.parametrize("P,ks", [(1, [1]), (31, [1, 30]), (129, [1, 64, 128]), (256, [7, 255]), (257, [1, 8, 200]), (512, [3, 256, 511])])
def test_threshold_of_the_minimum_keep(dd, oracle_mod, P, ks):
    """The k-th most reliable position at every size of the short decision stage: scores that differ everywhere, scores
    of three values (ties at the threshold) and scores that are all the same."""
    rng = np.random.default_rng(P)
    distinct = synth.verify_inputs(2, P, 64, P, 0.5, seed=P)
    for rows in (None, 3, 1):
        dra, ver, tokens, flags = (x.copy() for x in distinct)
        if rows:
            pick = rng.integers(0, min(rows, P), (2, P))
            for b in range(2):
                dra[b], ver[b] = distinct[0][b][pick[b]], distinct[1][b][pick[b]]
            tokens[:] = np.argmax(synth.bf16_bits_to_f32(dra), axis=2)
        for k in ks:
            compare(dd, oracle_mod, dra, ver, tokens, flags, KL, 1e-6, k, 1)
            compare(dd, oracle_mod, dra, ver, tokens, flags, CONF, 0.999999, k, 1)

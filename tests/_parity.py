"""Shared comparison rules of the GPU parity tests.

Attention: max-abs <= 1e-2 and mean-abs <= 1e-3 against the fp64 oracle.  The output is
bf16: from |out| = 4 upwards its grid is coarser than 2 x 1e-2 (spacing 2^-5 in [4, 8)), so
that no bf16 value need lie within 1e-2 of the exact result; there the max-abs bar scales with
the spacing (2e-2 in [4, 8), 4e-2 in [8, 16), ...).  Below 4 it is 1e-2 as stated.
Verify: scores within 1e-4 relative (absolute floor 1e-6 where the score is
near zero); remask sets and emitted tokens bit-exact except at positions the
oracle flags as lying within 1e-5 of a decision boundary.
"""
import numpy as np

ATTN_MAX_ABS = 1e-2
ATTN_MEAN_ABS = 1e-3
SCORE_REL = 1e-4
SCORE_ABS_FLOOR = 1e-6


def to_torch_bf16(bits, device=None, pin=False):
    import torch
    t = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16)
    if device is not None:
        return t.to(device)
    return t.pin_memory() if pin else t


def off_vector_boundary(bits):
    """The same numbers on the device in a tensor that starts in the middle of a 16-byte vector."""
    import torch
    big = torch.zeros(bits.size + 8, dtype=torch.bfloat16, device="cuda")
    view = big[3:3 + bits.size].view(bits.shape)
    view.copy_(to_torch_bf16(bits, "cuda"))
    assert view.data_ptr() % 16 != 0
    return view


def takes_the_streaming_kernel(B, P, V, kl):
    """Whether dd_verify's rule on sizes gives (aligned) logits of this shape to the streaming kernel on this GPU: more than 160 pieces
    of 4 KB per SM, and more than four rows per SM (of no more than 150000 logits)."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pieces = (V + 7) // (1024 if kl else 2048) + 1
    return B * P > 32768 or (B * P * pieces > 160 * sms and B * P > 4 * sms)


def bf16_tensor_to_f64(t):
    import torch
    return t.detach().to("cpu").to(torch.float64).numpy()


def attention_max_abs_bar(oracle_out):
    """1e-2, times the bf16 grid spacing relative to that of [2, 4) where the exact value is >= 4."""
    mag = np.maximum(np.abs(oracle_out), 1e-30)
    return ATTN_MAX_ABS * np.maximum(1.0, np.exp2(np.floor(np.log2(mag)) - 1.0))


# Stress inputs only (planted strength 6: one or two keys carry a row).  Where the exact value
# lies in [2, 4), half a unit of the bf16 output is already 2^-7 = 7.8e-3, and the bf16 rounding
# of the weights (2^-9 relative each) of two keys that share a row adds up to
# 2^-8 |v1 - v2| / 4 = 3.9e-3 for |v1 - v2| = 4: 1.17e-2 together.  Such elements are rare
# (they need both roundings near their worst case): at most STRESS_OVER_SHARE of all elements may
# pass 1e-2, none may pass STRESS_MAX_ABS.
STRESS_MAX_ABS = 1.2e-2
STRESS_OVER_SHARE = 1e-5


def check_attention(gpu_out_f64, oracle_out, stress=False):
    diff = np.abs(gpu_out_f64 - oracle_out)
    assert np.isfinite(gpu_out_f64).all()
    bar = attention_max_abs_bar(oracle_out)
    if stress:
        late = (diff > bar) & (np.abs(oracle_out) >= 2.0) & (np.abs(oracle_out) < 4.0)
        assert late.sum() <= max(1, int(STRESS_OVER_SHARE * diff.size)), f"{late.sum()} of {diff.size} elements over 1e-2"
        bar = np.where(late, STRESS_MAX_ABS, bar)
    over = diff > bar
    assert not over.any(), (f"{over.sum()} elements over the max-abs bar; worst {diff[over].max():.3e} "
                            f"at |exact| = {np.abs(oracle_out)[over][diff[over].argmax()]:.3f}")
    assert diff.mean() <= ATTN_MEAN_ABS, f"mean-abs {diff.mean():.3e}"
    return float(diff.max()), float(diff.mean())


def check_verify(gpu_tokens, gpu_mask, gpu_score, ref, flags, tokens_in, score_abs=SCORE_ABS_FLOOR):
    """ref: dict from oracle.verify; gpu_*: numpy arrays."""
    flags = flags.astype(bool)
    exempt = ref["exempt"].astype(bool)
    o_score = ref["out_score"]
    g_score = gpu_score.astype(np.float64)
    unbounded = np.isinf(o_score)                   # a token only the verifier excludes: KL = +inf
    assert np.array_equal(unbounded, np.isinf(g_score)), "infinite scores at different positions"
    assert (g_score[unbounded] == o_score[unbounded]).all()
    fin = ~unbounded
    tol = np.maximum(SCORE_REL * np.abs(o_score[fin]), score_abs)
    err = np.abs(g_score[fin] - o_score[fin])
    bad = ~(err <= tol)                             # a NaN is out of tolerance too
    assert not bad.any(), f"{bad.sum()} scores out of tolerance; worst {np.nanmax(err):.3e}"
    strict = ~exempt
    mism_mask = (gpu_mask != ref["out_mask"]) & strict
    assert not mism_mask.any(), f"{mism_mask.sum()} remask decisions differ outside the exempt set"
    mism_tok = (gpu_tokens != ref["out_tokens"]) & strict
    assert not mism_tok.any(), f"{mism_tok.sum()} emitted tokens differ outside the exempt set"
    # at exempt positions either decision is acceptable, but the token must match that decision
    ex = exempt & flags
    if ex.any():
        kept_tok = np.where(ref["out_mask"].astype(bool), -1, ref["out_tokens"])
        ok = (gpu_mask.astype(bool) & (gpu_tokens == tokens_in)) | \
             (~gpu_mask.astype(bool) & ((gpu_tokens == kept_tok) | (kept_tok < 0)))
        assert ok[ex].all()
    # unflagged positions pass through untouched
    assert (gpu_tokens[~flags] == tokens_in[~flags]).all()
    assert not gpu_mask[~flags].any() and not gpu_score[~flags].any()
    return int(exempt.sum())


# ----------------------------------------------------------------------------- guard regions
#
# Every GPU output is allocated inside a larger buffer filled with a sentinel; after the call the
# margins must be untouched.  An out-of-range store by a kernel (a decision stage that runs past
# the sequence, an epilogue tile that is not clipped) then fails the test that made it.

GUARD_ELEMS = 1024          # per side; a multiple of 8, so 2-byte views stay 16-byte aligned


class Guarded:
    """A device (or pinned host) tensor of `shape` with GUARD_ELEMS sentinel elements on both sides."""

    _SENTINEL = {"torch.bfloat16": -2.0078125e3, "torch.float32": -7.25e11, "torch.int32": -0x5A5A5A5B,
                 "torch.uint8": 0xA5}

    def __init__(self, shape, dtype, device="cuda", pin=False):
        import torch
        n = int(np.prod(shape))
        self.fill = self._SENTINEL[str(dtype)]
        if device is None:
            self.raw = torch.empty(n + 2 * GUARD_ELEMS, dtype=dtype)
            if pin:
                self.raw = self.raw.pin_memory()
        else:
            self.raw = torch.empty(n + 2 * GUARD_ELEMS, dtype=dtype, device=device)
        self.raw.fill_(self.fill)
        self.view = self.raw[GUARD_ELEMS:GUARD_ELEMS + n].view(*shape)
        self.n = n

    def check(self, what="output"):
        import torch
        lo = self.raw[:GUARD_ELEMS]
        hi = self.raw[GUARD_ELEMS + self.n:]
        ref = torch.full_like(lo, self.fill)
        assert torch.equal(lo, ref), f"{what}: the kernel wrote below the buffer"
        assert torch.equal(hi, ref), f"{what}: the kernel wrote past the buffer"

"""The workloads whose speed is watched: what a program built on this library has it do.

A case is a dict of plain values.  ``kind`` says which public call it makes:

  attention  binding.bidir_attention: one layer's full-sequence attention of a model's forward pass
  block      binding.block_attention: a drafter's query block over its stored keys and values
  verify     binding.verify: the verification algorithm on both models' logits
  unmask     binding.unmask: the drafter's unmasking step
  head       binding.lm_head_verify: language-model heads and verification from hidden states
  step       attention, then verify: the smallest whole step
  generate   pipeline.dualdiffusion_generate: Algorithm 1's loop around all of it

Inputs are drawn on the GPU from the seed alone, by the recipes of ``paper_2604_05250_b200.synth``.
"""
import math

import torch

from paper_2604_05250_b200 import binding, pipeline

KL, CONF, TRUST = binding.DD_MODE_KL, binding.DD_MODE_CONF, binding.DD_MODE_TRUST
MODES = {"kl": KL, "conf": CONF, "trust": TRUST,
         "kl_prob": KL | binding.DD_FLAG_PROBABILISTIC, "conf_prob": CONF | binding.DD_FLAG_PROBABILISTIC,
         "kl_emit": KL | binding.DD_FLAG_EMIT_DRAFTER}
TAU = 0.5
ERR = 0.10           # share of positions that the drafter gets wrong


def listed():
    return [
        # the smallest step: latency, launches and host work are all there is
        dict(name="step_tiny", kind="step", B=1, H=4, N=128, D=64, P=128, V=1024, share=0.25, mode="kl", k=8),
        # one sequence of 768 prompt and 256 generated tokens, one layer of an 8B-parameter verifier
        dict(name="attention_step", kind="attention", B=1, H=32, N=1024, D=128, planted=False),
        # sixteen sequences served together
        dict(name="attention_serving", kind="attention", B=16, H=32, N=512, D=128, planted=False),
        # a long context, with score rows as peaked as trained heads make them
        dict(name="attention_long", kind="attention", B=1, H=32, N=8192, D=128, planted=True),
        # sequences cut to no round length, the small head dimension
        dict(name="attention_ragged", kind="attention", B=3, H=24, N=1357, D=64, planted=False),
        # the drafter's step on a block-wise key-value cache: sequences of unequal length, heads interleaved
        dict(name="block_drafter", kind="block", B=16, H=32, Nq=32, Nkv=1024, D=128, ragged=True, layout="bnhd"),
        # the verification of one generated block of 256 tokens, every one of them drafted
        dict(name="verify_kl_step", kind="verify", B=1, P=256, V=126464, share=1.0, mode="kl", k=32),
        # a served batch in confidence mode, a quarter to all of each sequence's positions drafted
        dict(name="verify_conf_serving", kind="verify", B=16, P=256, V=126464, share=0.0, mode="conf", k=16),
        # a vocabulary that a mask token has made odd, half of the positions drafted
        dict(name="verify_odd_vocabulary", kind="verify", B=2, P=300, V=32001, share=0.5, mode="kl_prob", k=8),
        # verification straight from the verifier's hidden states, the served batch above
        dict(name="head_conf_serving", kind="head", B=16, P=256, K=4096, V=126464, share=0.0, mode="conf", k=16),
        # the same for one block, from both models' hidden states
        dict(name="head_kl_step", kind="head", B=1, P=256, K=4096, V=126464, share=1.0, mode="kl", k=32),
        # the whole loop on small models: many short calls, each waiting for the one before it
        dict(name="generate", kind="generate", B=4, P=128, V=4096, K=4, unmask_k=8, mode="kl", k=8),
    ]


def _ideal(case):
    """Seconds that `work` takes at 6.5 TB/s and 1600 TFLOP/s: what draws are bounded by."""
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.6e15)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["attention", "attention", "block", "verify", "verify", "unmask", "head", "step", "generate"])
    heads, dim = rng.choice([4, 8, 16, 24, 32]), rng.choice([64, 128, 128])
    batch = _log(rng, 1, 16)
    share = rng.choice([0.0, 1.0, round(rng.uniform(0.05, 0.95), 2)])
    k = rng.choice([0, 1, 8, 16, 32])
    vocab = _log(rng, 1000, 126464)
    if rng.random() < 0.6:
        vocab -= vocab % 64                     # most vocabularies are padded; the rest are as they come
    if kind == "attention":
        return dict(kind=kind, B=batch, H=heads, N=_log(rng, 64, 8192), D=dim, planted=rng.random() < 0.5)
    if kind == "block":
        return dict(kind=kind, B=_log(rng, 1, 64), H=heads, Nq=_log(rng, 1, 256), Nkv=_log(rng, 64, 4096), D=dim,
                    ragged=rng.random() < 0.6, layout=rng.choice(["bhnd", "bnhd"]))
    if kind == "verify":
        return dict(kind=kind, B=batch, P=_log(rng, 16, 512), V=vocab, share=share, mode=rng.choice(sorted(MODES)), k=k)
    if kind == "unmask":
        return dict(kind=kind, B=batch, P=_log(rng, 16, 512), V=vocab, share=share, k=max(1, k))
    if kind == "head":
        return dict(kind=kind, B=batch, P=_log(rng, 16, 512), K=64 * _log(rng, 8, 64), V=vocab, share=share,
                    mode=rng.choice(["kl", "conf", "conf_prob", "trust"]), k=k)
    if kind == "step":
        return dict(kind=kind, B=1, H=heads, N=_log(rng, 64, 512), D=dim, P=_log(rng, 16, 128), V=_log(rng, 128, 4000) * 8,
                    share=max(share, 0.25), mode=rng.choice(["kl", "conf", "trust"]), k=k)
    # a loop costs its number of calls: no more of them than the listed case makes
    unmask_k = rng.choice([8, 12, 16])
    return dict(kind=kind, B=_log(rng, 1, 8), P=_log(rng, 32, 16 * unmask_k - 64), V=_log(rng, 128, 1000) * 8, K=rng.choice([2, 4, 8]),
                unmask_k=unmask_k, mode=rng.choice(["kl", "trust"]), k=rng.choice([12, 16]))


def draw(rng):
    most = max(_ideal(c) for c in listed())
    while True:
        case = _draw(rng)
        if _ideal(case) <= most:
            return case


# ----------------------------------------------------------------------------- inputs


def _spread(n, lo, hi):
    """n whole numbers evenly spread over lo..hi (their order is drawn, their sum is not)."""
    return [int(round(lo + (hi - lo) * (i + 0.5) / n)) for i in range(n)]


def _counts(case):
    """Flagged positions per sequence: the given share of P, or 25 % to 100 % of it (share 0)."""
    P, B = case["P"], case["B"]
    if case["share"] == 0.0:
        return [max(1, c) for c in _spread(B, 0.25 * P, P)]
    return [max(1, int(round(case["share"] * P)))] * B


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _flags(case, gen):
    counts = torch.tensor(_counts(case), device="cuda")
    counts = counts[torch.randperm(case["B"], device="cuda", generator=gen)]
    rank = torch.rand(case["B"], case["P"], device="cuda", generator=gen).argsort(dim=1).argsort(dim=1)
    return (rank < counts[:, None]).to(torch.uint8)


def _attention_inputs(B, H, N, D, planted, gen):
    q, k, v = (torch.randn(B, H, N, D, device="cuda", generator=gen) for _ in range(3))
    if planted:
        # a shared component of rank 16 in q and k: peaked score rows
        w = torch.linalg.qr(torch.randn(B, H, D, 16, device="cuda", generator=gen))[0].transpose(-1, -2)
        q += 3.0 * (torch.randn(B, H, N, 16, device="cuda", generator=gen) @ w)
        k += 3.0 * (torch.randn(B, H, N, 16, device="cuda", generator=gen) @ w)
    return [t.to(torch.bfloat16) for t in (q, k, v)]


def _logits(B, P, V, gen, drafter):
    """Verifier N(0, 2^2) with +8 at one token per position; the drafter's differ by N(0, 0.5^2), or
    are another row on a share of the positions.  Returns (drafter or None, verifier), bf16."""
    ver = torch.randn(B, P, V, device="cuda", generator=gen).mul_(2.0)
    hot = torch.randint(0, V, (B, P, 1), device="cuda", generator=gen)
    ver.scatter_add_(2, hot, torch.full((B, P, 1), 8.0, device="cuda"))
    dra = None
    if drafter:
        dra = torch.randn(B, P, V, device="cuda", generator=gen)
        wrong = torch.rand(B, P, 1, device="cuda", generator=gen) < ERR
        dra = torch.where(wrong, 2.0 * dra, ver + 0.5 * dra).to(torch.bfloat16)
    return dra, ver.to(torch.bfloat16)


def _verify_state(case, gen, seed):
    dra, ver = _logits(case["B"], case["P"], case["V"], gen, MODES[case["mode"]] & 0xFF == KL)
    tokens = torch.randint(0, case["V"], (case["B"], case["P"]), device="cuda", generator=gen, dtype=torch.int32)
    return dict(drafter=dra, verifier=ver, tokens=tokens, flags=_flags(case, gen), seed=seed)


def _head_state(case, gen, seed):
    B, P, K, V = case["B"], case["P"], case["K"], case["V"]
    weight = torch.randn(V, K, device="cuda", generator=gen).mul_(2.0 / math.sqrt(K))
    hidden = torch.randn(B, P, K, device="cuda", generator=gen)
    hot = torch.randint(0, V, (B, P), device="cuda", generator=gen)
    hidden += 2.0 * weight[hot]                   # the hot token's logit rises by about 8
    s = dict(vh=hidden.to(torch.bfloat16), vw=weight.to(torch.bfloat16), dh=None, dw=None, seed=seed,
             tokens=hot.to(torch.int32), flags=_flags(case, gen))
    if MODES[case["mode"]] & 0xFF == KL:
        weight += (0.2 / math.sqrt(K)) * torch.randn(V, K, device="cuda", generator=gen)
        wrong = torch.rand(B, P, 1, device="cuda", generator=gen) < ERR
        other = torch.randn(B, P, K, device="cuda", generator=gen)
        s["dh"] = torch.where(wrong, other, hidden + 0.25 * other).to(torch.bfloat16)
        s["dw"] = weight.to(torch.bfloat16)
    return s


def _generate_state(case, gen):
    """Two small models: logits from the position and from the token that stands there."""
    B, P, V = case["B"], case["P"], case["V"]
    mask_id = V - 1
    dra, ver = _logits(B, P, V, gen, True)
    table = torch.randn(V, V, device="cuda", generator=gen).mul_(0.25).to(torch.bfloat16)
    for t in (dra, ver):
        t[:, :, mask_id] = -math.inf              # no model emits the mask token
    tokens = torch.full((B, P), mask_id, dtype=torch.int32, device="cuda")
    return dict(drafter=lambda x: dra + table[x], verifier=lambda x: ver + table[x], tokens=tokens, mask_id=mask_id)


def prepare(case, seed):
    gen, kind = _generator(seed), case["kind"]
    s = dict(case=case)
    if kind in ("attention", "step"):
        s["q"], s["k"], s["v"] = _attention_inputs(case["B"], case["H"], case["N"], case["D"], case.get("planted", False), gen)
    if kind == "block":
        B, H, Nq, Nkv, D = (case[x] for x in ("B", "H", "Nq", "Nkv", "D"))
        shape = (lambda n: (B, H, n, D)) if case["layout"] == "bhnd" else (lambda n: (B, n, H, D))
        s["q"], s["k"], s["v"] = (torch.randn(shape(n), device="cuda", generator=gen).to(torch.bfloat16) for n in (Nq, Nkv, Nkv))
        s["lens"] = None
        if case["ragged"]:
            lens = torch.tensor(_spread(B, 0.25 * Nkv, Nkv), dtype=torch.int32, device="cuda")
            s["lens"] = lens[torch.randperm(B, device="cuda", generator=gen)].contiguous()
    if kind in ("verify", "step"):
        s.update(_verify_state(case, gen, seed))
    if kind == "unmask":
        s.update(_verify_state(dict(case, mode="conf"), gen, seed))
    if kind == "head":
        s.update(_head_state(case, gen, seed))
    if kind == "generate":
        s.update(_generate_state(case, gen))
    return s


# ----------------------------------------------------------------------------- the calls


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "attention":
        return binding.bidir_attention(s["q"], s["k"], s["v"])
    if kind == "block":
        return binding.block_attention(s["q"], s["k"], s["v"], kv_len=s["lens"], layout=case["layout"])
    if kind == "unmask":
        return binding.unmask(s["verifier"], s["tokens"], s["flags"], TAU, case["k"])
    if kind == "head":
        return binding.lm_head_verify(s["dh"], s["dw"], s["vh"], s["vw"], s["tokens"], s["flags"],
                                      MODES[case["mode"]], TAU, case["k"], s["seed"])
    if kind == "generate":
        tokens, stats = pipeline.dualdiffusion_generate(
            s["drafter"], s["verifier"], s["tokens"], s["mask_id"], case["K"], MODES[case["mode"]], TAU, case["k"],
            unmask_k=case["unmask_k"], max_cycles=256)
        return tokens, stats.cycles, stats.drafter_calls, stats.remasked_by_verifier
    out = []
    if kind == "step":
        out.append(binding.bidir_attention(s["q"], s["k"], s["v"]))
    out.extend(binding.verify(s["drafter"], s["verifier"], s["tokens"], s["flags"], MODES[case["mode"]], TAU, case["k"], s["seed"]))
    return out


def work(case):
    kind, flops, size = case["kind"], 0.0, 0.0
    if kind in ("attention", "step"):
        flops += 4.0 * case["B"] * case["H"] * case["N"] ** 2 * case["D"]
        size += 8.0 * case["B"] * case["H"] * case["N"] * case["D"]
    if kind == "block":
        keys = sum(_spread(case["B"], 0.25 * case["Nkv"], case["Nkv"])) if case["ragged"] else case["B"] * case["Nkv"]
        flops += 4.0 * case["H"] * case["Nq"] * keys * case["D"]
        size += 4.0 * case["H"] * case["D"] * (keys + case["B"] * case["Nq"])
    if kind in ("verify", "unmask", "step"):
        models = 2 if MODES[case.get("mode", "conf")] & 0xFF == KL else 1
        size += sum(_counts(case)) * case["V"] * 2.0 * models + 14.0 * case["B"] * case["P"]
    if kind == "head":
        models = 2 if MODES[case["mode"]] & 0xFF == KL else 1
        rows = sum(_counts(case))                 # only flagged positions need logits
        flops += 2.0 * models * rows * case["K"] * case["V"]
        size += 2.0 * models * case["K"] * (rows + case["V"]) + 14.0 * case["B"] * case["P"]
    if kind == "generate":
        # every unmasking step reads the positions still masked, and every position is verified once at least
        masked = sum(range(case["P"], 0, -case["unmask_k"]))
        models = 2 if MODES[case["mode"]] & 0xFF == KL else 1
        size += 2.0 * case["B"] * case["V"] * (masked + models * case["P"])
    return {"bytes": size, "flops": flops}


def tolerance(case):
    # Four times the distance from the same definitions in 64 bits, as measured on the listed cases.
    # Whole values may differ where two candidates tie to within rounding.
    kind = case["kind"]
    if kind in ("attention", "block"):           # bf16 weights and results: rel 2.3e-3, max 1.3e-2
        return {"rel": 1e-2, "max": 5e-2}
    if kind == "step":
        return {"rel": 1e-2, "max": 5e-2, "differ": 2e-3}
    if kind == "head":                           # 4096 products per logit in fp32: rel 2.1e-5, max 4.2e-5
        return {"rel": 1e-4, "max": 2e-4, "differ": 5e-3}
    if kind == "generate":
        return {"rel": 0.0, "differ": 1e-2}
    return {"rel": 2e-6, "max": 1e-5, "differ": 2e-3}      # fp32 sums over the vocabulary: rel 1.5e-7, max 5e-7

"""Algorithm 1 (the DualDiffusion loop) as host-side orchestration of the library's calls.

The drafter and the verifier are callables supplied by the user (the models themselves are
not part of this library): each maps the current token tensor [B,P] (int32, on the device)
to logits [B,P,V] (bfloat16, on the device).  Every step of the algorithm that touches logits
runs in the CUDA library: ``dd_unmask`` for the drafter's K unmasking steps, ``dd_verify`` for
the verification algorithm A.  What is left here is the control flow of Algorithm 1: which
positions are masked, which were decoded by the drafter in the current cycle, and when to stop.

The host waits for the device once a cycle, for the number of positions that are masked in each
sequence.  Within the drafting phase it knows how many are left without looking, as long as the
unmasking rule is a fixed number per step; only under a confidence threshold, which may unmask more,
does it ask after every step.  (Four sequences of 128 tokens, 30 drafter calls in 7 cycles: 4.3-4.6 ms
with four waits a step, 1.65 now.)
"""
from __future__ import annotations

from dataclasses import dataclass, field

from . import binding as dd


@dataclass
class LoopStats:
    cycles: int = 0
    drafter_calls: int = 0
    verifier_calls: int = 0
    unmasked_by_drafter: int = 0
    remasked_by_verifier: int = 0
    masked_after_cycle: list = field(default_factory=list)


def dualdiffusion_generate(drafter, verifier, tokens, mask_id, K, mode, tau, k, seed=0,
                           unmask_tau=float("inf"), unmask_k=1, max_cycles=10_000):
    """Runs Algorithm 1 until no position holds ``mask_id`` (or ``max_cycles`` is reached).

    tokens: int32 [B,P] device tensor, ``mask_id`` where a token is still to be generated.
    K: drafter steps per cycle.  mode, tau, k, seed: as for ``dd_verify`` (the verification
    algorithm and its threshold, minimum-keep count and Philox seed; the seed is advanced by
    one per cycle).  unmask_tau, unmask_k: the drafter's unmasking rule as for ``dd_unmask``.
    In KL mode the drafter is evaluated once more on the drafted sequence, which is the
    distribution Eq. 5 names.  Returns (tokens, LoopStats).
    """
    import torch
    x = tokens.clone()
    stats = LoopStats()
    algo = mode & 0xFF
    fixed_number = unmask_tau == float("inf")          # no confidence reaches the threshold
    # positions of each sequence that hold mask_id: on the device as flags, and counted on the host
    masked = x == mask_id
    left = masked.sum(dim=1).tolist()
    while stats.cycles < max_cycles and any(left):
        # ---- drafting phase: K unmasking steps of the fast model
        flags = still = masked.view(torch.uint8)
        for step in range(K):
            if step > 0 and not fixed_number and any(left):
                left = [1] if bool(still.any()) else [0]
            if not any(left):
                break
            logits_d = drafter(x)
            stats.drafter_calls += 1
            x, still, _ = dd.unmask(logits_d, x, still, unmask_tau, unmask_k)
            if fixed_number:
                left = [max(0, n - unmask_k) for n in left]
        drafted = flags - still                        # 1 where a mask of this cycle's start is gone
        # ---- verification phase: one step of the accurate model over the drafted positions
        logits_v = verifier(x)
        stats.verifier_calls += 1
        logits_d = None
        if algo == dd.DD_MODE_KL:
            logits_d = drafter(x)
            stats.drafter_calls += 1
        out_tokens, remask, _ = dd.verify(logits_d, logits_v, x, drafted, mode, tau, k, seed + stats.cycles)
        x = out_tokens.masked_fill(remask.view(torch.bool), mask_id)
        masked = x == mask_id
        left, n_drafted, n_remasked = torch.stack((masked.view(torch.uint8), drafted, remask)).sum(dim=2).tolist()
        stats.unmasked_by_drafter += sum(n_drafted)
        stats.remasked_by_verifier += sum(n_remasked)
        stats.cycles += 1
        stats.masked_after_cycle.append(sum(left))
    return x, stats

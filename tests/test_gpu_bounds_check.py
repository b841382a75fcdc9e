"""A sample of the parity cases through the bounds-checked build of the library
(-DDD_BOUNDS_CHECK: every index the verification kernels form into a caller's tensor or into the
library's scratch is compared with its extent; a violation is recorded in the health word and
index 0 is used instead).  No memory checker can be run on these kernels here, so this build,
the guard regions around every output and the grid-size invariance tests are what speaks for
their addressing.  The checked build must report nothing and give the normal build's bits."""
import numpy as np
import pytest

from paper_2604_05250_b200 import synth
from tests._parity import off_vector_boundary, to_torch_bf16

pytestmark = pytest.mark.gpu

TRUST, KL, CONF, PROB, EMIT = 0, 1, 2, 0x100, 0x200


@pytest.fixture(scope="module")
def libs():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_05250_b200 import binding, build
    build.build()
    return binding, build.build_check()


def fresh_outputs(B, P):
    import torch
    return dict(out_tokens=torch.empty(B, P, dtype=torch.int32, device="cuda"),
                out_mask=torch.empty(B, P, dtype=torch.uint8, device="cuda"),
                out_score=torch.empty(B, P, dtype=torch.float32, device="cuda"))


def both_builds(binding, check_path, call):
    """call() under the normal and under the checked build; the checked one must stay silent."""
    import torch
    normal = [x.cpu().numpy() for x in call()]
    torch.cuda.synchronize()
    assert binding.verify_status() == 0
    with binding.use_library(check_path):
        checked = [x.cpu().numpy() for x in call()]
        torch.cuda.synchronize()
        word = binding.verify_status()
        assert word == 0, f"bounds-checked build recorded {word:#x} (site {(word >> 8) & 0xF}, CTA {word & 0xFF})"
    for a, b in zip(normal, checked):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("B,P,V,flagged,mode", [
    # the row kernel
    (1, 128, 1024, 32, KL),                      # cfg0
    (2, 96, 20000, 61, KL | PROB),               # two CTAs a row, ragged last piece
    (3, 40, 126464, 33, CONF),                   # the LLaDA vocabulary
    (1, 20, 126464, 20, KL),                     # clusters of eight
    (2, 50, 1003, 31, KL),                       # rows off vector boundaries
    (15, 700, 64, 380, CONF | PROB),             # many short rows, sequences beyond the short decision
    (1, 1500, 4104, 900, TRUST | EMIT),          # a sequence beyond the short decision
    (4, 8, 8, 0, KL),                            # nothing flagged: every sequence passes through
    # its deep form, flagged rows first
    (2, 200, 65000, 150, KL | PROB),
    (2, 200, 65003, 150, KL),
    # the streaming kernel: rows cut by range boundaries, on and off vector boundaries; short rows, several rounds
    (4, 200, 65000, 150, KL | PROB),
    (4, 200, 65003, 150, KL),
    (4, 256, 65003, 40, CONF),
    (60, 700, 64, 500, KL),
    (24, 1500, 37, 900, CONF | PROB),
    (6, 6000, 1003, 0, KL),
])
def test_verify_addresses_stay_inside(libs, B, P, V, flagged, mode):
    import torch
    binding, check_path = libs
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, flagged, 0.2, seed=P + V)
    t = [to_torch_bf16(dra, "cuda") if (mode & 0xFF) == KL else None, to_torch_bf16(ver, "cuda"),
         torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()]
    both_builds(binding, check_path, lambda: binding.verify(t[0], t[1], t[2], t[3], mode, 0.5, 4, 9))


@pytest.mark.parametrize("B,P,V,flagged,mode", [
    (2, 50, 1003, 31, KL), (1, 24, 20000, 17, CONF), (1, 1900, 203, 1000, KL | PROB), (1, 2500, 203, 1200, CONF),
])
@pytest.mark.parametrize("static", [False, True])
def test_element_wise_kernel(libs, B, P, V, flagged, mode, static):
    """Logits off 16-byte boundaries, sequences inside its key area and beyond it, both scratches."""
    import torch
    binding, check_path = libs
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, flagged, 0.2, seed=P + V)
    t = [off_vector_boundary(dra) if (mode & 0xFF) == KL else None, off_vector_boundary(ver),
         torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()]
    both_builds(binding, check_path, lambda: binding.verify(t[0], t[1], t[2], t[3], mode, 0.5, 4, 9, static_scratch=static,
                                                            **(fresh_outputs(B, P) if static else {})))


@pytest.mark.parametrize("B,P,V,flagged", [(2, 96, 20000, 61), (2, 200, 65003, 150), (4, 200, 65003, 150)])      # row kernel, its deep form, streaming kernel
def test_static_scratch_and_unmask(libs, B, P, V, flagged):
    import torch
    binding, check_path = libs
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, flagged, 0.2, seed=3)
    t = [to_torch_bf16(dra, "cuda"), to_torch_bf16(ver, "cuda"), torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()]
    both_builds(binding, check_path, lambda: binding.verify(t[0], t[1], t[2], t[3], KL, 0.5, 4, 9, static_scratch=True,
                                                            **fresh_outputs(B, P)))
    both_builds(binding, check_path, lambda: binding.unmask(t[1], t[2], t[3], 0.3, 2))


@pytest.mark.parametrize("B,P,K,V", [(2, 300, 128, 4100), (3, 700, 64, 20000), (1, 300, 64, 40000)])        # every row; flagged rows only; kernel chosen on the device
@pytest.mark.parametrize("mode", [CONF | PROB, KL])
def test_fused_heads(libs, mode, B, P, K, V):
    import torch
    binding, check_path = libs
    dh, dw, vh, vw, tokens, flags = synth.lm_head_pair_inputs(B, P, K, V, "uniform_25_100", 0.2, seed=8)
    t = [to_torch_bf16(x, "cuda") for x in (dh, dw, vh, vw)]
    tok, fl = torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()
    d = t[:2] if mode == KL else [None, None]
    both_builds(binding, check_path, lambda: binding.lm_head_verify(d[0], d[1], t[2], t[3], tok, fl, mode, 0.3, 3, 5))


@pytest.mark.parametrize("B,P", [(2, 37), (5, 8000)])          # row kernel; beyond its line the streaming kernel
@pytest.mark.parametrize("V", [1, 2, 3, 5, 7])
@pytest.mark.parametrize("mode", [KL, CONF])
def test_last_logits_of_rows_shorter_than_a_vector(libs, B, P, V, mode):
    """The last vector of several rows reaches beyond the tensor."""
    import torch
    binding, check_path = libs
    dra, ver, tokens, flags = synth.verify_inputs(B, P, V, P // 2, 0.2, seed=V)
    flags[-1, -9:] = 1
    t = [to_torch_bf16(dra, "cuda") if mode == KL else None, to_torch_bf16(ver, "cuda"),
         torch.from_numpy(tokens).cuda(), torch.from_numpy(flags).cuda()]
    both_builds(binding, check_path, lambda: binding.verify(t[0], t[1], t[2], t[3], mode, 0.5, 4, 9))

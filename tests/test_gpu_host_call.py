"""The native host side of the calls against its Python form: same results, same errors."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dd():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_05250_b200 import binding, build
    build.build()
    binding.lib()
    assert binding._fast is not None
    return binding


def calls(dd):
    """One call of every wrapper that has a native form, with and without its optional arguments."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    q, k, v, blk, inter = r(2, 3, 70, 64), r(2, 3, 70, 64), r(2, 3, 70, 64), r(2, 3, 9, 64), r(2, 9, 3, 64)
    ki, vi = r(2, 70, 3, 64), r(2, 70, 3, 64)
    lens = torch.tensor([70, 33], dtype=torch.int32, device="cuda")
    d, ve = r(2, 40, 999), r(2, 40, 999)
    tok = torch.randint(0, 999, (2, 40), device="cuda", generator=g, dtype=torch.int32)
    fl = (torch.rand(2, 40, device="cuda", generator=g) < 0.6).to(torch.uint8)
    new = lambda: dict(out_tokens=torch.empty_like(tok), out_mask=torch.empty_like(fl), out_score=torch.empty(2, 40, device="cuda"))
    return [
        lambda: dd.bidir_attention(q, k, v),
        lambda: dd.bidir_attention(q, k, v, out=torch.empty_like(q), scale=0.25),
        lambda: dd.block_attention(blk, k, v, kv_len=lens),
        lambda: dd.block_attention(inter, ki, vi, layout="bnhd", scale=0.25, out=torch.empty_like(inter)),
        lambda: dd.verify(d, ve, tok, fl, dd.DD_MODE_KL | dd.DD_FLAG_PROBABILISTIC, 0.5, 3, 2 ** 63 + 5),
        lambda: dd.verify(None, ve, tok, fl, dd.DD_MODE_CONF, 0.01, 3, -1, want_score=False),
        lambda: dd.verify(d, ve, tok, fl, dd.DD_MODE_KL, 0.5, 3, 0, static_scratch=True, **new()),
        lambda: dd.unmask(ve, tok, fl, float("inf"), 4),
    ]


def test_same_results(dd, monkeypatch):
    import torch
    native = [c() for c in calls(dd)]
    monkeypatch.setattr(dd, "_fast", None)
    for a, b in zip(native, [c() for c in calls(dd)]):
        for x, y in zip(*((t if isinstance(t, tuple) else (t,)) for t in (a, b))):
            assert (x is None and y is None) or (x.dtype == y.dtype and torch.equal(x, y))
    side = torch.cuda.Stream()                        # the current stream is the one that counts
    monkeypatch.undo()
    with torch.cuda.stream(side):
        other = calls(dd)[4]()
    side.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(other, native[4]))


def test_same_errors(dd, monkeypatch):
    import torch
    q = torch.zeros(1, 2, 16, 64, dtype=torch.bfloat16, device="cuda")
    l3 = torch.zeros(1, 4, 64, dtype=torch.bfloat16, device="cuda")
    tok, fl = torch.zeros(1, 4, dtype=torch.int32, device="cuda"), torch.ones(1, 4, dtype=torch.uint8, device="cuda")
    bad = [
        lambda: dd.bidir_attention(q, q.float(), q),
        lambda: dd.bidir_attention(q, q, q.transpose(2, 3)),
        lambda: dd.bidir_attention(q, q.cpu(), q),
        lambda: dd.bidir_attention(q, q, [1]),
        lambda: dd.bidir_attention(q, q, q, scale=float("nan")),
        lambda: dd.bidir_attention(q[..., :32].contiguous(), q[..., :32].contiguous(), q[..., :32].contiguous()),
        lambda: dd.block_attention(q, q, q, layout="other"),
        lambda: dd.block_attention(q, q, q, kv_len=tok),
        lambda: dd.verify(None, l3, tok, fl, dd.DD_MODE_KL, 0.5, 0, 0),
        lambda: dd.verify(None, l3, tok.long(), fl, dd.DD_MODE_CONF, 0.5, 0, 0),
        lambda: dd.verify(None, l3, tok, fl, 7, 0.5, 0, 0),
        lambda: dd.verify(None, l3, tok, fl, dd.DD_MODE_CONF, float("nan"), 0, 0),
        lambda: dd.unmask(l3, tok, fl, 0.5, -1),
        lambda: dd.unmask(l3, tok[:, :3], fl, 0.5, 1),
    ]

    def outcome(call):
        with pytest.raises(Exception) as e:
            call()
        return type(e.value), str(e.value)
    native = [outcome(c) for c in bad]
    monkeypatch.setattr(dd, "_fast", None)
    assert [outcome(c) for c in bad] == native


def test_what_is_left_to_the_python_form(dd, monkeypatch):
    """Wrapped tensors, a torch function mode and an allocation that fails: as without the native side."""
    import torch
    from torch.overrides import TorchFunctionMode
    q = torch.zeros(2, 2, 16, 64, dtype=torch.bfloat16, device="cuda")

    class Seen(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            names.append(getattr(func, "__name__", str(func)))
            return func(*args, **(kwargs or {}))

    def no_memory():
        big = torch.empty(64, 32, 2048, 64, dtype=torch.bfloat16, device="cuda")
        torch.cuda.empty_cache()
        total = torch.cuda.get_device_properties(0).total_memory
        torch.cuda.set_per_process_memory_fraction(torch.cuda.memory_reserved() / total)
        try:
            dd.bidir_attention(big, big, big)
        finally:
            torch.cuda.set_per_process_memory_fraction(1.0)

    def outcomes():
        seen = []
        with pytest.raises(RuntimeError) as e:
            torch.vmap(lambda t: dd.bidir_attention(t[None], t[None], t[None]))(q)
        seen.append(str(e.value))
        with pytest.raises(torch.OutOfMemoryError):
            no_memory()
        names.clear()
        with Seen():
            dd.bidir_attention(q, q, q)
        return seen, sorted(set(names))
    names = []
    native = outcomes()
    assert "empty_like" in native[1]
    monkeypatch.setattr(dd, "_fast", None)
    assert outcomes() == native

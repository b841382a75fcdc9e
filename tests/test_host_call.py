"""The native host side of the calls without a GPU: what it leaves to the Python form."""
import glob
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

ROOT = __file__.rsplit("/tests/", 1)[0]


@pytest.mark.parametrize("with_out", [True, False])
def test_fake_tensors_raise(with_out):
    """Tensors without memory behind them raise, as they do in the Python form (a process of its own: an exception
    that crosses code running without the GIL ends it)."""
    code = f"""
        import torch
        from torch._subclasses.fake_tensor import FakeTensorMode
        from paper_2604_05250_b200 import binding as dd, build
        build.build()
        dd.lib()
        assert dd._fast is not None
        with FakeTensorMode():
            t = lambda *s, dtype=torch.bfloat16: torch.empty(*s, dtype=dtype, device="cuda")
            q, l3, tok, fl = t(1, 2, 16, 64), t(1, 4, 64), t(1, 4, dtype=torch.int32), t(1, 4, dtype=torch.uint8)
            score = t(1, 4, dtype=torch.float32)
        given = {with_out}
        out = dict(out=q) if given else dict()
        dec = dict(out_tokens=tok, out_mask=fl) if given else dict()
        calls = [lambda: dd.bidir_attention(q, q, q, **out), lambda: dd.block_attention(q, q, q, **out),
                 lambda: dd.verify(l3, l3, tok, fl, dd.DD_MODE_KL, 0.5, 1, 0, **dec, **(dict(out_score=score) if given else dict())),
                 lambda: dd.unmask(l3, tok, fl, 0.5, 1, **dec, **(dict(out_conf=score) if given else dict()))]
        said = []
        for native in (dd._fast, None):
            dd._fast = native
            for c in calls:
                try:
                    c()
                    raise SystemExit("no error")
                except Exception as e:
                    said.append((type(e), str(e)))
        assert said[:4] == said[4:], said
        assert all(kind is RuntimeError for kind, text in said), said
        print("same errors")
    """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same errors" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])


@pytest.mark.parametrize("compiler", [True, False])
def test_module_built_after_the_binding_was_imported(tmp_path, compiler):
    """In a clean checkout build.build() gives an imported binding its native side; without a C++ compiler it warns,
    and the Python form serves."""
    from paper_2604_05250_b200 import build
    build.build()
    pkg = tmp_path / "paper_2604_05250_b200"
    shutil.copytree(os.path.join(ROOT, "paper_2604_05250_b200"), pkg, ignore=shutil.ignore_patterns("*.so", "__pycache__"))
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    shutil.copy(build.LIB, pkg)                                  # newer than its sources: only the module is missing
    env = dict(os.environ, PYTHONPATH=str(tmp_path))
    if not compiler:
        (tmp_path / "bin").mkdir()
        env["PATH"] = str(tmp_path / "bin")
    code = f"""
        import warnings
        from paper_2604_05250_b200 import binding, build
        assert binding.__file__.startswith({str(tmp_path)!r}) and binding._fast is None
        with warnings.catch_warnings(record=True) as seen:
            warnings.simplefilter("always")
            build.build()
        binding.lib()
        assert (binding._fast is not None) == {compiler} and any("native host side" in str(w.message) for w in seen) != {compiler}
        print("as it should be")
    """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=tmp_path, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "as it should be" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])
    assert len(glob.glob(str(pkg / "_host_call-*.so"))) == int(compiler)

"""The native calls of the binding (`_pycall`) take every argument that is no plain tensor as an error, never as the end of the
process.  Each case runs in a process of its own; the context is NULL, so nothing is ever launched."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes, sys, types
import torch
from paper_2408_15562_b200 import binding
what = sys.argv[1]
bf, f32, i32 = torch.bfloat16, torch.float32, torch.int32
ctx = types.SimpleNamespace(_h=ctypes.c_void_p())
stream = types.SimpleNamespace(cuda_stream=0)
B, N, V = 1, 4, 8
def step(q):
    z = lambda *s, dtype=i32: torch.zeros(s, dtype=dtype)
    return binding.Context.verify_step_host(ctx, None, q, z(B, 2, N, 128, dtype=bf), z(B, 2, N, 128, dtype=bf), z(B, N), z(B),
        z(B, N, V, dtype=f32), None, z(B, N), z(B, dtype=f32), None, z(B, N, 2, 128, dtype=bf), z(B, N), z(B), z(B), z(B), stream=stream)
q = torch.zeros((B, N, 2, 128), dtype=bf)
def attempt():
    if what == "plain": return step(q)
    if what == "vmap": return torch.vmap(lambda x: step(x) and x)(q[None])
    if what == "grad": return torch.func.grad(lambda x: (step(x.to(bf)), x.sum())[1])(q.float())
    if what == "fake":
        from torch._subclasses.fake_tensor import FakeTensorMode
        with FakeTensorMode() as m: return step(m.from_tensor(q))
    if what == "functional": return step(torch._to_functional_tensor(q))
    if what == "meta": return step(q.to("meta"))
    if what == "sparse": return step(q.to_sparse())
    if what == "nested": return step(torch.nested.nested_tensor([q[0], q[0]]))
    if what == "mkldnn": return step(q.float().to_mkldnn())
    if what == "array": return step(types.SimpleNamespace(shape=q.shape, dtype=bf))
    if what == "deleted": q.untyped_storage().resize_(0); return step(q)
try:
    attempt()
    print("returned")
except Exception as e:
    print(type(e).__name__, str(e).splitlines()[0] if str(e) else "")
"""


@pytest.mark.parametrize("what,want", [
    ("plain", "FspadError"),           # the NULL context, reported by the library
    ("vmap", "RuntimeError"), ("grad", ""), ("fake", ""), ("functional", ""), ("meta", "ValueError"), ("sparse", ""),
    ("nested", ""), ("mkldnn", ""), ("array", "TypeError"), ("deleted", "FspadError"),
])
def test_an_argument_without_ordinary_storage_raises(what, want):
    r = subprocess.run([sys.executable, "-c", SCRIPT, what], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    assert "Error" in r.stdout and r.stdout.startswith(want), r.stdout


def test_calls_built_for_another_torch_are_not_loaded(monkeypatch):
    import torch

    from paper_2408_15562_b200 import binding, build
    build.build()
    assert binding._calls() is not None and torch.__version__ in build.calls_path()
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.raises(RuntimeError, match="missing"):
        binding._calls()

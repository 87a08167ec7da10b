"""The linears' native marshalling away from a GPU: tensors that cannot say their size or address are refused with -1, for the Python code to
name the error, and end no process; without the module the library loads all the same; and it is built again for another torch."""
import os
import subprocess
import sys

from paper_2602_02711_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import torch
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import binding
from torch._subclasses.fake_tensor import FakeTensorMode
from torch.fx.experimental.symbolic_shapes import ShapeEnv

dmr.lib()
calls, env = binding._calls, ShapeEnv()
with FakeTensorMode(shape_env=env):  # tensors on a GPU, as far as anyone can ask, without one
    n = env.create_unbacked_symint()
    bf16 = dict(dtype=torch.bfloat16, device="cuda")
    W, Y, ws = torch.empty(128, 128, **bf16), torch.empty(4, 128, **bf16), torch.empty(512, dtype=torch.uint8, device="cuda")
    odd, bytes_ = torch.empty(n, 128, **bf16), torch.empty(n, dtype=torch.uint8, device="cuda")
    q = (W, W, W, 128, 128, 4, 64)
    asked = {"X": lambda: calls.dense(odd, W, Y, 0, ws, 0), "W": lambda: calls.dense(W, odd, Y, 0, ws, 0), "Y": lambda: calls.dense(W, W, odd, 0, ws, 0),
         "workspace": lambda: calls.dense(W, W, Y, 0, bytes_, 0), "lowbit": lambda: calls.lowbit(odd, *q, Y, 0, ws, 0),
         "mask": lambda: calls.routed(W, bytes_, W, *q, Y, 0, ws, 0), "number": lambda: calls.dense(W, 3, Y, 0, ws, 0),
         "stream": lambda: calls.dense(W, W, Y, 0, ws, "no stream"), "count": lambda: calls.dense(W)}
    for name, ask in asked.items():
        print(name, flush=True)
        assert ask() == -1, name
"""


def test_arguments_that_throw_are_refused():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.stdout.split()[-1:], r.stderr[-2000:])


def test_the_library_loads_without_the_module():
    script = """
import sys, warnings
sys.modules["paper_2602_02711_b200._calls"] = None  # an import of it fails
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import binding
with warnings.catch_warnings(record=True) as said:
    warnings.simplefilter("always")
    assert dmr.lib().dmr_workspace_bytes(0, 1, 128, 128, dmr.QFormat(4, 64)) > 0 and binding._calls is None
assert len(said) == 1 and "build" in str(said[0].message)
"""
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


def test_the_module_is_stale_for_another_torch(monkeypatch, tmp_path):
    stamp = tmp_path / "calls.txt"
    monkeypatch.setattr(build, "CALLS_STAMP", str(stamp))
    monkeypatch.setattr(build, "_stale", lambda target, deps: False)
    assert build.needs_build()  # nobody knows what it was built for
    stamp.write_text(build._calls_made_for())
    assert not build.needs_build()
    monkeypatch.setattr(build.metadata, "version", lambda name: "99.0")
    assert build.needs_build()

"""The native half of the binding with tensors that have no strides or memory of their own: an exception, not the end of
the process.  They run in a process of their own, so that an abort is a failed test."""
import os
import subprocess
import sys
import types

import pytest
import torch

from paper_2609_40335_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import sys, torch
sys.path.insert(0, %r)
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2609_40335_b200 import binding as dp, build
build.build_marshal()
nested = torch.nested.nested_tensor([torch.ones(2, 3), torch.ones(4, 3)])       # strides() throws
with FakeTensorMode():
    fake = torch.empty(2, 3, 8, device="cuda")            # says it is on a GPU; inside vmap data_ptr() throws

def refused(f):
    try:
        f()
    except Exception as e:
        print("refused:", type(e).__name__, str(e)[:80])
    else:
        sys.exit("accepted")

def in_vmap(f):
    torch.func.vmap(lambda x: (refused(lambda: f(x)), x)[1])(fake)

def step(x, layers, outs):
    tensors = dict.fromkeys("ids G_emb pos_ids wte wpe sq clip norms cross side_sq perm seg pos_perm pos_seg ws side_ws "
                            "dev_status".split(), x)
    dp.dp_step_enqueue(layers, outs, [0] * len(layers), [], [], [], stream=1, side_stream=2, events=[3, 4, 5, 6], V=8, d=8,
                       tied=False, noise=False, C_=1.0, sigma=1.0, seed=0, step=0, wte_id=0, wpe_id=0, **tensors)
""" % ROOT

CASES = """
refused(lambda: dp._descs([dp.Linear(nested, nested)]))
refused(lambda: dp._vdescs([dp.Vector(nested)]))
refused(lambda: step(nested, [], []))
refused(lambda: step(nested, [dp.Linear(nested, nested)], [nested]))
in_vmap(lambda x: dp._descs([dp.Linear(x, x)]))
in_vmap(lambda x: dp._vdescs([dp.Vector(x, x)]))
in_vmap(lambda x: dp._outputs([x]))
in_vmap(lambda x: step(x, [], []))
in_vmap(lambda x: step(x, [dp.Linear(x, x)], [x]))
"""


def test_tensors_without_memory_are_refused():
    r = subprocess.run([sys.executable, "-c", HEAD + CASES], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout[-500:], r.stderr[-800:])
    assert r.stdout.count("refused:") == 9


def test_extension_of_another_torch_is_built_again_and_never_used(tmp_path, monkeypatch):
    commands = []

    def compile_(cmd, **kw):
        commands.append(cmd)
        open(build.MARSHAL_PATH, "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(build, "MARSHAL_PATH", str(tmp_path / "_marshal.so"))
    monkeypatch.setattr(build, "MARSHAL_STAMP", str(tmp_path / "build" / "marshal.stamp"))
    monkeypatch.setattr(build.subprocess, "run", compile_)
    for expected in (1, 1):
        build.build_marshal()
        assert len(commands) == expected
    version = torch.__version__
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    build.build_marshal()
    assert len(commands) == 2
    monkeypatch.setattr(torch, "__version__", version)
    monkeypatch.setattr(binding, "_native", None)
    assert binding._marshal().torch_version == version
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.raises(binding.DpGhostError, match="built for torch"):
        binding._marshal()

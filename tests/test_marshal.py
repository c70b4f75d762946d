"""The binding's native marshalling: what it does not take it leaves to the binding's own checks, and nothing that torch
throws inside it ends the process."""
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import build as speca_build
from paper_2607_16673_b200 import synth

# each in a process of its own: an exception that leaves a C function ends it
NO_TENSORS = """
speca.decode_step(speca.Dims(1, 1, 1, 64, 64), *[None] * 7)         # without a GPU there is no stream either
"""
WITHOUT_STORAGE = """
from torch._subclasses.fake_tensor import FakeTensorMode
with FakeTensorMode():
    def make(*shape, dtype=torch.float32):
        return torch.empty(*shape, dtype=dtype, device="cuda")
    S, o, gate = make(1, 1, 1, 64, 64), make(1, 1, 1, 64), make(1, 1, 1)
    rec = make(1, 1, 1, 64, dtype=torch.bfloat16)
    speca.decode_step(speca.Dims(1, 1, 1, 64, 64), S, rec, rec, rec, gate, gate, o)
"""


@pytest.mark.parametrize("call", [NO_TENSORS, WITHOUT_STORAGE], ids=["no tensors", "without storage"])
def test_what_torch_throws_is_an_ordinary_exception(call):
    speca_build.build()
    code = ("import torch\nfrom paper_2607_16673_b200 import binding as speca\nspeca._load_native()\ntry:\n"
            + "\n".join("    " + line for line in call.strip().splitlines())
            + "\nexcept Exception as e:\n    print('raised', type(e).__name__)\n")
    run = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr[-2000:]
    assert run.stdout.startswith("raised")


@pytest.mark.gpu
def test_a_sparse_tensor_is_refused_by_name():
    dense = torch.zeros(1, 1, 1, 64, 64, device="cuda")
    rest = [torch.zeros(1, 1, 1, 64, dtype=torch.bfloat16, device="cuda")] * 3 + [torch.zeros(1, 1, 1, device="cuda")] * 2
    with pytest.raises(Exception):
        speca.decode_step(speca.Dims(1, 1, 1, 64, 64), dense.to_sparse(), *rest, torch.zeros(1, 1, 1, 64, device="cuda"))


@pytest.mark.gpu
def test_numpy_integers_and_whole_thresholds_are_taken_natively():
    native = speca._load_native()
    i32 = dict(dtype=torch.int32, device="cuda")
    offs = torch.tensor([0, 2, 4], **i32)
    parent, logp = torch.tensor([-1, 0, -1, -1], **i32), torch.zeros(4, device="cuda")
    out = [torch.zeros(3, **i32), torch.zeros(4, **i32), torch.zeros(4, **i32)]
    status = torch.zeros(1, **i32)
    assert native.prune_tree(np.int64(2), 5, np.int32(2), offs, parent, logp, *out, status) == 0
    assert out[0].tolist() == [0, 2, 4] and out[1].tolist() == [-1, 0, -1, -1] and int(status) == 0
    # a number that int() has to convert first is the binding's
    assert native.prune_tree(2.0, 5.0, 2, offs, parent, logp, *out, status) is None
    speca.prune_tree(2.0, 5.0, 2, offs, parent, logp, *out, status)


def test_another_torch_does_not_load_this_binary(tmp_path):
    """The marshalling reads torch's and Python's objects directly: its file carries both versions in its name, and under
    another version it is missing, not misread."""
    speca_build.build()
    assert torch.__version__ in speca.MARSHAL_PATH
    code = ("import torch\ntorch.__version__ = '0.0.1'\nfrom paper_2607_16673_b200 import binding as speca\ntry:\n"
            "    speca._load_native()\nexcept speca.SpecaError as e:\n    print('refused', e)\n")
    run = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and run.stdout.startswith("refused") and "build" in run.stdout, run.stderr[-2000:]

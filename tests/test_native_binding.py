"""The native half of the binding refuses what it cannot hand to a kernel, before anything is launched (no GPU needed:
a CPU tensor is one of the things it refuses)."""
import os
import subprocess
import sys

import pytest
import torch

import paper_2510_07535_b200 as pkg
from paper_2510_07535_b200 import binding
from paper_2510_07535_b200 import build as owl_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def native():
    owl_build.build()
    pkg.load_library()
    return binding._native


@pytest.mark.parametrize("args,message", [
    ((0, 0), "expected 10 arguments"),
    ((0, 0, b"short") + (None,) * 7, "OwlDims"),
    ((0, 0, bytes(pkg.OwlDims(1, 1, 1))) + (None,) * 7, "OwlDims"),
    ((0, 0, pkg.OwlDims(), [1.0]) + (None,) * 6, "k_cache: expected a tensor"),
    ((0, 0, pkg.OwlDims(), torch.zeros(4, dtype=torch.bfloat16)) + (None,) * 6, "k_cache: expected contiguous torch.bfloat16 tensor on cuda:0"),
    ((None, 0, pkg.OwlDims()) + (None,) * 7, ""),
])
def test_bad_arguments_raise_type_errors(native, args, message):
    with pytest.raises(TypeError, match=message):
        native.kv_commit(*args)


def test_what_torch_throws_is_an_exception(native):
    """A device that is not there ends in an error of the call.  (In a process of its own: an exception that nobody catches
    would end it.)"""
    code = """
import paper_2510_07535_b200 as pkg
from paper_2510_07535_b200 import binding
pkg.load_library()
try:
    binding._native.kv_commit(0, 99, pkg.OwlDims(), *(None,) * 7)
except RuntimeError:
    print("raised")
"""
    run = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT)
    assert run.returncode == 0 and run.stdout.startswith("raised"), run.stdout + run.stderr[-2000:]


@pytest.mark.parametrize("value", [2 ** 32 - 1, -1, 2 ** 70 + 5])
def test_integers_are_taken_modulo_2_to_the_32(native, value):
    """As ctypes takes an int32: nothing that used to be accepted is refused for its size (the call itself fails later, for
    the missing tensors)."""
    with pytest.raises(TypeError, match="node_offsets: expected a tensor"):
        native.prepare_spec_tree(0, 0, pkg.OwlDims(), value, 1, *(None,) * 8)

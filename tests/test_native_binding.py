"""The native half of the binding refuses what it cannot hand to a kernel, before anything is launched (no GPU needed:
a CPU tensor is one of the things it refuses)."""
import pytest
import torch

import paper_2510_07535_b200 as pkg
from paper_2510_07535_b200 import binding
from paper_2510_07535_b200 import build as owl_build


@pytest.fixture(scope="module")
def native():
    owl_build.build()
    pkg.load_library()
    return binding._native


@pytest.mark.parametrize("args,message", [
    ((0, 0), "expected 10 arguments"),
    ((0, 0, b"short") + (None,) * 7, "OwlDims"),
    ((0, 0, pkg.OwlDims(), [1.0]) + (None,) * 6, "k_cache: expected a tensor"),
    ((0, 0, pkg.OwlDims(), torch.zeros(4, dtype=torch.bfloat16)) + (None,) * 6, "k_cache: expected contiguous torch.bfloat16 tensor on cuda:0"),
    ((None, 0, pkg.OwlDims()) + (None,) * 7, ""),
])
def test_bad_arguments_raise_type_errors(native, args, message):
    with pytest.raises(TypeError, match=message):
        native.kv_commit(*args)

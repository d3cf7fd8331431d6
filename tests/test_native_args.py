"""Argument checks of the marshalling extension (no GPU: every case is refused before the library is called)."""
import types

import pytest
import torch

from paper_2609_34054_b200 import binding, inputs as I


@pytest.fixture(scope="module")
def native():
    from paper_2609_34054_b200 import build
    build.build()
    binding.load_library()
    return binding._native


@pytest.mark.parametrize("what", ["host tensor", "none where required", "not a descriptor", "not a tensor", "argument count"])
def test_bad_arguments_raise(native, what):
    desc, H = binding.layer_desc(I.C1), torch.zeros(4, I.C1.d_model, dtype=torch.bfloat16)
    cache = types.SimpleNamespace(k_base=None, v_base=None, lr_k=None, lr_v=None, n_blocks=1)
    args = [0, desc, H, None, cache, 0, None, 1]
    if what == "none where required":
        args[2] = None
    elif what == "not a descriptor":
        args[1] = b"short"
    elif what == "not a tensor":
        args[2] = [1, 2]
    elif what == "argument count":
        args.pop()
    with pytest.raises(TypeError if what == "argument count" else binding.PreccError):
        native.turn_project(*args)

"""Argument checks of the marshalling extension (no GPU: every case is refused before the library is called)."""
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
    args = [0, desc, H, None, _NO_CACHE, 0, None, 1]
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


def _fake(*shape):
    """A tensor that says it lies on a GPU and has no storage: its sizes can be read, there is nothing at its address."""
    from torch._subclasses import FakeTensorMode
    with FakeTensorMode():
        return torch.empty(shape, dtype=torch.float32, device="cuda")


_NO_CACHE = binding.Cache.__new__(binding.Cache)
_NO_CACHE.__dict__.update(k_base=None, v_base=None, lr_k=None, lr_v=None, n_blocks=1)


def _valid(call):
    """Arguments of `call` that pass the marshalling up to the look-up of the stream."""
    desc, x, table = binding.layer_desc(I.C1), _fake(4, 2, 64), _fake(4, 8)
    project = [0, desc, x, x, _NO_CACHE, 0, None, 1]
    rope, decode = _fake(64, 32, 2), [0, desc, x, None, None, 64, None, None]
    prefill = [0, desc, x, 0, 64, None, None]
    return {"turn_project": project, "lr_precompute": project, "rebase_project": project[:7],
            "turn_project_rows": [0, desc, x, x, _NO_CACHE, None, None, None],
            "rebase_project_rope": [0, desc, x, x, _NO_CACHE, rope, None, 0, 0, None],
            "turn_project_rope": [0, desc, x, x, _NO_CACHE, rope, None, 0, 0, None, 1],
            "lr_attend_decode": decode + [_NO_CACHE, x, x, table, None],
            "lr_attend_decode_rope": decode + [rope, _NO_CACHE, x, x, table, None],
            "lr_attend_decode_static": decode + [_NO_CACHE, x, table, None],
            "lr_attend_decode_partial": decode[:7] + [_NO_CACHE, x, x, table, None],
            "combine_partials": [0, desc, x, None, None, x],
            "lr_attend_prefill": prefill + [_NO_CACHE, x, table, 0],
            "lr_attend_prefill_ws": prefill + [_NO_CACHE, x, x, table, 0],
            "lr_attend_prefill_rope": prefill + [rope, _NO_CACHE, x, table, 0],
            "lr_attend_prefill_rope_scratch": prefill + [rope, _NO_CACHE, x, x, table, 0]}[call]


_CALLS = ("turn_project", "lr_precompute", "rebase_project", "turn_project_rows", "rebase_project_rope", "turn_project_rope",
          "lr_attend_decode", "lr_attend_decode_rope", "lr_attend_decode_static", "lr_attend_decode_partial", "combine_partials",
          "lr_attend_prefill", "lr_attend_prefill_ws", "lr_attend_prefill_rope", "lr_attend_prefill_rope_scratch")


@pytest.mark.parametrize("call", _CALLS)
def test_torch_exceptions_arrive_as_errors(native, call):
    """Without a device torch throws where the stream is looked up; with one the library refuses the context."""
    with pytest.raises(binding.PreccError):
        getattr(native, call)(*_valid(call))


@pytest.mark.parametrize("call", _CALLS)
def test_no_dimension_raises(native, call):
    args = _valid(call)
    args[2] = _fake()
    with pytest.raises(binding.PreccError, match="has no dimensions"):
        getattr(native, call)(*args)


@pytest.mark.parametrize("call", [c for c in _CALLS if "decode" in c])
def test_flat_block_table_of_a_batch_raises(native, call):
    args = _valid(call)
    args[-2] = _fake(8)                     # what a prefill call takes
    with pytest.raises(binding.PreccError, match="block_table must be"):
        getattr(native, call)(*args)


class _Window(binding.Cache):
    """A cache with its own idea of what the library sees of it."""

    def __init__(self, seen):
        self.seen = seen

    def desc(self):
        self.seen.append(self)
        return binding.CacheDesc(None, None, None, None, 1) if len(self.seen) < 2 else b"short"


def test_a_cache_class_of_ones_own_is_asked_for_its_descriptor(native):
    seen, args = [], _valid("turn_project")
    args[4] = _Window(seen)
    with pytest.raises(binding.PreccError):          # (the context is refused, after the descriptor has been read)
        native.turn_project(*args)
    assert len(seen) == 1
    with pytest.raises(binding.PreccError, match="CacheDesc"):
        native.turn_project(*args)
    args[4] = object()
    with pytest.raises(AttributeError, match="desc"):
        native.turn_project(*args)

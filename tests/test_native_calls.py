"""The natively marshalled calls refuse what the ctypes calls refuse (no compute: this runs without a GPU)."""
import ctypes

import pytest


class _Tensor:
    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


def _native():
    from paper_1803_09877_b200 import build
    build.build()
    from paper_1803_09877_b200 import binding
    return binding, binding._native


CALLS = {"encode": 3, "locate": 4, "decode": 4, "decode_update": 4, "locate_decode": 5}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_arguments(name):
    binding, native = _native()
    call, count = getattr(native, name), CALLS[name]
    tail = (0.5, 7) if name == "decode_update" else (7,)                    # (scale,) stream handle
    with pytest.raises(binding.DracoError, match="invalid argument"):       # no plan, as after close()
        call(*([None] * count), *tail)
    with pytest.raises(binding.DracoError, match="invalid argument"):
        call(None, *([_Tensor(4096)] * (count - 1)), *tail)
    plan = ctypes.create_string_buffer(4096)                                # refused before it is looked at: no vectors
    with pytest.raises(binding.DracoError, match="invalid argument"):
        call(ctypes.addressof(plan), *([None] * (count - 1)), *tail)
    with pytest.raises(AttributeError):
        call(None, object(), *([None] * (count - 2)), *tail)
    with pytest.raises(AttributeError):
        call(*([None] * count), *tail[:-1], object())                       # neither a handle nor a stream
    with pytest.raises(TypeError):
        call(*([None] * count))


def test_scale_has_to_be_a_number():
    _, native = _native()
    with pytest.raises(TypeError):
        native.decode_update(None, None, None, None, "1", 7)

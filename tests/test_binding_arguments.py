"""What the binding refuses and accepts before anything is launched (no device needed)."""
import ctypes

import pytest

import paper_2009_08065_b200 as bsp
from paper_2009_08065_b200 import binding


def test_descriptors_of_another_kind_are_refused():
    # eight of them hold more bytes than the one job that would be read
    chain = (binding._ChainOp * 8)()
    with pytest.raises(ctypes.ArgumentError):
        bsp.bsp_prepare_batched(chain, 16, stream=0)
    with pytest.raises(ctypes.ArgumentError):
        bsp.bsp_percentile_threshold_batched(chain, 16, [2.0] * 8, stream=0)
    with pytest.raises(ctypes.ArgumentError):
        bsp.bsp_linear_run((binding._LinearCall * 1)(), stream=0)
    with pytest.raises(ctypes.ArgumentError):
        bsp.bsp_linear_run(binding._LayerJob(), stream=0)
    with pytest.raises(bsp.BspError) as e:                    # the right kind reaches the library's own checks
        bsp.bsp_prepare_batched((binding._LayerJob * 1)(), 16, stream=0)
    assert e.value.status == -1


@pytest.mark.parametrize("stream", [0, ctypes.c_void_p(0), ctypes.c_void_p(16), ctypes.c_void_p(None)])
def test_raw_stream_handles(stream):
    """A stream may be a raw handle, as a number or as ctypes holds it: the call gets as far as the library's checks."""
    with pytest.raises(bsp.BspError) as e:
        bsp.bsp_prepare_batched((binding._LayerJob * 1)(), 16, stream=stream)
    assert e.value.status == -1


@pytest.mark.parametrize("stream", ["0", 1.5, object(), 1 << 80])
def test_other_objects_are_no_streams(stream):
    with pytest.raises((AttributeError, TypeError, OverflowError)):
        bsp.bsp_prepare_batched((binding._LayerJob * 1)(), 16, stream=stream)

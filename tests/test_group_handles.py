"""What cs_compute_group takes for a plan: handles and plain addresses, not any object with bytes (whose bytes
would be read as an address, past their end when there are fewer than eight)."""
import ctypes

import numpy as np
import pytest


@pytest.mark.parametrize("plan", [b"12345678", np.int32(3), np.uint64(3), bytearray(8), np.zeros(1)])
def test_buffers_are_not_handles(plan):
    import paper_1902_09931_gb300 as cs
    cs.load()
    for plans in ([plan], [plan, plan], [ctypes.c_void_p(None), plan]):
        with pytest.raises(TypeError):
            cs.cs_compute_group(plans, 0)


def test_null_handles_are_refused():
    import paper_1902_09931_gb300 as cs
    cs.load()
    for plans in ([ctypes.c_void_p(None)], [None], [ctypes.c_void_p(None), None]):
        with pytest.raises(cs.CSError) as e:
            cs.cs_compute_group(plans, 0)
        assert e.value.code == cs.CS_EINVAL

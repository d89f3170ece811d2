"""The time model by which calls are cut (no GPU)."""
import ctypes

import pytest


def prologue_us(streams, pieces, sms=152):
    from paper_1108_0486_gb300 import _lib as L
    try:
        fn = L.lib()._ZN2xg15cut_prologue_usEjmi
    except RuntimeError as e:  # pragma: no cover
        pytest.skip(str(e))
    fn.argtypes, fn.restype = [ctypes.c_uint32, ctypes.c_uint64, ctypes.c_int], ctypes.c_double
    return fn(streams, pieces, sms)


@pytest.mark.parametrize("pieces", [2, 3, 4, 5, 8])
def test_steps_are_priced_as_they_run(pieces):
    """Up to 191 results a step runs on the table kernel (5.5 us and 0.05 us per
    result, after 5 us of set-up), from 192 on on the tensor cores."""
    for streams in range(1, 400):
        results = streams * (pieces - 1)
        table = 5.0 + 5.5 + 0.05 * results
        assert (abs(prologue_us(streams, pieces) - table) < 1e-9) == (results < 192), (streams, results)

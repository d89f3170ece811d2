"""The binding's rows and pointers (no GPU): what reaches the C ABI is what
was given, or the call is refused before it."""
import ctypes

import numpy as np
import pytest

from paper_1108_0486_gb300 import _lib as L

ROWS = [(3, 1, 5000000000, 1 << 40), (0, 2, 7, 16), (4294967295, 0, 0, 0)]


def items(a):
    return [(x.stream, x.type, x.count, x.out or 0) for x in a]


@pytest.mark.parametrize("rows", [ROWS, tuple(ROWS), np.array(ROWS, dtype=np.uint64), np.array(ROWS, dtype=np.int64),
                                  [np.array(r, dtype=np.uint64) for r in ROWS], L.pack_rows(ROWS), L.make_requests(ROWS),
                                  L.pack_rows(ROWS[::-1])[::-1], L.pack_rows([r for r in ROWS for _ in range(2)])[::2]])
def test_rows_in_every_form(rows):
    assert items(L.make_items(rows)) == ROWS
    rec = L.make_requests(rows)
    assert rec.flags.c_contiguous and rec.itemsize == ctypes.sizeof(L.XgRequest)
    assert [tuple(int(v) for v in r) for r in rec] == ROWS


@pytest.mark.parametrize("dtype", [[("a", "<i8"), ("b", "<i8"), ("c", "<i8"), ("d", "<i8")],
                                   [("stream", "<u8"), ("type", "<u8"), ("count", "<u8"), ("out", "<u8")],
                                   [("out", "<u8"), ("count", "<u8"), ("type", "<u4"), ("stream", "<u4")],
                                   [("stream", ">u4"), ("type", ">u4"), ("count", ">u8"), ("out", ">u8")]])
def test_records_of_another_layout_are_refused(dtype):
    """Their bytes would be read as rows with other streams and addresses."""
    rec = np.zeros(4, dtype=dtype)
    for make in (L.make_items, L.make_requests):
        with pytest.raises(TypeError):
            make(rec)


@pytest.mark.parametrize("out", ["text", b"bytes", 1.5])
def test_outputs_that_are_no_address_are_refused(out):
    """Text and bytes have an address, which is not to be written to."""
    for fn in (L.xg_generate_u32, L.xg_generate_uniform, L.xg_generate_normal, L.xg_w64_generate_u64,
               L.xg_w64_generate_uniform_f64):
        with pytest.raises(TypeError):
            fn(None, 0, 1, 1, out, 1)
    with pytest.raises(TypeError):
        L.xg_generate_normal_sum(None, 0, 1, 1, out)

"""Kernel variants and dispatch rules at the sizes where they change, against
the CPU oracle: words, uniforms and 64-bit outputs bit for bit, normals within
4 ulp of the FP64 oracle rounded to FP32."""
import numpy as np
import pytest

import oracle as O
from paper_1108_0486_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KINDS = ["u32", "uniform", "normal"]


def words_of(kind, n):
    return n + (n & 1) if kind == "normal" else n


def check(kind, got, words, n):
    """got: one row's outputs; words: the oracle's words of the call."""
    words = np.asarray(words)[:words_of(kind, n)]
    if kind == "u32":
        assert np.array_equal(np.asarray(got).view(np.uint32), words)
    elif kind == "uniform":
        assert np.array_equal(got, O.uniform_of(words))
    else:
        z = O.normal_pairs64(words)[:n]
        ulp = np.spacing(np.abs(z.astype(np.float32))).astype(np.float64)
        assert float((np.abs(got.astype(np.float64) - z) / ulp).max()) <= 4.0


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("edge", [9, 18])
def test_default_launch_on_both_sides_of_its_thresholds(kind, edge):
    """Two calls (a partial last round in the first) around the stream counts
    where the default launch of a type changes; first and last streams."""
    from paper_1108_0486_gb300 import Streams
    parts = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    n = 65
    for streams in (edge * parts - 1, edge * parts):
        with Streams(streams, seeds=W.seeds(streams)) as st:
            rows = torch.cat([st.generate(kind, n), st.generate(kind, n)], 1).cpu().numpy()
        for s in (0, 1, streams - 1):
            w = O.streams(W.seeds(1, 1 + s), 2 * words_of(kind, n))[0]
            check(kind, rows[s, :n], w, n)
            check(kind, rows[s, n:], w[words_of(kind, n):], n)

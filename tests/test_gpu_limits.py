"""What calls do where something runs out -- a bounded wait, memory for the
jump tables -- or goes on beside them: a capture, another CUDA stream.  Values
against the CPU oracle or an undisturbed call, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1108_0486_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hear", ["whole call", "sum", "checkpoint", "jump", "batch", "close", "64-bit call", "64-bit close"])
def test_wait_that_runs_out_in_a_cut_call_reaches_its_owner(hear, monkeypatch):
    """One copy of a cut call's tensor-core prologue never starts (its waits
    give up after 2 s): another context's jump and batch are right and hear
    nothing of it, the next call on the failed context is refused, once, and
    reseeded it is as good as new."""
    from paper_1108_0486_gb300 import Streams, Streams64, XGError, _lib as L
    wide = hear.startswith("64-bit")
    n = 16 if wide else 64
    seeds, n_other = W.seeds(n), 200
    st = Streams64(n, seeds=seeds) if wide else Streams(n, seeds=seeds)
    (st.set_split if wide else st.set_batch_split)(4096 if wide else 32768)
    with Streams(n_other, seeds=W.seeds(n_other)) as other:
        other.set_batch_split(4096)
        torch.cuda.synchronize()
        monkeypatch.setenv("XG_TC_TEST_STALL", "1")
        st.u64(1 << 18) if wide else st.u32(1 << 18)
        monkeypatch.delenv("XG_TC_TEST_STALL")
        torch.cuda.synchronize()
        other.jump(3)
        outs = [torch.empty(32768, dtype=torch.int32, device="cuda") for _ in range(n_other)]
        other.batch([(i, "u32", 32768, o) for i, o in enumerate(outs)])
        got = other.u32(5)
        for s in (0, n_other - 1):
            w = O.streams(W.seeds(1, 1 + s), 3 + 32768 + 5)[0]
            assert np.array_equal(outs[s].cpu().numpy().view(np.uint32), w[3:-5])
            assert np.array_equal(got[s].cpu().numpy().view(np.uint32), w[-5:])
    calls = {"whole call": lambda: st.u32(10), "sum": lambda: st.normal_sum(10), "checkpoint": lambda: st.checkpoint(),
             "jump": lambda: st.jump(1), "batch": lambda: st.batch([(0, "u32", 32768, outs[0])]), "close": st.close,
             "64-bit call": lambda: st.u64(10), "64-bit close": st.close}
    with pytest.raises(XGError) as err:
        calls[hear]()
    assert err.value.status == L.XG_EDEVICE and "gave up waiting" in str(err.value)
    if hear.endswith("close"):
        assert st.ctx is None
        return
    st.seed(seeds)
    got = (st.u64(70) if wide else st.u32(70)).cpu().numpy()
    assert np.array_equal(got.view(np.uint64), O.streams64(seeds, 70)) if wide else \
        np.array_equal(got.view(np.uint32), O.streams(seeds, 70))
    st.close()


def test_wait_that_runs_out_fails_the_servers_cut_requests(monkeypatch):
    """The same in a server's batch: the request that was cut fails, the
    uncut one of the batch and a later one are right."""
    from paper_1108_0486_gb300 import Streams, XGError, _lib as L
    seeds = W.seeds(3)
    with Streams(3, seeds=seeds) as st:
        monkeypatch.setenv("XG_TC_TEST_STALL", "1")
        with st.serve(mem_cap_bytes=1 << 28, lanes=1) as srv:
            cut, small = srv.submit_many([(0, "u32", 1 << 23), (1, "u32", 1000)])
            with pytest.raises(XGError) as err:
                srv.wait(cut, 60000)
            assert err.value.status == L.XG_EDEVICE
            monkeypatch.delenv("XG_TC_TEST_STALL")
            got = srv.result(small, "u32", 1000).cpu().numpy().view(np.uint32)
            assert np.array_equal(got, O.streams(seeds[1:2], 1000)[0])
            late = srv.submit(2, "u32", 1 << 23)
            got = srv.result(late, "u32", 1 << 23).cpu().numpy().view(np.uint32)
            assert np.array_equal(got, O.streams(seeds[2:], 1 << 23)[0])


def test_cut_calls_on_two_streams_of_one_handle():
    """Cut calls of one context from two threads in turn on their per-thread
    default streams: two streams with the same handle, which nothing else
    orders (the calls are on disjoint streams of the context)."""
    from concurrent.futures import ThreadPoolExecutor
    from paper_1108_0486_gb300 import Streams, _lib as L
    per_thread = 2   # cudaStreamPerThread
    n, calls = 1 << 20, 12
    outs = [torch.empty((1, n), dtype=torch.int32, device="cuda") for _ in range(calls)]
    with Streams(2, seeds=W.seeds(2)) as st, ThreadPoolExecutor(1) as a, ThreadPoolExecutor(1) as b:
        torch.cuda.synchronize()
        L.xg_set_stream(st.ctx, per_thread)
        for k, out in enumerate(outs):
            (a, b)[k % 2].submit(st.u32, n, first=k % 2, count=1, out=out).result()
        torch.cuda.synchronize()
        L.xg_set_stream(st.ctx, torch.cuda.current_stream().cuda_stream)
        for s in range(2):
            got = torch.cat(outs[s::2], 1).cpu().numpy().view(np.uint32)[0]
            assert np.array_equal(got, O.streams(W.seeds(1, 1 + s), n * calls // 2)[0])


FIRST_BURSTS = """
import sys
import torch
from paper_1108_0486_gb300 import Streams, workloads as W
with Streams(12, seeds=W.seeds(12)) as st:
    st.u32(10)
    with st.serve(mem_cap_bytes=5 << 28, max_batch=2048, lanes=8) as srv:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        # pieces of 2^15 words, and of 2^16 beside enough words in flight; at most 2048 at once
        for sizes in ([1 << 24], [3 << 24, 1 << 24], [1 << 24, 1 << 22, 1 << 18], [1 << 20] * 10):
            tickets = [srv.submit(i, "u32", n) for i, n in enumerate(sizes)]
            for t in tickets:
                srv.wait(t, 60000)
                srv.release(t)
        print(free - torch.cuda.mem_get_info()[0])
"""


def test_first_cut_requests_allocate_nothing():
    """In a process of its own, where no matrix exists before the server:
    free device memory stays as it is from the server's start through the
    first requests of several lengths, cut into few and many pieces."""
    import subprocess
    import sys
    out = subprocess.run([sys.executable, "-c", FIRST_BURSTS], capture_output=True, text=True,
                         cwd=W.__file__.rsplit("/", 2)[0])
    assert out.returncode == 0, out.stderr
    assert out.stdout.strip() == "0"


WITHOUT_TABLES = """
import sys
import numpy as np
import torch
from paper_1108_0486_gb300 import Streams, Streams64, workloads as W
torch.zeros(1, device="cuda")
start = None
rows = []
for kind in (Streams, Streams64):
    for n in (9, 300):
        with kind(n, seeds=W.seeds(n)) as st:
            draw = st.u64 if kind is Streams64 else st.u32
            draw(77)
            if start is None:
                torch.cuda.synchronize()
                start = torch.cuda.mem_get_info()[0]
            st.jump(1 << 20)
            rows.append(draw(70))
            st.seed_substreams(5, 12)
            rows.append(draw(70))
    with kind(3, seeds=W.seeds(3)) as st:
        (st.set_split if kind is Streams64 else st.set_batch_split)(4096)
        rows += [(st.u64 if kind is Streams64 else st.u32)(1 << 18) for _ in range(2)]
calls = (1, 9, 65, 600) + (13,) * 30
with Streams(len(calls), seeds=W.seeds(len(calls))) as st:
    st.set_batch_split(64)
    for _ in range(2):
        outs = [torch.zeros(64 * k + 5, dtype=torch.int32, device="cuda") for k in calls]
        st.batch([(i, "u32", o.numel(), o) for i, o in enumerate(outs)])
        rows += [torch.cat(outs), st.u32(9)]
with Streams(2, seeds=W.seeds(2)) as st:
    with st.serve(mem_cap_bytes=1 << 28, lanes=2) as srv:
        tickets = [srv.submit(i % 2, "u32", 5 << 20) for i in range(4)]
        rows += [srv.result(t, "u32", 5 << 20) for t in tickets]
        rows = [r.cpu().numpy().reshape(-1) for r in rows]
torch.cuda.synchronize()
torch.cuda.empty_cache()
print(start - torch.cuda.mem_get_info()[0])
np.savez(sys.argv[1], *rows)
"""


def test_calls_without_memory_for_derived_tables(tmp_path):
    """Jumps, substreams, cut calls, batches and requests where no odd multiple
    and no FP4 copy of a power may be built, in a process where none exists: the
    results of a process without the limit, and no more memory kept than the
    powers (2 MiB, 33 in the 32-bit family, 24 in the other) and their scratch."""
    import os
    import subprocess
    import sys
    got = []
    for limit in ("0", "3072"):
        path = str(tmp_path / f"{limit}.npz")
        out = subprocess.run([sys.executable, "-c", WITHOUT_TABLES, path], capture_output=True, text=True,
                             cwd=W.__file__.rsplit("/", 2)[0], env=dict(os.environ, XG_JUMP_TABLE_MIB=limit))
        assert out.returncode == 0, out.stderr
        if limit == "0":
            assert int(out.stdout) <= (57 * 2 + 6) << 20
        got.append(np.load(path))
    assert len(got[0].files) == 20
    for name in got[0].files:
        assert np.array_equal(got[0][name], got[1][name]), name


@pytest.mark.parametrize("wide", [False, True])
def test_first_cut_call_beside_a_capture(wide):
    """A context's first cut call, which allocates and may build matrices,
    while another CUDA stream is captured in the default mode, by this thread
    or another: the call's words and the captured graph are both good."""
    from concurrent.futures import ThreadPoolExecutor
    from paper_1108_0486_gb300 import Streams, Streams64
    n, dtype = 1 << 20, torch.int64 if wide else torch.int32
    cs, own = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(1000, device="cuda")
    for other_thread in (False, True):
        with (Streams64 if wide else Streams)(2, seeds=W.seeds(2), stream=own) as st, ThreadPoolExecutor(1) as pool:
            draw = st.u64 if wide else st.u32
            out = torch.empty((2, n), dtype=dtype, device="cuda")
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=cs, capture_error_mode="global"):
                x += 1
                pool.submit(draw, n, out=out).result() if other_thread else draw(n, out=out)
                x += 1
            g.replay()
            torch.cuda.synchronize()
            ref = O.streams64(W.seeds(2), n) if wide else O.streams(W.seeds(2), n)
            assert np.array_equal(out.cpu().numpy().view(ref.dtype), ref)
    assert float(x.sum()) == 4000.0


def sum_in_pieces(z, q):
    """One row's normals added in the documented order of a call cut into
    pieces of 2^q: per piece, each lane's values in sequence and a butterfly in
    FP32; lane l of 32 adds the pieces l, l + 32, ... in FP64, a butterfly."""
    def butterfly(v):
        for off in (16, 8, 4, 2, 1):
            v = v + v[..., np.arange(32) ^ off]
        return v[..., 0]
    pieces = -(-(z.size + (z.size & 1)) >> q)
    v = np.zeros((pieces << q,), dtype=np.float32)
    v[:z.size] = z
    v = v.reshape(pieces, -1, 32, 2).transpose(0, 2, 1, 3).reshape(pieces, 32, -1)
    sums = butterfly(np.add.accumulate(v, axis=2, dtype=np.float32)[..., -1]).astype(np.float64)
    lanes = np.zeros((-(-pieces // 32) * 32,))
    lanes[:pieces] = sums
    return np.float32(butterfly(np.add.accumulate(lanes.reshape(-1, 32), axis=0)[-1]))


@pytest.mark.parametrize("streams,n,piece", [(1, 32769, 0), (1, (1 << 18) + 3, 4096), (3, 262145, 64), (2, 1 << 20, 0),
                                              (7, 300001, 0), (64, 1 << 18, 65536), (100, 70001, 0), (500, 200001, 0)])
def test_sums_of_cut_calls_bit_for_bit(streams, n, piece):
    """Sums of calls cut into pieces of a set or a chosen length (none is left
    out or taken twice: the exact bits), called, then captured and replayed
    twice; the streams end where whole calls end."""
    import ctypes
    from paper_1108_0486_gb300 import Streams, _lib as L
    choose = L.lib()._ZN2xg10cut_chooseEijmim   # xg::cut_choose, kind 3: fused sums
    choose.argtypes = [ctypes.c_int, ctypes.c_uint32, ctypes.c_uint64, ctypes.c_int, ctypes.c_uint64]
    q = choose(3, streams, n, torch.cuda.get_device_properties(0).multi_processor_count, piece)
    assert q >= 6 and (not piece or 1 << q == piece)
    ps, cs = streams % 2, torch.cuda.Stream()
    with Streams(streams, param_set=ps, seeds=W.seeds(streams), stream=cs) as a, \
            Streams(streams, param_set=ps, seeds=W.seeds(streams), stream=cs) as b, torch.cuda.stream(cs):
        a.set_batch_split(piece)
        b.set_batch_split(1)
        got = [a.normal_sum(n)]
        out = torch.empty(streams, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=cs):
            a.normal_sum(n, out=out)
        for _ in range(2):
            g.replay()
            got.append(out.clone())
        for sums in got:
            z = b.normal(n).cpu().numpy()
            for s in {0, streams // 2, streams - 1}:
                assert float(sums[s]) == float(sum_in_pieces(z[s], q)), s
        assert torch.equal(a.u32(77), b.u32(77))
        assert np.array_equal(a.checkpoint()["pos"], b.checkpoint()["pos"])


def test_tensor_core_jump_at_the_edges_of_its_tiles():
    """One power applied to as many states as fill the last tile, leave one
    place free in it or start another, for tiles of every width between 16 and
    240 that the library takes: the table kernel's states."""
    import ctypes
    import os
    from paper_1108_0486_gb300 import Streams, _lib as L
    fn, waves = L.lib()._ZN2xg11gf2_tc_tileEPKjiiPj, ctypes.c_uint32()   # xg::gf2_tc_tile
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tile = lambda n: fn(ctypes.byref(ctypes.c_uint32(n)), 1, sms, ctypes.byref(waves))
    sizes = {}
    for n in range(8, 20000):
        w = tile(n)
        if n % w in (0, 1, w - 1):
            sizes.setdefault((w, n % w), n)
    assert {w for w, _ in sizes} >= {16, 240} and len(sizes) >= 20
    for n in sorted(set(sizes.values())):
        rows = []
        for tc in ("1", "0"):
            os.environ["XG_JUMP_TENSOR_CORES"] = tc
            try:
                with Streams(n, seeds=W.seeds(n)) as st:
                    st.jump(1 << 37)
                    rows.append(st.u32(128))
            finally:
                del os.environ["XG_JUMP_TENSOR_CORES"]
        assert torch.equal(*rows), n


@pytest.mark.parametrize("family", [0, 1, 64])
@pytest.mark.parametrize("words", [(1 << 33) + 12, (1 << 30) + (1 << 20) + 9, (1 << 41) + 0x3F])
def test_table_kernel_jumps_at_the_limits_of_products(family, words, monkeypatch):
    """Without the tensor cores: streams on both sides of the counts from which
    3, 4 or 7 powers are multiplied first (65, 5, 1) and of the table kernel's
    forms (4, 192 states), against jumps by one power after another."""
    from paper_1108_0486_gb300 import Streams, Streams64
    monkeypatch.setenv("XG_JUMP_TENSOR_CORES", "0")
    rows = []
    for n in (1, 4, 5, 64, 65, 191, 192):
        for jumps in ([words], [1 << k for k in range(64) if words >> k & 1]):
            seeds = W.seeds(n)
            with (Streams64(n, seeds=seeds) if family == 64 else Streams(n, param_set=family, seeds=seeds)) as st:
                for j in jumps:
                    st.jump(j)
                rows.append((st.u64 if family == 64 else st.u32)(140))
        assert torch.equal(rows[-1], rows[-2]), n
        assert torch.equal(rows[-1][0], rows[0][0])

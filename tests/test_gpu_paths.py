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


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("tpg,wpl", [(4, 8), (8, 4), (16, 2), (16, 4), (32, 2)])
@pytest.mark.parametrize("ps", [0, 1])
def test_rows_at_every_word_offset(kind, tpg, wpl, ps):
    """Two calls in a row whose rows start 0 .. 3 words off a 16-byte boundary:
    lengths below and above one turn of the ring and the limit from which the
    ring is moved on; the words around each row stay untouched, and the second
    call continues the first."""
    from paper_1108_0486_gb300 import Streams
    streams = 5
    seeds = W.seeds(streams)
    for n in (3, 128, 131, 132, 133, 2047, 2049, 2211):
        ld = n + 4 + (1 - n) % 4          # rows 1 word further off each time
        m = words_of(kind, n)
        ref = O.streams(seeds, 2 * m, param_set=ps)
        for off in (1, 2):
            with Streams(streams, param_set=ps, seeds=seeds) as st:
                st.set_launch(kind, tpg, wpl)
                dt = torch.int32 if kind == "u32" else torch.float32
                for call in range(2):
                    buf = torch.full((streams * ld + 8,), -7, dtype=dt, device="cuda")
                    st.generate(kind, n, out=buf[off:], ld=ld)
                    h = buf.cpu().numpy()
                    assert np.all(h[:off] == -7)
                    for i in range(streams):
                        row = h[off + i * ld:off + i * ld + ld]
                        check(kind, row[:n], ref[i, call * m:(call + 1) * m], n)
                        assert np.all(row[n:n + 1] == -7)


def test_batch_rows_at_every_word_offset():
    """Cut and uncut calls of a batch with outputs 0 .. 3 words off."""
    from paper_1108_0486_gb300 import Streams
    seeds = W.seeds(24)
    with Streams(24, seeds=seeds) as st:
        st.set_batch_split(2048)
        items, outs = [], []
        for i in range(24):
            kind, off, n = KINDS[i % 3], i // 3 % 4, (130, 5000, 777, 4099)[i % 4]
            buf = torch.full((n + 8,), -7, dtype=torch.int32 if kind == "u32" else torch.float32, device="cuda")
            outs.append((kind, off, n, buf))
            items.append((i, kind, n, buf[off:off + n]))
        st.batch(items)
        st.batch(items)
        torch.cuda.synchronize()
    for i, (kind, off, n, buf) in enumerate(outs):
        m = words_of(kind, n)
        h = buf.cpu().numpy()
        check(kind, h[off:off + n], O.streams(seeds[i:i + 1], 2 * m)[0, m:], n)
        assert np.all(h[:off] == -7) and np.all(h[off + n:] == -7)


@pytest.mark.parametrize("tpg,wpl", [(0, 0), (4, 8), (8, 4), (16, 2), (32, 1)])
def test_fp64_uniforms_of_words_with_many_leading_zeros(tpg, wpl):
    """A nearly empty ring without the Weyl word gives zeros and words of every
    small size, which leave the conversion of the common words: values against
    the closed form of the words themselves, at lengths around one and two
    iterations of the kernel's loop and ends of rows."""
    from paper_1108_0486_gb300 import Streams64
    for n in (1, 33, 511, 512, 513, 577, 1025, 4000):
        got = []
        for kind in ("u64", "uniform"):
            with Streams64(3, weyl=False, seeds=W.seeds(3)) as st:
                for s in range(3):
                    ring = np.zeros(64, dtype=np.uint64)
                    ring[(7 * s + 1) % 64] = 1 << (20 * s)
                    st.set_state(s, ring, 0)
                if tpg:
                    st.set_launch(kind, tpg, wpl)
                got.append(np.concatenate([st.generate(kind, n).cpu().numpy(), st.generate(kind, n).cpu().numpy()], 1))
        words = got[0].view(np.uint64)
        assert np.array_equal(got[1], O.uniform64_of(words).reshape(words.shape))
        if n > 1000:
            small = words < (1 << 43)
            assert small.any() and not small.all()


@pytest.mark.parametrize("family", [0, 1, 64])
@pytest.mark.parametrize("words", [3, (1 << 40) + (1 << 20) + 12345, 0x9E3779B97F4A7C15])
def test_jump_on_both_sides_of_its_thresholds(family, words):
    """The same jump of 64 states (one power after another), 65 (product of the
    powers, table kernel) and 192 or 1024 (product, tensor cores): equal streams end
    in equal states, and those of the single-stream jump; short jumps equal
    stepping by the oracle."""
    from paper_1108_0486_gb300 import Streams, Streams64

    def make(n):
        seeds = W.seeds(n)
        return Streams64(n, seeds=seeds) if family == 64 else Streams(n, param_set=family, seeds=seeds)

    def draw(st):
        return (st.u64(70) if family == 64 else st.u32(140)).cpu().numpy()

    rows = {}
    for n in (1, 64, 65, 192, 1024):
        with make(n) as st:
            st.jump(words)
            rows[n] = draw(st)
    assert np.array_equal(rows[64], rows[65][:64]) and np.array_equal(rows[65], rows[1024][:65])
    assert np.array_equal(rows[192], rows[1024][:192])
    assert np.array_equal(rows[1][0], rows[64][0])
    if words == 3:
        seeds = W.seeds(4)
        ref = O.streams64(seeds, 73) if family == 64 else O.streams(seeds, 143, param_set=family)
        assert np.array_equal(rows[65][:4].view(ref.dtype), ref[:, 3:])


@pytest.mark.parametrize("n", [191, 192, 239, 240, 241, 480, 1141])
def test_tensor_core_jump_at_tile_edges(n, monkeypatch):
    """One power applied to n states on the tensor cores (tiles of 240 states,
    used from 192) equals the table kernel's result."""
    from paper_1108_0486_gb300 import Streams
    rows = []
    for tc in ("1", "0"):
        monkeypatch.setenv("XG_JUMP_TENSOR_CORES", tc)
        with Streams(n, seeds=W.seeds(n)) as st:
            st.jump(1 << 37)
            rows.append(st.u32(128).cpu().numpy())
    assert np.array_equal(rows[0], rows[1])


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("streams,n,piece", [(1, 16385, 0), (1, (1 << 18) + 3, 0), (1, 1 << 18, 4096), (3, 262145, 64),
                                              (7, 300001, 0), (64, 1 << 18, 65536), (100, 70001, 0), (600, 140002, 0)])
def test_cut_calls_equal_whole_calls(kind, streams, n, piece):
    """Calls cut into pieces (chosen by the library, or of a set length; one
    and several prologue steps, on the tensor cores and not; the last piece
    full, short and odd) against whole calls on the same streams, twice in a
    row, at aligned and unaligned rows; two streams against the oracle."""
    from paper_1108_0486_gb300 import Streams
    ps = streams % 2
    rows = []
    for split in (piece, 1):
        with Streams(streams, param_set=ps, seeds=W.seeds(streams)) as st:
            st.set_batch_split(split)
            a = st.generate(kind, n)
            b = st.generate(kind, n, ld=n + 5)[:, :n]
            c = st.generate(kind, 77)
            rows.append([a, b, c])
            pos = st.checkpoint()["pos"]
            assert np.all(pos == 2 * words_of(kind, n) + words_of(kind, 77))
    for x, y in zip(*rows):
        assert torch.equal(x, y)
    if streams <= 7:
        m = words_of(kind, n)
        for s in {0, streams - 1}:
            w = O.streams(W.seeds(1, 1 + s), 2 * m, param_set=ps)[0]
            check(kind, rows[0][1][s].cpu().numpy(), w[m:], n)


def test_cut_calls_on_two_cuda_streams():
    """Cut calls of one context on alternating CUDA streams, each ordered after
    the other: the workspace they share follows."""
    from paper_1108_0486_gb300 import Streams, _lib as L
    n = 1 << 18
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with Streams(5, seeds=W.seeds(5)) as st:
        outs = []
        for k in range(6):
            cs, other = (s1, s2) if k % 2 else (s2, s1)
            # calls on disjoint streams need no order between the CUDA streams
            L.xg_set_stream(st.ctx, cs.cuda_stream)
            with torch.cuda.stream(cs):
                outs.append(st.u32(n, first=k % 2, count=1))
        torch.cuda.synchronize()
        L.xg_set_stream(st.ctx, torch.cuda.current_stream().cuda_stream)
        got = [o.cpu().numpy().view(np.uint32)[0] for o in outs]
    for s in (0, 1):
        w = O.streams(W.seeds(1, 1 + s), 3 * n)[0]
        assert np.array_equal(np.concatenate(got[s::2]), w)


def test_call_in_a_captured_graph_is_not_cut():
    """A call that would be cut runs whole while its CUDA stream is captured;
    replays continue the streams."""
    from paper_1108_0486_gb300 import Streams
    n, streams = 50000, 200
    cs = torch.cuda.Stream()
    with Streams(streams, seeds=W.seeds(streams), stream=cs) as st:
        out = torch.empty((streams, n), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=cs):
            st.u32(n, out=out)
        for k in range(2):
            g.replay()
            torch.cuda.synchronize()
            w = O.streams(W.seeds(1, streams), (k + 1) * n)[0, k * n:]
            assert np.array_equal(out[streams - 1].cpu().numpy().view(np.uint32), w)


@pytest.mark.parametrize("n", [3071, 3072, 3327, 3329, 8191, 8192, 8193, 8447, 8448, 8449, 8703, 8705])
@pytest.mark.parametrize("ps", [0, 1])
def test_long_normals_and_sums_with_tail_pairs(n, ps):
    """Lengths around the limits of the voted loop and around its iterations,
    rows that vector stores fit and others; nearly empty rings without the Weyl
    word, whose small words put many pairs into the FP64 tail, beside seeded
    streams: the bits of another launch shape, and sums within the rounding of
    each lane's additions."""
    from paper_1108_0486_gb300 import Streams
    streams = 40

    def make():
        st = Streams(streams, param_set=ps, weyl=False, seeds=W.seeds(streams))
        for s in range(3):
            ring = np.zeros(128, dtype=np.uint32)
            ring[(41 * s + 1) % 128] = 1 << (9 * s)
            st.set_state(s, ring, 0)
        return st

    with make() as a, make() as b, make() as c:
        b.set_launch("normal", 16, 2)
        for ld in (n, n + (-n) % 4):
            x, y = a.normal(n, ld=ld)[:, :n], b.normal(n, ld=ld)[:, :n]
            assert torch.equal(x, y)
            assert torch.equal(torch.from_numpy(a.checkpoint()["rings"]), torch.from_numpy(b.checkpoint()["rings"]))
            got = c.normal_sum(n).double()
            z = x.double()
            bound = (n / 32 + 6) * 2.0 ** -24 * z.abs().sum(1)
            assert bool(((got - z.sum(1)).abs() <= bound).all())


@pytest.mark.parametrize("kind", KINDS)
def test_short_calls_on_many_streams(kind):
    """Lengths on both sides of the limits under which many streams take
    another shape, and of the storing of rows that no vector store fits on both
    sides of its stream count: two calls each, first and last streams."""
    from paper_1108_0486_gb300 import Streams
    parts = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    for streams, lengths in ((18 * parts, (3, 129, 511, 512, 1535, 1536, 2047, 2048)), (5 * parts - 1, (2047, 2049)),
                             (5 * parts, (2047, 2049)), (1, (2049,))):
        for n in lengths:
            with Streams(streams, seeds=W.seeds(streams)) as st:
                rows = torch.cat([st.generate(kind, n), st.generate(kind, n)], 1)
                for s in (0, streams - 1):
                    got = rows[s].cpu().numpy()
                    w = O.streams(W.seeds(1, 1 + s), 2 * words_of(kind, n))[0]
                    check(kind, got[:n], w, n)
                    check(kind, got[n:], w[words_of(kind, n):], n)


@pytest.mark.parametrize("streams", [2047, 2048])
def test_short_fp64_uniforms_on_many_streams(streams):
    from paper_1108_0486_gb300 import Streams64
    for n in (1, 65, 255, 257, 1023, 1024):
        with Streams64(streams, seeds=W.seeds(streams)) as st:
            rows = torch.cat([st.uniform(n), st.uniform(n)], 1)
            for s in (0, streams - 1):
                ref = O.uniform64_of(O.streams64(W.seeds(1, 1 + s), 2 * n))
                assert np.array_equal(rows[s].cpu().numpy(), np.asarray(ref).reshape(-1))


@pytest.mark.parametrize("streams,n,piece", [(1, 16385, 0), (1, (1 << 18) + 3, 4096), (3, 262145, 64), (7, 300001, 0),
                                              (64, 1 << 18, 65536), (100, 70001, 0), (600, 140002, 0)])
def test_cut_sums(streams, n, piece):
    """Sums of calls cut into pieces (chosen by the library, or of a set
    length): within the rounding of each lane's additions of the FP64 sum of
    the same normals, twice in a row; the streams end where whole calls end,
    and a set launch shape keeps its order of additions."""
    from paper_1108_0486_gb300 import Streams
    ps = streams % 2
    make = lambda: Streams(streams, param_set=ps, seeds=W.seeds(streams))
    with make() as a, make() as b, make() as c, make() as d:
        a.set_batch_split(piece)
        b.set_batch_split(1)
        c.set_launch("normal", 32, 2)
        d.set_batch_split(1)
        d.set_launch("normal", 32, 2)
        for _ in range(2):
            z = b.normal(n).double()
            bound = (n / 32 + 6) * 2.0 ** -24 * z.abs().sum(1)
            assert bool(((a.normal_sum(n).double() - z.sum(1)).abs() <= bound).all())
            assert torch.equal(c.normal_sum(n), d.normal_sum(n))
        assert torch.equal(a.u32(77), b.u32(77))
        assert np.array_equal(a.checkpoint()["pos"], b.checkpoint()["pos"])


@pytest.mark.parametrize("streams,piece,pieces", [(33, 65536, 5), (40, 32768, 9), (60, 8192, 33), (64, 4096, 65),
                                                  (17, 16384, 17), (49, 131072, 2), (49, 131072, 3), (64, 32768, 8)])
@pytest.mark.parametrize("tensor_cores", ["1", "0"])
def test_cut_prologue_steps(streams, piece, pieces, tensor_cores, monkeypatch):
    """Piece counts that make the steps of the prologue take one to seven
    matrices, the last one only in part, on the tensor cores and by the table
    kernel: outputs and streams of whole calls."""
    from paper_1108_0486_gb300 import Streams
    monkeypatch.setenv("XG_JUMP_TENSOR_CORES", tensor_cores)
    n = max(1 << 18, piece * (pieces - 1) + 321)
    rows = []
    for split in (piece, 1):
        with Streams(streams, param_set=streams % 2, seeds=W.seeds(streams)) as st:
            st.set_batch_split(split)
            rows.append((st.u32(n), st.u32(n), st.u32(99)))
    for x, y in zip(*rows):
        assert torch.equal(x, y)


@pytest.mark.parametrize("kind", ["u64", "uniform"])
@pytest.mark.parametrize("streams,n,piece", [(1, 32769, 0), (1, (1 << 18) + 3, 4096), (3, 262145, 64), (16, 1 << 18, 32768),
                                              (17, 70001, 0), (100, 131072, 0), (400, 262147, 0)])
def test_cut_64bit_calls_equal_whole_calls(kind, streams, n, piece):
    """64-bit calls cut into pieces (chosen by the library, or of a set length)
    against whole calls on the same streams, twice in a row, with rows of odd
    strides; a stream against the oracle."""
    from paper_1108_0486_gb300 import Streams64
    rows = []
    for split in (piece, 1):
        with Streams64(streams, seeds=W.seeds(streams)) as st:
            st.set_split(split)
            rows.append([st.generate(kind, n), st.generate(kind, n, ld=n + 5)[:, :n], st.generate(kind, 77)])
            rows[-1].append(torch.from_numpy(np.concatenate([st.get_state(streams - 1)[0]]).view(np.int64)))
    for x, y in zip(*rows):
        assert torch.equal(x, y)
    w = O.streams64(W.seeds(1, streams), 2 * n)[0, n:]
    got = rows[0][1][streams - 1].cpu().numpy()
    assert np.array_equal(got.view(np.uint64), w) if kind == "u64" else np.array_equal(got, O.uniform64_of(w))


def test_64bit_call_in_a_captured_graph_is_not_cut():
    from paper_1108_0486_gb300 import Streams64
    n, streams = 1 << 18, 3
    cs = torch.cuda.Stream()
    with Streams64(streams, seeds=W.seeds(streams), stream=cs) as st:
        out = torch.empty((streams, n), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=cs):
            st.u64(n, out=out)
        for k in range(2):
            g.replay()
            torch.cuda.synchronize()
            w = O.streams64(W.seeds(1, streams), (k + 1) * n)[0, k * n:]
            assert np.array_equal(out[streams - 1].cpu().numpy().view(np.uint64), w)


@pytest.mark.parametrize("family", [0, 1, 64])
@pytest.mark.parametrize("words", [1 << 21, (1 << 33) + (1 << 9) + 5, 0x9E3779B97F4A7C15])
def test_jump_in_the_windows(family, words, monkeypatch):
    """Jumps of 192 and more consecutive streams in the middle of a context, in
    place on the tensor cores, after draws that leave pending words: the
    states, positions and next words of the table kernel's jump, and the other
    streams untouched."""
    from paper_1108_0486_gb300 import Streams, Streams64
    n = 500
    for first, count in ((0, 500), (7, 192), (3, 241)):
        got = []
        for tc in ("1", "0"):
            monkeypatch.setenv("XG_JUMP_TENSOR_CORES", tc)
            seeds = W.seeds(n)
            with (Streams64(n, seeds=seeds) if family == 64 else Streams(n, param_set=family, seeds=seeds)) as st:
                draw = st.u64 if family == 64 else st.u32
                draw(77)
                st.jump(words, first=first, count=count)
                rows = [draw(45), draw(200)]
                if family != 64:
                    c = st.checkpoint()
                    rows += [torch.from_numpy(c[k].view(np.int64 if k == "pos" else np.int32)) for k in ("rings", "weyl", "pos")]
                got.append([r.cpu() for r in rows])
        for x, y in zip(*got):
            assert torch.equal(x, y)


@pytest.mark.parametrize("family", [0, 1, 64])
@pytest.mark.parametrize("bits", [2, 5, 6, 7, 9, 10, 11, 33])
def test_jump_by_the_number_of_set_bits(family, bits):
    """Jumps whose powers form one or two chains, few streams on both sides of
    the number of bits from which their powers are multiplied first, and many:
    the same power after power."""
    from paper_1108_0486_gb300 import Streams, Streams64
    rng = np.random.default_rng(bits)
    at = sorted(rng.choice(45, bits, replace=False).tolist())
    words = sum(1 << k for k in at)

    def make(n):
        seeds = W.seeds(n)
        return Streams64(n, seeds=seeds) if family == 64 else Streams(n, param_set=family, seeds=seeds)

    def draw(st):
        return (st.u64(70) if family == 64 else st.u32(140)).cpu()

    with make(3) as st:
        for k in at:
            st.jump(1 << k)
        ref = draw(st)
    for n in (3, 70, 200):
        with make(n) as st:
            st.jump(words)
            assert torch.equal(draw(st)[:3], ref)


@pytest.mark.parametrize("tensor_cores", ["1", "0"])
@pytest.mark.parametrize("calls", [(2,), (8, 9), (3, 64, 65, 1), (7, 512, 513, 20, 2, 100), tuple(range(1, 90)), (600,) * 40])
def test_batch_prologue_steps(calls, tensor_cores, monkeypatch):
    """Batches whose calls are cut into the given numbers of pieces (one to
    three prologue steps, sources with one to seven results each) against
    uncut batches, twice in a row."""
    from paper_1108_0486_gb300 import Streams
    monkeypatch.setenv("XG_JUMP_TENSOR_CORES", tensor_cores)
    rows = []
    for split in (64, 1):
        with Streams(len(calls), param_set=len(calls) % 2, seeds=W.seeds(len(calls))) as st:
            st.set_batch_split(split)
            got = []
            for call in range(2):
                outs = [torch.zeros(64 * k - (5 if k % 3 else 0), dtype=torch.int32, device="cuda") for k in calls]
                st.batch([(i, "u32", o.numel(), o) for i, o in enumerate(outs)])
                got.append(torch.cat(outs))
            got.append(st.u32(99).reshape(-1))
            rows.append(torch.cat(got))
    assert torch.equal(*rows)


@pytest.mark.parametrize("family", [0, 64])
@pytest.mark.parametrize("words", [1 << 21, (1 << 33) + (1 << 9) + 5, (1 << 30) + 12345])
def test_jump_of_a_few_streams_in_the_windows(family, words, monkeypatch):
    """The same on both sides of the least stream count that is jumped in place."""
    from paper_1108_0486_gb300 import Streams, Streams64
    for n, first, count in ((8, 0, 8), (20, 3, 7), (20, 3, 8), (20, 2, 17), (150, 50, 64), (150, 50, 65)):
        got = []
        for tc in ("1", "0"):
            monkeypatch.setenv("XG_JUMP_TENSOR_CORES", tc)
            seeds = W.seeds(n)
            with (Streams64(n, seeds=seeds) if family == 64 else Streams(n, seeds=seeds)) as st:
                draw = st.u64 if family == 64 else st.u32
                draw(77)
                st.jump(words, first=first, count=count)
                got.append(torch.cat([draw(45), draw(200)], 1))
        assert torch.equal(*got)

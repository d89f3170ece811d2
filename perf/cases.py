"""The work that users of the library have it do, as cases to be timed and compared.

A case is one pass through the public entry points of ``Streams``,
``Streams64`` and ``Server`` with the launch configuration the library picks
by itself.  Sizes are those of ``workloads.py``, ``bench.py`` and the tests,
and generic odd ones between them.

``exact`` computes the same outputs with plain torch integer and FP64
operations from the definitions of arXiv:1108.0486 (Sec. 1.5, Sec. 2) and the
library's stated seeding and conversions.
"""
import math

import numpy as np
import torch

from paper_1108_0486_gb300 import Streams, Streams64
from paper_1108_0486_gb300 import workloads as W

KINDS = ("u32", "uniform", "normal")
DTYPES = {"u32": torch.int32, "uniform": torch.float32, "normal": torch.float32}
JUMP = (1 << 40) + (1 << 20) + 12345


def listed():
    return [
        # a simulation that asks for a little at a time: launch and host time
        {"name": "small_uniform", "do": "generate", "kind": "uniform", "params": 0, "streams": 64, "n": 1000},
        # one generator, one long run of words (the serial chain of the method)
        {"name": "single_stream_u32", "do": "generate", "kind": "u32", "params": 0, "streams": 1, "n": 1 << 20},
        # many streams, raw words, at a length no power of two divides: rows are not 16-byte aligned
        {"name": "many_u32_odd", "do": "generate", "kind": "u32", "params": 0, "streams": 10000, "n": 100003},
        # the many-streams workload of the benchmark, uniforms
        {"name": "many_uniform", "do": "generate", "kind": "uniform", "params": 0, "streams": 16384, "n": 1 << 16},
        # the normals workload of the benchmark: 2^30 normals
        {"name": "many_normal", "do": "generate", "kind": "normal", "params": 0, "streams": 16384, "n": 1 << 16},
        # a few hundred long streams (one per worker of a simulation), the paper's parameter set
        {"name": "mid_normal_paper", "do": "generate", "kind": "normal", "params": 1, "streams": 500, "n": 500000},
        # Monte Carlo estimate: only each stream's sum of normals is wanted
        {"name": "normal_sum", "do": "sum", "kind": "normal", "params": 0, "streams": 10000, "n": 65537},
        # one batch of calls of very different lengths and mixed types
        {"name": "batch_uneven", "do": "batch", "params": 0, "streams": 4096, "lo": 1 << 10, "hi": 1 << 22, "mix": 1108},
        # requests of uneven size that arrive together at the server
        {"name": "serve_burst", "do": "serve", "params": 0, "streams": 65536, "requests": 256, "lo": 1 << 10, "hi": 1 << 22,
         "mix": 486},
        # every stream skips ahead to its own far block, then draws a little
        {"name": "jump_many", "do": "jump", "params": 0, "streams": 16384, "words": JUMP, "n": 128},
        # FP64 uniforms of the 64-bit generator at the benchmark's size
        {"name": "w64_uniform", "do": "generate64", "kind": "uniform", "streams": 16384, "n": 1 << 15},
        # raw 64-bit words on a middling number of streams, odd length
        {"name": "w64_mid_u64", "do": "generate64", "kind": "u64", "streams": 1000, "n": 100001},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(("generate", "generate", "generate", "sum", "batch", "serve", "jump", "generate64"))
    params = rng.randint(0, 1)
    if do in ("generate", "sum", "generate64"):
        streams = _log(rng, 1, 40000)
        # at most 2^30 words in all, and no stream so long that one call is a matter of seconds
        n = _log(rng, 100, max(200, min(1 << 21, (1 << (29 if do == "generate64" else 30)) // streams)))
        if rng.random() < 0.5:
            n = max(64, n // 64 * 64)
        if do == "generate64":
            return {"do": do, "kind": rng.choice(("u64", "uniform")), "streams": streams, "n": n}
        return {"do": do, "kind": "normal" if do == "sum" else rng.choice(KINDS), "params": params, "streams": streams, "n": n}
    if do == "batch":
        lo = _log(rng, 64, 4096)
        return {"do": do, "params": params, "streams": _log(rng, 16, 4096), "lo": lo, "hi": _log(rng, 16 * lo, 1 << 22),
                "mix": rng.randint(1, 1 << 30)}
    if do == "serve":
        lo = _log(rng, 64, 4096)
        return {"do": do, "params": params, "streams": _log(rng, 64, 65536), "requests": _log(rng, 1, 512), "lo": lo,
                "hi": _log(rng, 16 * lo, 1 << 22), "mix": rng.randint(1, 1 << 30)}
    return {"do": do, "params": params, "streams": _log(rng, 1, 20000), "words": _log(rng, 1 << 10, 1 << 62), "n": 128}


def _seeds(streams, seed):
    # block ids, as the paper seeds (Sec. 4), from a start that the seed gives
    return W.seeds(streams, 1 + (int(seed) * 1000003) % 0x70000000)


def _words(kind, n):
    return n + (n & 1) if kind == "normal" else n


def _calls(case):
    """(stream, kind, count) of a batch's or a burst's calls, as workloads.py draws them."""
    if case["do"] == "batch":
        items = W.batched_uneven(case["streams"], case["lo"], case["hi"], seed=case["mix"])
        return [(it.stream, KINDS[it.kind], it.count) for it in items]
    rng = np.random.Generator(np.random.PCG64(case["mix"]))
    m = case["requests"]
    sizes = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), m)).astype(np.int64)
    kinds = rng.choice(3, size=m, p=(0.1, 0.3, 0.6))
    streams = rng.integers(0, case["streams"], m)
    return [(int(s), KINDS[int(k)], int(c)) for s, k, c in zip(streams, kinds, sizes)]


def _places(calls):
    """Each call's place in one buffer of its type (starts are multiples of 4), and the buffers' sizes."""
    size, at = dict.fromkeys(KINDS, 0), []
    for _, kind, count in calls:
        at.append(size[kind])
        size[kind] += (count + 3) // 4 * 4
    return at, size


def prepare(case, seed):
    do = case["do"]
    seeds = _seeds(case["streams"], seed)
    if do == "generate64":
        return {"case": case, "streams": Streams64(case["streams"], seeds=seeds)}
    st = Streams(case["streams"], param_set=case["params"], seeds=seeds)
    state = {"case": case, "streams": st}
    if do in ("batch", "serve"):
        calls = _calls(case)
        at, size = _places(calls)
        bufs = {k: torch.zeros(max(4, size[k]), dtype=DTYPES[k], device="cuda") for k in KINDS}
        state["bufs"] = bufs
        state["calls"] = [(s, k, c, bufs[k][a:a + c]) for (s, k, c), a in zip(calls, at)]
        torch.cuda.synchronize()
        if do == "serve":
            state["server"] = st.serve()
    return state


def run(state):
    case, st = state["case"], state["streams"]
    do = case["do"]
    if do in ("generate", "generate64"):
        return st.generate(case["kind"], case["n"])
    if do == "sum":
        return st.normal_sum(case["n"])
    if do == "jump":
        st.jump(case["words"])
        return st.u32(case["n"])
    if do == "batch":
        st.batch(state["calls"])
        return state["bufs"]
    srv = state["server"]
    tickets = srv.submit_many(state["calls"])
    for t in tickets:
        srv.wait(t)
        srv.release(t)
    return state["bufs"]


def work(case):
    do = case["do"]
    if do in ("batch", "serve"):
        # the mean of the log-uniform lengths; arithmetic as for the mean of the types
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        words = mean * (case["streams"] if do == "batch" else case["requests"])
        return {"bytes": 4.0 * words, "flops": 25.0 * words}
    size = 8.0 if do == "generate64" else 4.0
    state = 2.0 * 528.0 * case["streams"]                 # ring, Weyl word and position, read and written
    words = float(case["streams"]) * case["n"]
    out = case["streams"] * 4.0 if do == "sum" else size * words
    ops = {"u32": 12, "u64": 24, "uniform": 15, "normal": 36}[case.get("kind", "u32")]
    return {"bytes": out + state, "flops": ops * words}


# ---- the same outputs in plain torch, FP64 ------------------------------------

SETS = {0: (128, 95, 17, 12, 13, 15, 32, 0x9E3779B9), 1: (128, 65, 15, 14, 12, 17, 32, 0x9E3779B9),
        64: (64, 55, 42, 27, 25, 22, 64, 0x9E3779B97F4A7C15)}
MOST_WORDS, MOST_ROUNDS = 1 << 30, 70000


def _signed(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _shr(x, k):
    """Logical right shift of 64-bit patterns."""
    return (x >> k) & ((1 << (64 - k)) - 1)


class _Generator:
    """The serial definition, a block of consecutive words (fewer than the lag s) at a time, all streams at once."""

    def __init__(self, seeds, which):
        self.r, self.s, self.a, self.b, self.c, self.d, self.w, self.omega = SETS[which]
        self.full = -1 if self.w == 64 else 0xFFFFFFFF
        self.step = 32 if self.w == 64 else 64
        seed = torch.from_numpy(seeds.astype(np.int64)).cuda()
        v = (seed << 32) | (~seed & 0xFFFFFFFF)
        ring = []
        for j in range(64 + self.r + 1):
            v = v ^ (v << 13)
            v = v ^ _shr(v, 7)
            v = v ^ (v << 17)
            if j >= 64:
                ring.append(v if self.w == 64 else _shr(v, 32))
        self.weyl = ring.pop()
        self.ring = torch.stack(ring, 1)
        self.more(4 * self.r)

    def _half(self, x, left, right):
        x = x ^ ((x << left) & self.full)
        return x ^ (_shr(x, right) if self.w == 64 else x >> right)

    def more(self, n):
        """The next n outputs (Eq. 1) of every stream, as int64."""
        r, step = self.r, self.step
        rounds = -(-n // step)
        x = torch.empty(self.ring.shape[0], r + rounds * step, dtype=torch.int64, device="cuda")
        x[:, :r] = self.ring
        for k in range(r, r + rounds * step, step):
            x[:, k:k + step] = self._half(x[:, k - r:k - r + step], self.a, self.b) ^ \
                self._half(x[:, k - self.s:k - self.s + step], self.c, self.d)
        self.ring = x[:, n:n + r].clone()
        omega = _signed(self.omega)
        out = x[:, r:r + n]
        part = max(1, (1 << 27) // max(1, n))
        for i in range(0, out.shape[0], part):
            w = self.weyl[i:i + part, None] + torch.arange(1, n + 1, dtype=torch.int64, device="cuda") * omega
            w &= self.full
            w ^= _shr(w, self.w // 2)
            out[i:i + part] = (out[i:i + part] + w) & self.full
        self.weyl = (self.weyl + _signed(n * self.omega % (1 << 64))) & self.full
        return out

    def keep(self, rows):
        self.ring, self.weyl = self.ring[:rows], self.weyl[:rows]


def _value(kind, words):
    """FP64 values of the last dimension's words (an even number of them for normals)."""
    if kind == "uniform":
        return (words >> 8).double() * 2.0 ** -24
    if kind == "uniform64":
        return _shr(words, 11).double() * 2.0 ** -53
    if kind != "normal":
        return words
    out = torch.empty(words.shape, dtype=torch.float64, device="cuda")
    radius = torch.sqrt(-2.0 * torch.log(((words[..., 0::2] >> 8) + 1).double() * 2.0 ** -24))
    # the angle is reduced exactly: 2 pi u = q pi/2 + a with |a| <= pi/4
    m = words[..., 1::2] >> 8
    q = (m + (1 << 21)) >> 22
    a = (m - (q << 22)).double() * (2.0 * math.pi * 2.0 ** -24)
    sin, cos, q = torch.sin(a), torch.cos(a), q & 3
    odd = (q & 1).bool()
    flip = lambda bit: 1.0 - 2.0 * ((bit >> 1) & 1).double()  # noqa: E731
    out[..., 0::2] = radius * torch.where(odd, sin, cos) * flip(q + 1)
    out[..., 1::2] = radius * torch.where(odd, cos, sin) * flip(q)
    return out


def exact(case, seed):
    do = case["do"]
    seeds = _seeds(case["streams"], seed)
    if do == "jump" or case.get("kind") in ("u32", "u64"):
        return None          # whole numbers
    which = 64 if do == "generate64" else case["params"]
    if do in ("batch", "serve"):
        calls = _calls(case)
        at, size = _places(calls)
        lengths = {}
        for s, kind, count in calls:
            lengths[s] = lengths.get(s, 0) + _words(kind, count)
        if sum(lengths.values()) > 1 << 28 or max(lengths.values()) > 64 * MOST_ROUNDS:
            return None
        order = sorted(lengths, key=lambda s: -lengths[s])
        g = _Generator(seeds[np.array(order)], which)
        words = {s: torch.empty(lengths[s], dtype=torch.int64, device="cuda") for s in order}
        done, live = 0, len(order)
        while live:
            part = min(lengths[order[live - 1]] - done, 1 << 16)
            got = g.more(part)
            for i in range(live):
                words[order[i]][done:done + part] = got[i]
            done += part
            while live and lengths[order[live - 1]] == done:
                live -= 1
            g.keep(live)
        out = {k: torch.zeros(max(4, size[k]), dtype=torch.float64, device="cuda") for k in KINDS}
        pos = dict.fromkeys(lengths, 0)
        for (s, kind, count), a in zip(calls, at):
            if kind != "u32":
                out[kind][a:a + count] = _value(kind, words[s][pos[s]:pos[s] + _words(kind, count)])[:count]
            pos[s] += _words(kind, count)
        out["u32"] = None
        return out
    streams, n = case["streams"], case["n"]
    total = _words(case["kind"], n)
    if streams * total > MOST_WORDS + (1 << 24) or total > 64 * MOST_ROUNDS:
        return None
    kind = "uniform64" if do == "generate64" else case["kind"]
    g = _Generator(seeds, which)
    if do == "sum":
        acc = torch.zeros(streams, dtype=torch.float64, device="cuda")
        for k in range(0, total, 1 << 14):
            z = _value(kind, g.more(min(1 << 14, total - k)))
            acc += z[:, :min(1 << 14, n - k)].sum(1)
        return acc
    out = torch.empty(streams, total, dtype=torch.float64, device="cuda")
    for k in range(0, total, 1 << 14):
        out[:, k:k + (1 << 14)] = _value(kind, g.more(min(1 << 14, total - k)))
    return out[:, :n].contiguous()

// Host runtime of the 64-bit-word generators: contexts with device-resident
// state, argument checking, launch choice, host-output staging, autotuning,
// and the extern "C" entry points of include/xorgens_w64.h.
#include "xorgens_w64.h"

#include <algorithm>
#include <cstring>
#include <mutex>
#include <new>

#include "xg_cut.h"
#include "xg_gf2_tc.h"
#include "xg_jump.h"
#include "xg_runtime.h"
#include "xg_w64.h"

using xg::cuda_fail;
using xg::fail;

struct xg_w64_ctx {
    int device = 0;
    int sm_count = 148;
    uint32_t n = 0;
    uint32_t weyl_on = 1;
    cudaStream_t stream = nullptr;
    void* state_mem = nullptr;
    size_t state_bytes = 0;
    xg64::State st{};
    int cfg[2] = {-1, -1};
    int blk[2] = {0, 0};
    void* staging = nullptr;
    size_t staging_bytes = 0;
    uint64_t split_words = 0;   // cut calls: 0 automatic, 1 never, else the piece length
    xg::CutWorkspace cut;
    xg::TcStatus tc;            // of cut calls, jumps and substreams
    // xg_w64_jump's workspace (grow-only, freed with the context): a call ends
    // synchronised, so that no use outlives it.  16384 streams, 404 us per jump
    // with an allocation per call, 148 us without
    void* jump_ws = nullptr;
    size_t jump_ws_bytes = 0;
    std::mutex mu;
};

namespace {

#define XG_CUDA(call, what)                                \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

bool is_device_pointer(const void* p)
{
    cudaPointerAttributes attr{};
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
}

// XG_EDEVICE, once, when a tensor-core kernel of an earlier call gave up
// waiting: looked at by every call that reads or advances streams.
xg_status earlier_failure(xg_w64_ctx* c)
{
    return c->tc.take() ? fail(XG_EDEVICE, "a tensor-core kernel of this context gave up waiting: the outputs of that "
                                           "call and the streams it advanced are not valid")
                        : XG_OK;
}

// Without a tuned choice, one warp per stream: the fastest shape for both
// outputs in a sweep of 100 .. 65536 streams (ps per output at 1000 / 8000 /
// 16384 streams: u64 1.59 / 1.21 / 1.16 against 2.39 / 1.27 / 1.20 at (16,2)
// and 4.19 / 1.95 / 2.04 at (8,4); uniforms 1.90 / 1.52 / 1.43 against
// 2.66 / 1.54 / 1.47 and 4.62 / 1.85 / 1.56), and its stores are whole lines
// at every row address (rows of an odd length at (8,4): 3.62).
int pick_cfg(const xg_w64_ctx* c, int kind)
{
    return c->cfg[kind] >= 0 ? c->cfg[kind] : xg64::cfg_index(32, 1);
}

xg_status enqueue(xg_w64_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* d_out,
                  uint64_t ld, int force_cfg = -1, int force_block = 0)
{
    xg64::GenArgs a{};
    a.st = c->st;
    a.first = first;
    a.nstreams = nstreams;
    a.n = n;
    a.out = d_out;
    a.ld = ld;
    a.omega = c->weyl_on ? xg64::kOmega : 0;
    const int cfg = force_cfg >= 0 ? force_cfg : pick_cfg(c, kind);
    int block = force_block;
    if (block <= 0) block = (c->cfg[kind] == cfg && c->blk[kind] > 0) ? c->blk[kind] : xg64::kCfgs[cfg].block;
    const bool vec = ((reinterpret_cast<uintptr_t>(d_out) & 15u) == 0) && (nstreams == 1 || ld % 2 == 0);
    cudaError_t e = xg64::launch_gen(cfg, kind, vec, block, a, c->stream);
    return e == cudaSuccess ? XG_OK : cuda_fail(e, "64-bit generate kernel launch");
}

// log2 of the piece length that a device call is cut into (one stream is one
// serial chain of one warp), 0 for a whole call.  A piece length set by the
// caller applies to at most 16 streams of at least 2^18 outputs; by itself the
// library cuts where its prediction says so, unless a launch shape was set or
// tuned for other calls than those.  Not while the stream is being captured: a
// first use builds matrices and the workspace.
//
// 16 streams of 400000 words: 476 us whole, 1648 us in pieces of 2^16 words
// with one launch per stream and a doubling step per factor of two (the
// earlier form of the cut), 52 us this way; one stream 131 and 28 us; 200
// streams of 400000 FP64 uniforms 505 us whole, 211 us.
int cut_length(const xg_w64_ctx* c, int kind, uint32_t nstreams, uint64_t n)
{
    if (c->split_words == 1 || n < (uint64_t(1) << 13)) return 0;
    const bool always = nstreams <= 16 && n >= (uint64_t(1) << 18);   // whatever the launch shape set
    if (!always && (c->split_words > 1 || c->cfg[kind] >= 0)) return 0;
    const int q = xg::cut_choose(kind == xg64::kU64 ? xg::kCutU64 : xg::kCutUniform64, nstreams, n, c->sm_count,
                                 c->split_words);
    if (!q) return 0;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c->stream, &cap) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return cap == cudaStreamCaptureStatusNone ? q : 0;
}

// The call in pieces of 2^q outputs; *ran = false when the whole call is to be
// taken (no memory for the workspace).  The output is exactly the whole call's.
xg_status generate_cut(xg_w64_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* d_out, uint64_t ld,
                       int q, bool* ran)
{
    // the prologue reads windows and rings as 32-bit words, two per word
    static_assert(xg64::kWin * 2 == xg::kWin && xg64::kRingBase * 2 == xg::kRingBase && xg64::kR * 2 == 128,
                  "window layout in 32-bit words");
    const uint32_t pieces = (uint32_t)((n + (uint64_t(1) << q) - 1) >> q);
    const xg::CutStreams streams{c->device, c->sm_count, xg::kJumpSetW64, reinterpret_cast<const uint32_t*>(c->st.win),
                                 c->st.pend, reinterpret_cast<const uint32_t*>(c->st.weyl), 2, &c->tc};
    xg::CutRings r{};
    xg_status st = xg::cut_prologue(c->cut, streams, first, nstreams, pieces, q, 0, c->stream, &r, ran);
    if (st != XG_OK || !*ran) return st;
    xg64::CutArgs a{};
    a.st = c->st;
    a.first = first;
    a.nstreams = nstreams;
    a.pieces = pieces;
    a.log2_len = (uint32_t)q;
    a.n = n;
    a.out = d_out;
    a.ld = ld;
    a.rings = reinterpret_cast<const uint64_t*>(r.rings);
    a.weyl0 = reinterpret_cast<const uint64_t*>(r.weyl0);
    a.omega = c->weyl_on ? xg64::kOmega : 0;
    const cudaError_t e = xg64::launch_cut(kind, a, c->stream);
    st = c->cut.release(c->stream);
    return e == cudaSuccess ? st : cuda_fail(e, "64-bit cut generation");
}

// Host output: generate into one device buffer piece by piece and copy each
// piece out (synchronously); pieces split the stream range and, for long
// requests, each stream's length.
xg_status to_host(xg_w64_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* h_out,
                  uint64_t ld)
{
    const size_t kPieceBytes = size_t(128) << 20;
    if (c->staging_bytes < kPieceBytes) {
        if (c->staging) cudaFree(c->staging);
        c->staging = nullptr;
        c->staging_bytes = 0;
        XG_CUDA(cudaMalloc(&c->staging, kPieceBytes), "cudaMalloc(staging)");
        c->staging_bytes = kPieceBytes;
    }
    const uint64_t words = kPieceBytes / 8;
    const uint64_t ncols = std::max<uint64_t>(1, std::min<uint64_t>(n, words));
    const uint64_t ld_stage = align_up(ncols, 2);
    const uint32_t rows_per = (uint32_t)std::max<uint64_t>(1, words / ld_stage);
    for (uint32_t r0 = 0; r0 < nstreams; r0 += rows_per) {
        const uint32_t rows = std::min<uint32_t>(rows_per, nstreams - r0);
        for (uint64_t c0 = 0; c0 < n; c0 += ncols) {
            const uint64_t cols = std::min<uint64_t>(ncols, n - c0);
            xg_status st = enqueue(c, kind, first + r0, rows, cols, c->staging, ld_stage);
            if (st != XG_OK) return st;
            char* dst = static_cast<char*>(h_out) + ((uint64_t)r0 * ld + c0) * 8;
            XG_CUDA(cudaMemcpy2DAsync(dst, ld * 8, c->staging, ld_stage * 8, cols * 8, rows,
                                      cudaMemcpyDeviceToHost, c->stream),
                    "cudaMemcpy2DAsync(device to host)");
        }
    }
    XG_CUDA(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    return XG_OK;
}

xg_status generate(xg_w64_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* out,
                   uint64_t ld)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if ((uint64_t)first + nstreams > c->n)
        return fail(XG_EINVAL, "streams [%u, %u) out of range (context has %u)", first, first + nstreams, c->n);
    if (nstreams == 0 || n == 0) return XG_OK;
    if (!out) return fail(XG_EINVAL, "null output pointer");
    if (nstreams > 1 && ld < n)
        return fail(XG_EINVAL, "ld (%llu) < n_per_stream (%llu)", (unsigned long long)ld, (unsigned long long)n);
    if (nstreams == 1 && ld < n) ld = n;
    if (ld > (UINT64_MAX / 16) / nstreams) return fail(XG_EINVAL, "output extent overflows");
    if (reinterpret_cast<uintptr_t>(out) & 7u) return fail(XG_EINVAL, "output must be 8-byte aligned");
    std::lock_guard<std::mutex> lk(c->mu);
    if (xg_status f = earlier_failure(c)) return f;
    if (is_device_pointer(out)) {
        if (const int q = cut_length(c, kind, nstreams, n)) {
            bool ran = false;
            const xg_status st = generate_cut(c, kind, first, nstreams, n, out, ld, q, &ran);
            if (ran || st != XG_OK) return st;
        }
        return enqueue(c, kind, first, nstreams, n, out, ld);
    }
    const xg_status st = to_host(c, kind, first, nstreams, n, out, ld);
    return st == XG_OK ? earlier_failure(c) : st;
}

}  // namespace

extern "C" {

xg_status xg_w64_params(uint32_t* rsabcd, uint64_t* omega)
{
    if (!rsabcd || !omega) return fail(XG_EINVAL, "null output");
    const uint32_t v[6] = {xg64::kR, xg64::kS, xg64::kA, xg64::kB, xg64::kC, xg64::kD};
    std::memcpy(rsabcd, v, sizeof v);
    *omega = xg64::kOmega;
    return XG_OK;
}

xg_status xg_w64_create(xg_w64_ctx** out, uint32_t n_streams, uint32_t weyl_on, void* cuda_stream)
{
    if (!out) return fail(XG_EINVAL, "null output handle");
    *out = nullptr;
    if (n_streams == 0) return fail(XG_EINVAL, "n_streams must be positive");
    xg_w64_ctx* c = new (std::nothrow) xg_w64_ctx();
    if (!c) return fail(XG_ENOMEM, "host allocation failed");
    c->n = n_streams;
    c->weyl_on = weyl_on ? 1u : 0u;
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e = cudaGetDevice(&c->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device);
    const size_t off_weyl = align_up((size_t)n_streams * xg64::kWin * 8, 256);
    const size_t off_pend = align_up(off_weyl + (size_t)n_streams * 8, 256);
    const size_t off_pos = align_up(off_pend + (size_t)n_streams * 4, 256);
    const size_t total = off_pos + (size_t)n_streams * 8;
    if (e == cudaSuccess) e = cudaMalloc(&c->state_mem, total);
    if (e != cudaSuccess) {
        xg_status st = e == cudaErrorMemoryAllocation ? fail(XG_ENOMEM, "cudaMalloc(state, %zu bytes) failed", total)
                                                      : cuda_fail(e, "create");
        cudaGetLastError();
        delete c;
        return st;
    }
    c->state_bytes = total;
    char* base = static_cast<char*>(c->state_mem);
    c->st.win = reinterpret_cast<uint64_t*>(base);
    c->st.weyl = reinterpret_cast<uint64_t*>(base + off_weyl);
    c->st.pend = reinterpret_cast<uint32_t*>(base + off_pend);
    c->st.pos = reinterpret_cast<uint64_t*>(base + off_pos);
    e = cudaMemsetAsync(c->state_mem, 0, total, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        xg_status st = cuda_fail(e, "create");
        xg_w64_destroy(c);
        return st;
    }
    *out = c;
    return XG_OK;
}

xg_status xg_w64_destroy(xg_w64_ctx* c)
{
    if (!c) return XG_OK;
    if (c->state_mem) cudaStreamSynchronize(c->stream);
    if (c->staging) cudaFree(c->staging);
    c->cut.destroy();
    const xg_status failed = earlier_failure(c);
    if (c->jump_ws) cudaFree(c->jump_ws);
    if (c->state_mem) cudaFree(c->state_mem);
    delete c;
    return failed;
}

xg_status xg_w64_set_stream(xg_w64_ctx* c, void* cuda_stream)
{
    if (!c) return fail(XG_EINVAL, "null context");
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    return XG_OK;
}

xg_status xg_w64_seed(xg_w64_ctx* c, uint32_t first, uint32_t count, const uint32_t* host_seeds)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if ((uint64_t)first + count > c->n) return fail(XG_EINVAL, "seed range out of bounds");
    if (count == 0) return XG_OK;
    if (!host_seeds) return fail(XG_EINVAL, "null seeds");
    std::lock_guard<std::mutex> lk(c->mu);
    uint32_t* d = nullptr;
    XG_CUDA(cudaMallocAsync(reinterpret_cast<void**>(&d), (size_t)count * 4, c->stream), "cudaMallocAsync(seeds)");
    cudaError_t e = cudaMemcpyAsync(d, host_seeds, (size_t)count * 4, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = xg64::launch_seed(c->st, d, first, count, c->stream);
    cudaError_t e2 = cudaFreeAsync(d, c->stream);
    if (e != cudaSuccess) return cuda_fail(e, "seed");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFreeAsync(seeds)");
    if (!c->weyl_on)
        XG_CUDA(cudaMemsetAsync(c->st.weyl + first, 0, (size_t)count * 8, c->stream), "cudaMemsetAsync");
    return XG_OK;
}

xg_status xg_w64_get_state(xg_w64_ctx* c, uint32_t stream, uint64_t* ring, uint64_t* weyl)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if (stream >= c->n) return fail(XG_EINVAL, "stream %u out of range", stream);
    if (!ring || !weyl) return fail(XG_EINVAL, "null output");
    std::lock_guard<std::mutex> lk(c->mu);
    uint64_t win[xg64::kWin], w = 0;
    uint32_t pend = 0;
    XG_CUDA(cudaMemcpyAsync(win, c->st.win + (size_t)stream * xg64::kWin, sizeof win, cudaMemcpyDeviceToHost,
                            c->stream), "get_state");
    XG_CUDA(cudaMemcpyAsync(&pend, c->st.pend + stream, 4, cudaMemcpyDeviceToHost, c->stream), "get_state");
    XG_CUDA(cudaMemcpyAsync(&w, c->st.weyl + stream, 8, cudaMemcpyDeviceToHost, c->stream), "get_state");
    XG_CUDA(cudaStreamSynchronize(c->stream), "get_state");
    if (xg_status f = earlier_failure(c)) return f;
    if (pend >= (uint32_t)xg64::kRingBase) return fail(XG_EDEVICE, "corrupt stream state (pend %u)", pend);
    std::memcpy(ring, win + xg64::kRingBase - pend, xg64::kR * 8);
    *weyl = w;
    return XG_OK;
}

xg_status xg_w64_set_state(xg_w64_ctx* c, uint32_t stream, const uint64_t* ring, uint64_t weyl)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if (stream >= c->n) return fail(XG_EINVAL, "stream %u out of range", stream);
    if (!ring) return fail(XG_EINVAL, "null ring");
    std::lock_guard<std::mutex> lk(c->mu);
    if (xg_status f = earlier_failure(c)) return f;
    uint64_t win[xg64::kWin] = {0};
    std::memcpy(win + xg64::kRingBase, ring, xg64::kR * 8);
    const uint32_t pend = 0;
    const uint64_t w = c->weyl_on ? weyl : 0;
    XG_CUDA(cudaMemcpyAsync(c->st.win + (size_t)stream * xg64::kWin, win, sizeof win, cudaMemcpyHostToDevice,
                            c->stream), "set_state");
    XG_CUDA(cudaMemcpyAsync(c->st.pend + stream, &pend, 4, cudaMemcpyHostToDevice, c->stream), "set_state");
    XG_CUDA(cudaMemcpyAsync(c->st.weyl + stream, &w, 8, cudaMemcpyHostToDevice, c->stream), "set_state");
    XG_CUDA(cudaStreamSynchronize(c->stream), "set_state");
    return XG_OK;
}

xg_status xg_w64_generate_u64(xg_w64_ctx* c, uint32_t first, uint32_t nstreams, uint64_t n, uint64_t* out,
                              uint64_t ld)
{
    return generate(c, xg64::kU64, first, nstreams, n, out, ld);
}

xg_status xg_w64_generate_uniform_f64(xg_w64_ctx* c, uint32_t first, uint32_t nstreams, uint64_t n, double* out,
                                      uint64_t ld)
{
    return generate(c, xg64::kUniformF64, first, nstreams, n, out, ld);
}

xg_status xg_w64_set_split(xg_w64_ctx* c, uint64_t piece_words)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if (piece_words > 1 && (piece_words < 64 || (piece_words & (piece_words - 1))))
        return fail(XG_EINVAL, "piece length must be 0, 1 or a power of two >= 64");
    c->split_words = piece_words;
    return XG_OK;
}

static xg_status ensure_jump_ws(xg_w64_ctx* c, size_t bytes)
{
    if (c->jump_ws_bytes >= bytes) return XG_OK;
    if (c->jump_ws) cudaFree(c->jump_ws);
    c->jump_ws = nullptr;
    c->jump_ws_bytes = 0;
    if (cudaMalloc(&c->jump_ws, bytes) != cudaSuccess) {
        cudaGetLastError();
        c->jump_ws = nullptr;
        return fail(XG_ENOMEM, "cudaMalloc(xg_w64_jump workspace, %zu bytes) failed", bytes);
    }
    c->jump_ws_bytes = bytes;
    return XG_OK;
}

xg_status xg_w64_jump(xg_w64_ctx* c, uint32_t first, uint32_t nstreams, uint64_t words)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if ((uint64_t)first + nstreams > c->n) return fail(XG_EINVAL, "streams out of range");
    if (nstreams == 0 || words == 0) return XG_OK;
    std::lock_guard<std::mutex> lk(c->mu);
    if (xg_status f = earlier_failure(c)) return f;
    cudaStream_t s = c->stream;
    int top = 63;
    while (!((words >> top) & 1)) --top;
    xg_status st = XG_OK;
    for (int k = 0; k <= top; ++k)
        if (((words >> k) & 1) && !xg::jump_matrix(c->device, xg::kJumpSetW64, k, s, &st)) return st;
    const uint64_t omega = c->weyl_on ? xg64::kOmega : 0;
    const bool in_place = xg::gf2_jump_in_place(c->device, xg::kJumpSetW64, nstreams, words, c->tc, s) &&
                          ensure_jump_ws(c, xg::gf2_jump_work_bytes(c->device, nstreams, words, true)) == XG_OK;
    cudaError_t e;
    if (in_place) {
        // the windows as 32-bit words, two per word (layout checked in generate_cut)
        e = xg::gf2_jump_windows(c->device, xg::kJumpSetW64, words,
                                 xg::JumpWindows{reinterpret_cast<uint32_t*>(c->st.win + (size_t)first * xg64::kWin),
                                                 c->st.pend + first, 2},
                                 nstreams, static_cast<uint8_t*>(c->jump_ws), c->tc, c->sm_count, s, &st);
        if (e == cudaSuccess) e = xg64::launch_finish_jump(c->st, first, nstreams, words, omega, s);
    } else {
        // one allocation: rings[0, n) hold the states, rings[n, 2n) the second
        // buffer (the shared GF(2) kernels work on 4096-bit states as 128 32-bit
        // words); index lists (0 .. n-1, then 0 .. 2n-1, built on the device);
        // the jump's work area
        const size_t rings_bytes = (size_t)2 * nstreams * xg64::kR * 8;
        const size_t work_off = (rings_bytes + (size_t)3 * nstreams * 4 + 255) / 256 * 256;
        const size_t wbytes = xg::gf2_jump_work_bytes(c->device, nstreams, words, false);
        if (xg_status g = ensure_jump_ws(c, work_off + wbytes)) return g;
        char* ws = static_cast<char*>(c->jump_ws);
        uint64_t* rings = reinterpret_cast<uint64_t*>(ws);
        uint32_t* rings32 = reinterpret_cast<uint32_t*>(ws);
        uint32_t* ids = reinterpret_cast<uint32_t*>(ws + rings_bytes);
        const uint32_t* lo_idx = ids + nstreams;  // 0 .. 2n-1
        e = xg::launch_jump_index(ids, nstreams, 0u, s);
        if (e == cudaSuccess) e = xg64::launch_gather_rings(c->st, first, nstreams, rings, s);
        bool hi = false;
        if (e == cudaSuccess)
            e = xg::gf2_jump_states(c->device, xg::kJumpSetW64, words, rings32, nstreams, lo_idx,
                                    reinterpret_cast<uint8_t*>(ws + work_off), c->tc, c->sm_count, s, &st, &hi);
        if (e == cudaSuccess)
            e = xg64::launch_scatter_rings(c->st, first, nstreams, hi ? rings + (size_t)nstreams * xg64::kR : rings,
                                           words, omega, s);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (st != XG_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "xg_w64_jump");
    return earlier_failure(c);
}

xg_status xg_w64_seed_substreams(xg_w64_ctx* c, uint32_t first, uint32_t count, uint32_t seed,
                                 uint32_t log2_spacing)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if ((uint64_t)first + count > c->n) return fail(XG_EINVAL, "streams out of range");
    if (count == 0) return XG_OK;
    int steps = 0;   // doubling steps: bits of count - 1
    while (steps < 32 && ((uint64_t)(count - 1) >> steps)) ++steps;
    if (log2_spacing > 63 || (count > 1 && (int)log2_spacing + steps > 64))
        return fail(XG_EINVAL, "(count - 1) * 2^%u does not fit in 64 bits", log2_spacing);
    if (xg_status s = xg_w64_seed(c, first, 1, &seed)) return s;
    std::lock_guard<std::mutex> lk(c->mu);
    cudaStream_t s = c->stream;
    const int q = (int)log2_spacing;
    xg_status st = XG_OK;
    for (int b = 0; b < steps; ++b)
        if (!xg::jump_matrix(c->device, xg::kJumpSetW64, q + b, s, &st)) return st;
    // step b takes the states m - 2^b to the states m, m in [2^b, min(2^(b+1), count)):
    // its sources are the identity list from 0 and its destinations the same
    // list from 2^b, so one device-built list 0 .. 2 count - 1 serves every step
    uint32_t most = 0;
    for (int b = 0; b < steps; ++b) {
        const uint32_t lo = 1u << b, hi = (uint32_t)std::min<uint64_t>((uint64_t)lo << 1, count);
        most = std::max(most, hi - lo);
    }
    // one workspace: rings of all count states; the index lists (0 .. count - 1,
    // then 0 .. 2 count - 1); the base Weyl word (8-byte aligned); the
    // tensor-core operand (256-byte aligned, when used)
    const size_t rings_bytes = (size_t)count * xg64::kR * 8;
    const size_t ids_off = rings_bytes;
    const size_t w0_off = (ids_off + (size_t)3 * count * 4 + 7) / 8 * 8;
    const size_t tc_off = (w0_off + 8 + 255) / 256 * 256;
    const size_t tc_bytes = xg::gf2_apply_scratch(c->device, most);
    char* ws = nullptr;
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&ws), tc_off + tc_bytes, s);
    if (e != cudaSuccess) return cuda_fail(e, "xg_w64_seed_substreams scratch");
    uint64_t* rings = reinterpret_cast<uint64_t*>(ws);
    uint32_t* ids = reinterpret_cast<uint32_t*>(ws + ids_off);
    const uint32_t* iota = ids + count;
    uint64_t* d_w0 = reinterpret_cast<uint64_t*>(ws + w0_off);
    uint8_t* tc_scratch = tc_bytes ? reinterpret_cast<uint8_t*>(ws + tc_off) : nullptr;
    uint32_t* rings32 = reinterpret_cast<uint32_t*>(rings);
    e = xg::launch_jump_index(ids, count, 0u, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_w0, c->st.weyl + first, 8, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = xg64::launch_gather_rings(c->st, first, 1, rings, s);
    // the destinations 1 .. count - 1, zeroed once for all the steps
    if (e == cudaSuccess && count > 1)
        e = cudaMemsetAsync(rings + xg64::kR, 0, (size_t)(count - 1) * xg64::kR * 8, s);
    for (int b = 0; b < steps && e == cudaSuccess; ++b) {
        const uint32_t lo = 1u << b, hi = (uint32_t)std::min<uint64_t>((uint64_t)lo << 1, count);
        e = xg::gf2_apply(c->device, xg::kJumpSetW64, q + b, rings32, hi - lo, iota, iota + lo, tc_scratch,
                          c->tc, c->sm_count, s, &st, true);
    }
    if (e == cudaSuccess)
        e = xg64::launch_substream_scatter(c->st, first, count, rings, d_w0, q, c->weyl_on ? xg64::kOmega : 0, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(ws, s);
    if (st != XG_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "xg_w64_seed_substreams");
    return earlier_failure(c);
}

xg_status xg_w64_transform_uniform_f64(xg_w64_ctx* c, const uint64_t* d_words, uint64_t n, double* d_out)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if (n == 0) return XG_OK;
    if (!d_words || !d_out) return fail(XG_EINVAL, "null pointer");
    if ((reinterpret_cast<uintptr_t>(d_words) | reinterpret_cast<uintptr_t>(d_out)) & 7u)
        return fail(XG_EINVAL, "buffers must be 8-byte aligned");
    cudaError_t e = xg64::launch_transform_uniform(d_words, n, reinterpret_cast<uint64_t*>(d_out), c->sm_count,
                                                   c->stream);
    return e == cudaSuccess ? XG_OK : cuda_fail(e, "64-bit transform_uniform");
}

xg_status xg_w64_set_launch(xg_w64_ctx* c, xg_w64_type type, uint32_t tpg, uint32_t wpl, uint32_t block)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if ((unsigned)type > XG_W64_UNIFORM_F64) return fail(XG_EINVAL, "unknown output type");
    if (block > 1024 || (block & 31u)) return fail(XG_EINVAL, "block must be a multiple of 32, at most 1024");
    if (tpg == 0 && wpl == 0) {
        c->cfg[type] = -1;
        c->blk[type] = 0;
        return XG_OK;
    }
    const int ci = xg64::cfg_index((int)tpg, (int)wpl);
    if (ci < 0) return fail(XG_EINVAL, "unsupported launch (tpg %u, wpl %u)", tpg, wpl);
    c->cfg[type] = ci;
    c->blk[type] = (int)block;
    return XG_OK;
}

xg_status xg_w64_autotune(xg_w64_ctx* c, xg_w64_type type, uint32_t nstreams, uint64_t n_per_stream,
                          uint32_t* tpg, uint32_t* wpl, uint32_t* block, float* best_ms)
{
    if (!c) return fail(XG_EINVAL, "null context");
    if ((unsigned)type > XG_W64_UNIFORM_F64) return fail(XG_EINVAL, "unknown output type");
    if (nstreams == 0 || nstreams > c->n) nstreams = c->n;
    if (n_per_stream == 0) return fail(XG_EINVAL, "n_per_stream must be positive");
    uint64_t nt = std::min<uint64_t>(n_per_stream, std::max<uint64_t>(128, (uint64_t(1) << 26) / nstreams));
    nt = align_up(nt, 32);
    std::lock_guard<std::mutex> lk(c->mu);
    if (xg_status f = earlier_failure(c)) return f;
    void* saved = nullptr;
    void* out = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    auto cleanup = [&]() {
        if (saved) {
            cudaMemcpyAsync(c->state_mem, saved, c->state_bytes, cudaMemcpyDeviceToDevice, c->stream);
            cudaStreamSynchronize(c->stream);
            cudaFree(saved);
        }
        if (out) cudaFree(out);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
    };
    cudaError_t e = cudaMalloc(&saved, c->state_bytes);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(saved, c->state_mem, c->state_bytes, cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess) e = cudaMalloc(&out, (size_t)nstreams * nt * 8);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e != cudaSuccess) {
        cleanup();
        cudaGetLastError();
        return cuda_fail(e, "autotune set-up");
    }
    static const int kBlocks[] = {32, 64, 128, 256};
    int best_cfg = -1, best_block = 0;
    float best = 1e30f;
    xg_status st = XG_OK;
    for (int ci = 0; ci < xg64::kNumCfgs && st == XG_OK; ++ci) {
        for (int b : kBlocks) {
            st = enqueue(c, type, 0, nstreams, nt, out, nt, ci, b);
            if (st != XG_OK) break;
            cudaEventRecord(e0, c->stream);
            for (int r = 0; r < 3 && st == XG_OK; ++r) st = enqueue(c, type, 0, nstreams, nt, out, nt, ci, b);
            cudaEventRecord(e1, c->stream);
            if (cudaEventSynchronize(e1) != cudaSuccess) {
                st = cuda_fail(cudaGetLastError(), "autotune timing");
                break;
            }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            ms /= 3.f;
            if (ms < best) {
                best = ms;
                best_cfg = ci;
                best_block = b;
            }
        }
    }
    cleanup();
    if (st != XG_OK) return st;
    c->cfg[type] = best_cfg;
    c->blk[type] = best_block;
    if (tpg) *tpg = (uint32_t)xg64::kCfgs[best_cfg].tpg;
    if (wpl) *wpl = (uint32_t)xg64::kCfgs[best_cfg].wpl;
    if (block) *block = (uint32_t)best_block;
    if (best_ms) *best_ms = best;
    return XG_OK;
}

}  // extern "C"

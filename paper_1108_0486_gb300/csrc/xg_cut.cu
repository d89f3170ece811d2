// Cut calls (see xg_cut.h): choice of the piece length, the jump-ahead
// prologue and its launch.
//
// One stream is a serial chain of rounds that one warp runs (Sec. 2), so a
// call on few streams leaves most of the GPU idle.  Piece m of a stream starts
// from its ring advanced by m 2^q words.  The prologue computes those rings in
// a few steps: a step takes the pieces m < B of every stream to the pieces
// m + j B, j = 1 .. J, with the matrices M^(j B 2^q).  All of it is regular,
// so the index lists are built on the device and nothing is uploaded.
//
// One stream of 2^20 words: 73 us with a planned batch (two uploads, a gather,
// five doubling steps, pieces of 2^15 words), 26 us this way; 500 streams of
// 500000 normals 537 us whole, 379 us cut; 200 streams of 2^18 words 153 and 70.
#include "xg_cut.h"

#include <algorithm>

#include "xg_gf2_tc.h"
#include "xg_jump.h"
#include "xg_launch.h"
#include "xg_runtime.h"

namespace xg {
namespace {

constexpr int kMaxSteps = 32;
constexpr uint64_t kMaxPieces = uint64_t(1) << 22;   // 2 GiB of rings

// One prologue step: sources are the pieces m < have of every stream,
// destinations m + j have for j = 1 .. mats (kNoState past the last piece).
struct Step {
    uint32_t have;
    uint32_t mats;
    uint32_t tc;    // by the tensor cores, where they are to be had
    uint64_t at;    // its sources in the list, then mats destination lists
};
struct Steps {
    Step step[kMaxSteps];
    int n;
    uint64_t entries;
};

// Up to 7 matrices per step, which makes the pieces eight times as many.  By
// the table kernel as long as the results are few, where a step costs a launch
// and the matrix read rather than the lookups (0.05 us per result); by the
// tensor cores from kTcMinResults on, where it costs the launches and one
// tile's time and hardly more for seven matrices than for one.  The price of a
// step (cut_prologue_us) and its launch go by the same limit.
Steps plan_steps(uint32_t nstreams, uint32_t pieces)
{
    Steps p{};
    for (uint64_t have = 1; have < pieces && p.n < kMaxSteps; ++p.n) {
        const uint64_t sources = have * nstreams;
        const uint64_t left = std::min<uint64_t>(7, (pieces + have - 1) / have - 1);
        p.step[p.n] = Step{(uint32_t)have, (uint32_t)left, sources * left >= kTcMinResults ? 1u : 0u, p.entries};
        p.entries += sources * (1 + left);
        have *= 1 + left;
    }
    return p;
}

// Piece 0 of a stream takes its ring, the other pieces zero rings (the table
// kernel XORs into them); weyl0[i] = stream i's Weyl word; then the lists of
// all steps.  A warp per piece, 8 to a block; blocks past the pieces write
// the lists.
__global__ void __launch_bounds__(256) cut_setup_kernel(CutStreams st, uint32_t first, uint32_t nstreams,
                                                        uint32_t pieces, uint32_t piece_blocks,
                                                        uint32_t* __restrict__ rings, uint32_t* __restrict__ weyl0,
                                                        Steps steps, uint32_t* __restrict__ lists)
{
    cudaTriggerProgrammaticLaunchCompletion();
    if (blockIdx.x < piece_blocks) {
        const uint32_t p = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
        if (p >= nstreams * pieces) return;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (p % pieces == 0) {
            const uint32_t s = first + p / pieces;
            const uint32_t* src = st.win + (size_t)s * kWin + (kRingBase - st.pend[s] * st.word) + 4 * lane;
            v = make_uint4(src[0], src[1], src[2], src[3]);
            if (lane < st.word) weyl0[p / pieces * st.word + lane] = st.weyl[(size_t)s * st.word + lane];
        }
        reinterpret_cast<uint4*>(rings + (size_t)p * 128)[lane] = v;
        return;
    }
    const uint64_t e = (uint64_t)(blockIdx.x - piece_blocks) * 256 + threadIdx.x;
    if (e >= steps.entries) return;
    int k = 0;
    while (k + 1 < steps.n && e >= steps.step[k + 1].at) ++k;
    const uint32_t have = steps.step[k].have, sources = have * nstreams;
    const uint64_t r = e - steps.step[k].at;
    const uint32_t j = (uint32_t)(r / sources), x = (uint32_t)(r % sources);   // j = 0: the sources
    const uint32_t i = x / have, m = x % have + j * have;
    lists[e] = m < pieces ? i * pieces + m : kNoState;
}

// sums[i] = the sum of stream i's pieces' sums, in FP64 and rounded once.  A
// warp per stream.
__global__ void __launch_bounds__(64) cut_sum_kernel(const float* __restrict__ piece_sums, uint32_t pieces,
                                                     uint32_t nstreams, float* __restrict__ sums)
{
    const uint32_t i = blockIdx.x * 2 + threadIdx.x / 32, lane = threadIdx.x % 32;
    cudaGridDependencySynchronize();
    if (i >= nstreams) return;
    double acc = 0.0;
    for (uint32_t m = lane; m < pieces; m += 32) acc += (double)piece_sums[(size_t)i * pieces + m];
#pragma unroll
    for (int off = 16; off >= 1; off /= 2) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (lane == 0) sums[i] = (float)acc;
}

// Time of one word on a sub-partition of an SM that runs w warps, in ns,
// fitted to a sweep of 100 .. 4000 whole streams: one warp alone is bound by
// its own chain, several by the pipes.
double word_ns(int kind, double w)
{
    switch (kind) {
    case kU32: return std::max(0.585, 0.365 * w);
    case kUniform: return std::max(0.62, 0.42 * w);
    case kNormal: return std::max(1.18, 0.35 + 0.705 * w);
    case kNormalSum: return std::max(1.08, 0.27 + 0.67 * w);
    case kCutU64: return std::max(1.19, 0.735 * w);
    default: return std::max(1.26, 0.25 + 0.86 * w);   // kCutUniform64
    }
}

// While it lives, what this thread allocates and waits for is no part of a
// capture that another CUDA stream is in: in the default (global) capture mode
// that capture would be refused and invalidated.
class OutsideCaptures {
public:
    OutsideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode_); }
    ~OutsideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode_); }
    OutsideCaptures(const OutsideCaptures&) = delete;
    OutsideCaptures& operator=(const OutsideCaptures&) = delete;

private:
    cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};

}  // namespace

// The set-up launch, then per step a table-kernel launch
// or an application on the tensor cores (18 ns per operand row of a tile; the
// last wave is rarely full).
double cut_prologue_us(uint32_t nstreams, uint64_t pieces, int sm_count)
{
    const Steps p = plan_steps(nstreams, (uint32_t)pieces);
    double t = 5.0;
    for (int k = 0; k < p.n; ++k) {
        const uint64_t n = (uint64_t)p.step[k].have * nstreams;
        if (!p.step[k].tc) {
            t += 5.5 + 0.05 * (double)(n * p.step[k].mats);
        } else {
            uint32_t counts[kGf2TcMaxMats], waves = 1;
            for (uint32_t& c : counts) c = (uint32_t)n;
            const uint32_t bn = gf2_tc_tile(counts, (int)p.step[k].mats, sm_count, &waves);
            t += 11.4 + 0.018 * (double)(128 + bn) * (1.0 + 0.7 * (double)(waves - 1));
        }
    }
    return t;
}

int cut_choose(int kind, uint32_t nstreams, uint64_t n, int sm_count, uint64_t forced)
{
    const uint64_t words = kind == kNormal || kind == kNormalSum ? n + (n & 1u) : n;
    if (forced) {
        int q = 6;
        while ((uint64_t(1) << q) < forced) ++q;
        if (words < (uint64_t)2 << q || ((words + (uint64_t(1) << q) - 1) >> q) * nstreams > kMaxPieces) return 0;
        return q;
    }
    const double parts = 4.0 * sm_count;
    if (nstreams > 6 * parts) return 0;   // the pipes are busy as it is
    // warps on the fullest sub-partition: blocks of two warps over the SMs
    auto warps = [&](uint64_t blocks) { return (double)(((blocks + sm_count - 1) / sm_count + 1) / 2); };
    // A launch's own start and end are 3.5 us; a piece's ring comes from
    // memory that was just written.  5% in favour of the whole call, so that a
    // cut has to be clearly the faster.
    double best = 0.95 * (3.5 + 1e-3 * (double)words * word_ns(kind, warps((nstreams + 1) / 2)));
    int best_q = 0;
    for (int q = 12; q <= 32; ++q) {
        const uint64_t len = uint64_t(1) << q;
        if (words < 2 * len) break;
        const uint64_t pieces = (words + len - 1) / len;
        if (pieces * nstreams > kMaxPieces) continue;
        const double run = 6.0 + 1e-3 * (double)len * word_ns(kind, warps(nstreams * ((pieces + 1) / 2)));
        if (run >= best) continue;
        const double t = cut_prologue_us(nstreams, pieces, sm_count) + run + (kind == kNormalSum ? 2.0 : 0.0);
        if (t < best) {
            best = t;
            best_q = q;
        }
    }
    return best_q;
}

xg_status CutWorkspace::ensure(size_t want)
{
    if (bytes >= want) return XG_OK;
    if (mem) {
        if (used) cudaEventSynchronize(event);
        cudaFree(mem);
    }
    mem = nullptr;
    bytes = 0;
    if (!event && cudaEventCreateWithFlags(&event, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        event = nullptr;
        return fail(XG_ENOMEM, "cudaEventCreate(cut workspace) failed");
    }
    if (cudaMalloc(&mem, want) != cudaSuccess) {
        cudaGetLastError();
        mem = nullptr;
        return fail(XG_ENOMEM, "cudaMalloc(cut workspace, %zu bytes) failed", want);
    }
    bytes = want;
    return XG_OK;
}

xg_status CutWorkspace::acquire(cudaStream_t s)
{
    if (!used) return XG_OK;
    unsigned long long id = 0;
    cudaError_t e = cudaStreamGetId(s, &id);
    if (e == cudaSuccess && id != stream_id) e = cudaStreamWaitEvent(s, event, 0);
    if (e != cudaSuccess) return cuda_fail(e, "cut workspace");
    return XG_OK;
}

xg_status CutWorkspace::release(cudaStream_t s)
{
    cudaError_t e = cudaStreamGetId(s, &stream_id);
    if (e == cudaSuccess) e = cudaEventRecord(event, s);
    if (e != cudaSuccess) return cuda_fail(e, "cut workspace");
    used = true;
    return XG_OK;
}

void CutWorkspace::destroy()
{
    if (event) {
        if (used) cudaEventSynchronize(event);
        cudaEventDestroy(event);
    }
    if (mem) cudaFree(mem);
    *this = CutWorkspace{};
}

xg_status cut_prologue(CutWorkspace& ws, const CutStreams& streams, uint32_t first, uint32_t nstreams, uint32_t pieces,
                       int q, size_t extra_bytes, cudaStream_t s, CutRings* out, bool* ran)
{
    *ran = false;
    OutsideCaptures outside;   // the workspace, the matrices
    const uint32_t total = pieces * nstreams;
    const Steps steps = plan_steps(nstreams, pieces);
    uint32_t most_tc = 0;   // states of the largest tensor-core step
    bool use_tc[kMaxSteps] = {};
    for (int k = 0; k < steps.n; ++k) {
        const uint32_t m = steps.step[k].have * nstreams;
        use_tc[k] = steps.step[k].tc && gf2_use_tc(streams.device, m * steps.step[k].mats);
        if (use_tc[k]) most_tc = std::max(most_tc, m);
    }
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t weyl_off = (size_t)total * 512;
    const size_t list_off = up(weyl_off + (size_t)nstreams * streams.word * 4);
    const size_t tc_off = up(list_off + (size_t)steps.entries * 4);
    const size_t extra_off = up(tc_off + (most_tc ? gf2_tc_scratch_bytes(most_tc) : 0));
    if (ws.ensure(extra_off + extra_bytes) != XG_OK) return XG_OK;
    if (most_tc && !streams.tc->device()) return XG_OK;
    char* base = static_cast<char*>(ws.mem);
    uint32_t* rings = reinterpret_cast<uint32_t*>(base);
    uint32_t* weyl0 = reinterpret_cast<uint32_t*>(base + weyl_off);
    uint32_t* lists = reinterpret_cast<uint32_t*>(base + list_off);
    uint8_t* tc = reinterpret_cast<uint8_t*>(base + tc_off);
    // the matrices first: building one on its first use synchronises
    const uint64_t* mats[kMaxSteps][kMaxMats] = {};
    const uint8_t* tc_mats[kMaxSteps][kGf2TcMaxMats] = {};
    static_assert(kMaxMats >= 7 && kGf2TcMaxMats >= 7, "matrices per step");
    xg_status st = XG_OK;
    for (int k = 0; k < steps.n; ++k)
        for (uint32_t j = 1; j <= steps.step[k].mats; ++j) {
            uint64_t f = (uint64_t)j * steps.step[k].have;   // the exponent is f 2^q
            int e = q;
            while (f % 2 == 0) {
                f /= 2;
                ++e;
            }
            const void* m;
            if (use_tc[k]) m = tc_mats[k][j - 1] = jump_matrix_tc(streams.device, streams.family, (int)f, e, s, &st);
            else m = mats[k][j - 1] = jump_matrix_multiple(streams.device, streams.family, (int)f, e, s, &st);
            if (!m) return st == XG_ENOMEM ? XG_OK : st;   // no memory: the whole call needs none
        }
    *ran = true;
    if (xg_status w = ws.acquire(s)) return w;
    const uint32_t piece_blocks = (total + 7) / 8;
    const uint32_t list_blocks = (uint32_t)((steps.entries + 255) / 256);
    cut_setup_kernel<<<piece_blocks + list_blocks, 256, 0, s>>>(streams, first, nstreams, pieces, piece_blocks, rings,
                                                                weyl0, steps, lists);
    cudaError_t e = cudaGetLastError();
    for (int k = 0; k < steps.n && e == cudaSuccess; ++k) {
        const uint32_t m = steps.step[k].have * nstreams;
        const int n_mats = (int)steps.step[k].mats;
        const uint32_t* src = lists + steps.step[k].at;
        const uint32_t* dst = src + m;
        if (use_tc[k])
            e = gf2_tc_apply(streams.device, tc_mats[k], n_mats, TcStates{rings, kGf2Words, src, nullptr, 0}, m, rings, kGf2Words,
                             dst, tc, *streams.tc, s, true);
        else
            e = launch_gf2_apply_multi(mats[k], n_mats, rings, rings, m, src, dst, streams.sm_count, s, true,
                                       k + 1 < steps.n);
    }
    if (e != cudaSuccess) {
        ws.release(s);
        return cuda_fail(e, "cut prologue");
    }
    *out = CutRings{rings, weyl0, base + extra_off};
    return XG_OK;
}

xg_status cut_generate(xg_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* out, uint64_t ld,
                       int q, bool* ran)
{
    const bool sum = kind == kNormalSum;
    const uint64_t words = kind == kNormal || sum ? n + (n & 1u) : n;
    const uint32_t pieces = (uint32_t)((words + (uint64_t(1) << q) - 1) >> q);
    const CutStreams streams{c->device, c->sm_count, (int)c->param_set, c->st.win, c->st.pend, c->st.weyl, 1, &c->tc};
    CutRings r{};
    xg_status st = cut_prologue(c->cut, streams, first, nstreams, pieces, q, sum ? (size_t)pieces * nstreams * 4 : 0,
                                c->stream, &r, ran);
    if (st != XG_OK || !*ran) return st;
    CutArgs a{};
    a.st = c->st;
    a.first = first;
    a.nstreams = nstreams;
    a.pieces = pieces;
    a.log2_len = (uint32_t)q;
    a.n = n;
    a.out = sum ? r.extra : out;
    a.ld = ld;
    a.rings = r.rings;
    a.weyl0 = r.weyl0;
    a.omega = c->weyl_on ? 0x9E3779B9u : 0u;
    const bool vec = sum || ((reinterpret_cast<uintptr_t>(out) & 15u) == 0 && (ld % 4 == 0 || nstreams == 1));
    cudaError_t e = launch_cut((int)c->param_set, kind, vec, a, c->stream);
    if (sum && e == cudaSuccess)
        e = launch_dependent(true, dim3((nstreams + 1) / 2), dim3(64), c->stream, cut_sum_kernel,
                             reinterpret_cast<const float*>(r.extra), pieces, nstreams, static_cast<float*>(out));
    st = c->cut.release(c->stream);
    return e == cudaSuccess ? st : cuda_fail(e, "cut generation");
}

}  // namespace xg

// Jump-ahead for xorgens streams.
//
// The recurrence of Sec. 2 is linear over GF(2) on the 4096-bit state (the
// 128-word ring): one step maps a state v to M v.  A stream advanced by J
// words is M^J v, and with the powers C_k = M^(2^k) at hand, M^J v is the
// product of the C_k for the set bits of J.  This lets one long stream be cut
// into pieces that run on different warps (Sec. 2's independent subsequences,
// here exact consecutive pieces of one sequence) and lets xg_jump skip ahead
// without generating.  The Weyl word needs no matrix: w + J omega.
//
// Matrices are kept in column form: column j of C is the state reached from
// the unit state e_j (bit j of ring word j/32).  Applying C to v is the XOR of
// the columns selected by v's bits.  The columns of M itself are one step of
// the recurrence applied to e_j.
//
// Any M^J follows from its columns for the newest ring word alone (32 of the
// 4096, or 64 for 64-bit words).  Let E_b be the state whose newest word is
// bit b and the rest zero.  After i < r steps that word has moved to position
// r - 1 - i, and the only other nonzero word is the one made from it when it
// passed the lag-s tap at step s: (I+L^c)(I+R^d) e_b =: U e_b, by then at
// position r - 1 - (i - s) (it meets no tap itself, since r - 1 - s < s).  So
//   e_(r-1-i, b) = M^i E_b + [i >= s] sum_{b' in U e_b} M^(i-s) E_b',
// and M^J e_(r-1-i, b) = M^i Y_b + [i >= s] sum M^(i-s) Y_b' with Y_b = M^J E_b:
// windows of the sequences that go on from the states Y_b for r more words.
// Products of matrices are therefore applications to 32 (64) states and one
// pass that writes the columns, instead of applications to 4096 states.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "xg_gf2_tc.h"
#include "xg_jump.h"
#include "xg_kernels.cuh"
#include "xg_runtime.h"
#include "xg_w64.h"

namespace xg {

constexpr int kBits = 4096;      // state bits
constexpr int kWords64 = 64;     // uint64 words per state
constexpr int kMaxNewest = 64;   // most columns of one ring word

// The ring and operator pairs of a matrix family.
template <class P>
struct Ring32 {
    using Word = uint32_t;
    static constexpr int R = kR, S = P::S, BITS = 32;
    static __host__ __device__ Word lag_r(Word t) { t ^= t << P::A; return t ^ (t >> P::B); }
    static __host__ __device__ Word lag_s(Word u) { u ^= u << P::C; return u ^ (u >> P::D); }
};
struct Ring64 {
    using Word = uint64_t;
    static constexpr int R = xg64::kR, S = xg64::kS, BITS = 64;
    static __host__ __device__ Word lag_r(Word t) { t ^= t << xg64::kA; return t ^ (t >> xg64::kB); }
    static __host__ __device__ Word lag_s(Word u) { u ^= u << xg64::kC; return u ^ (u >> xg64::kD); }
};

// seq[b][0 .. 2R) = state b's ring and the R raw words after it (no Weyl
// word): one block per state, S words at a time.
template <class F>
__global__ void __launch_bounds__(128) continue_kernel(const typename F::Word* __restrict__ states,
                                                       typename F::Word* __restrict__ seq)
{
    constexpr int R = F::R, S = F::S;
    static_assert(S <= 128 && R <= 128 && R - 1 - S < S, "one word of a step per thread");
    __shared__ typename F::Word x[2 * R];
    const int t = threadIdx.x;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    if (t < R) x[t] = states[(size_t)blockIdx.x * R + t];
    __syncthreads();
    for (int k = R; k < 2 * R; k += S) {
        if (t < S && k + t < 2 * R) x[k + t] = F::lag_r(x[k + t - R]) ^ F::lag_s(x[k + t - S]);
        __syncthreads();
    }
    for (int k = t; k < 2 * R; k += 128) seq[(size_t)blockIdx.x * 2 * R + k] = x[k];
}

// All columns of M^J from the sequences that go on from Y_b = M^J E_b.
template <class F>
__global__ void __launch_bounds__(256) columns_kernel(const typename F::Word* __restrict__ seq,
                                                      typename F::Word* __restrict__ C)
{
    using Word = typename F::Word;
    constexpr int R = F::R, S = F::S;
    const uint32_t id = blockIdx.x * 256 + threadIdx.x;   // grid covers kBits * R exactly
    const int j = (int)(id / R), k = (int)(id % R);
    const int b = j % F::BITS, i = R - 1 - j / F::BITS;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    Word v = seq[(size_t)b * 2 * R + i + k];
    if (i >= S)
        for (Word u = F::lag_s(Word(1) << b); u; u &= u - 1) {
            const int bb = __ffsll((long long)u) - 1;
            v ^= seq[(size_t)bb * 2 * R + (i - S) + k];
        }
    C[id] = v;
}

// Columns of M for parameter set P: column j = one step from e_j.
template <class P>
__global__ void __launch_bounds__(128) step_columns_kernel(uint32_t* __restrict__ cols)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kBits) return;
    const int wj = j >> 5, bj = j & 31;
    uint32_t* out = cols + (size_t)j * kR;
    // the ring shifts by one word: word w of the result is word w+1 of e_j
    for (int w = 0; w < kR - 1; ++w) out[w] = (w + 1 == wj) ? (1u << bj) : 0u;
    // the new word: x_{k-r} is ring word 0, x_{k-s} is ring word r - s
    uint32_t t = (wj == 0) ? (1u << bj) : 0u;
    uint32_t u = (wj == kR - P::S) ? (1u << bj) : 0u;
    t ^= t << P::A;
    t ^= t >> P::B;
    u ^= u << P::C;
    u ^= u >> P::D;
    out[kR - 1] = t ^ u;
}

// dst[i] ^= C src[i] for n (src, dst) pairs, dst zeroed beforehand.  Block
// (x, y, z): matrix z, pairs [NV x, NV x + NV), columns [y*cols, (y+1)*cols);
// 128 threads, thread t owns 32-bit word t of every result.  Columns go four
// at a time: each thread tabulates the 16 XOR combinations of its word of the
// four columns (in shared memory, its own column of the table, so no barrier
// is needed), and a state then costs one lookup and one XOR per four columns.
// Partial results are folded into dst with one atomic XOR per pair.  The
// shared-memory traffic of the lookups and of building the tables bounds the
// kernel, so many states per block (NV = 48) spread each table over more
// lookups: on GB300, 16384 states x 8 applications take 3.3 ms against
// 5.1 ms with 16 (64 gains no more and needs 168 registers a thread).  Few
// states take NV = 16, which pads less, and up to 4 states NV = 4 without
// tables: there the latency of the loads is the cost, so a block asks for its
// first 32 columns, which no earlier kernel writes, before it waits for the
// kernel before it (programmatic dependent launch).
struct MatSet {
    const uint32_t* C[kMaxMats];
    const uint32_t* in[kMaxMats];   // the states that each one is applied to
    uint32_t n[kMaxMats];           // how many of them
    uint32_t at[kMaxMats];          // its destinations in the list
};
// The states and out may be the same array (sources are read, distinct
// destinations are written), so neither is declared __restrict__.
template <int kPairVecs>
__global__ void __launch_bounds__(128) gf2_apply_pairs_kernel(MatSet mats, const uint32_t* __restrict__ src,
                                                              const uint32_t* __restrict__ dst, uint32_t* out, int cols, bool early)
{
    __shared__ uint32_t vbits[kPairVecs * kR];   // this block's words of its states
    __shared__ uint32_t tbl[kPairVecs > 4 ? 16 : 1][kR];
    const uint32_t* __restrict__ C = mats.C[blockIdx.z];
    const uint32_t* rings = mats.in[blockIdx.z];
    const uint32_t n = mats.n[blockIdx.z];
    const int t = threadIdx.x;
    const uint32_t base = blockIdx.x * kPairVecs;
    if (base >= n) return;   // fewer states than the first matrix has
    const int nv = (int)umin((uint32_t)kPairVecs, n - base);
    const int nw = cols / 32, w0 = blockIdx.y * nw;
    uint32_t col[32];   // 32 columns of one input word
    auto load_columns = [&](int w) {
        const uint32_t* colw = C + (size_t)w * 32 * kR + t;
#pragma unroll
        for (int b = 0; b < 32; ++b) col[b] = __ldg(colw + (size_t)b * kR);
    };
    if (early) cudaTriggerProgrammaticLaunchCompletion();
    load_columns(w0);
    cudaGridDependencySynchronize();
    for (int k = t; k < kPairVecs * nw; k += 128) {
        const int v = k / nw;
        vbits[k] = v < nv ? rings[(size_t)(src ? src[base + v] : base + v) * kR + w0 + k % nw] : 0u;
    }
    __syncthreads();
    uint32_t acc[kPairVecs];
#pragma unroll
    for (int v = 0; v < kPairVecs; ++v) acc[v] = 0;
    for (int w = 0;;) {
        uint32_t bw[kPairVecs];
#pragma unroll
        for (int v = 0; v < kPairVecs; ++v) bw[v] = vbits[v * nw + w];
        if constexpr (kPairVecs <= 4) {
#pragma unroll
            for (int b = 0; b < 32; ++b)
#pragma unroll
                for (int v = 0; v < kPairVecs; ++v) acc[v] ^= col[b] & (0u - ((bw[v] >> b) & 1u));
        } else {
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const uint32_t c0 = col[4 * g], c1 = col[4 * g + 1], c2 = col[4 * g + 2], c3 = col[4 * g + 3];
                const uint32_t c01 = c0 ^ c1, c23 = c2 ^ c3;
                tbl[0][t] = 0u;        tbl[1][t] = c0;         tbl[2][t] = c1;         tbl[3][t] = c01;
                tbl[4][t] = c2;        tbl[5][t] = c2 ^ c0;    tbl[6][t] = c2 ^ c1;    tbl[7][t] = c2 ^ c01;
                tbl[8][t] = c3;        tbl[9][t] = c3 ^ c0;    tbl[10][t] = c3 ^ c1;   tbl[11][t] = c3 ^ c01;
                tbl[12][t] = c23;      tbl[13][t] = c23 ^ c0;  tbl[14][t] = c23 ^ c1;  tbl[15][t] = c23 ^ c01;
#pragma unroll
                for (int v = 0; v < kPairVecs; ++v) acc[v] ^= tbl[(bw[v] >> (4 * g)) & 15u][t];
            }
        }
        if (++w == nw) break;
        load_columns(w0 + w);
    }
#pragma unroll
    for (int v = 0; v < kPairVecs; ++v)
        if (v < nv && acc[v]) {
            const uint32_t at = mats.at[blockIdx.z] + base + v, d = dst ? dst[at] : at;
            if (d != kNoState) atomicXor(&out[(size_t)d * kR + t], acc[v]);
        }
}

__global__ void zero_listed_kernel(uint32_t* __restrict__ rings, const uint32_t* __restrict__ idx, uint32_t n)
{
    const uint32_t j = blockIdx.x;
    if (j < n) rings[(size_t)idx[j] * kR + threadIdx.x] = 0u;
}

// Copy each listed stream's current ring (window at its pend offset) into
// rings[k]; also rings' Weyl words advanced by skip[k] words.  With skips,
// an entry with a nonzero skip gets a zero ring instead: its ring is the
// result of a later jump-ahead step, which XORs into it.
__global__ void gather_rings_kernel(State st, const uint32_t* __restrict__ streams, uint32_t n,
                                    uint32_t* __restrict__ rings, const uint64_t* __restrict__ skip,
                                    uint32_t* __restrict__ weyl0, uint32_t weyl0_stride, uint32_t omega)
{
    const uint32_t k = blockIdx.x;
    if (k >= n) return;
    const uint32_t s = streams[k];
    const uint32_t pend = st.pend[s];
    const uint32_t* src = st.win + (size_t)s * kWin + (kRingBase - pend);
    const bool zero = skip && skip[k] != 0;
    for (int w = threadIdx.x; w < kR; w += blockDim.x) rings[(size_t)k * kR + w] = zero ? 0u : src[w];
    if (threadIdx.x == 0 && weyl0)
        weyl0[(size_t)k * weyl0_stride] = st.weyl[s] + (uint32_t)(skip ? skip[k] : 0) * omega;
}

// Write jumped rings back as the streams' state (pend = 0; the ring sits at
// window[kRingBase, kWin)).
__global__ void scatter_rings_kernel(State st, uint32_t first, uint32_t n, const uint32_t* __restrict__ rings,
                                     uint64_t jump, uint32_t omega)
{
    const uint32_t k = blockIdx.x;
    if (k >= n) return;
    const uint32_t s = first + k;
    uint32_t* dst = st.win + (size_t)s * kWin + kRingBase;
    for (int w = threadIdx.x; w < kR; w += blockDim.x) dst[w] = rings[(size_t)k * kR + w];
    if (threadIdx.x == 0) {
        st.weyl[s] += (uint32_t)jump * omega;
        st.pend[s] = 0;
        st.pos[s] += jump;
    }
}

// The same where the windows hold the jumped rings already.
__global__ void finish_jump_kernel(State st, uint32_t first, uint32_t n, uint64_t jump, uint32_t omega)
{
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint32_t s = first + k;
    st.weyl[s] += (uint32_t)jump * omega;
    st.pend[s] = 0;
    st.pos[s] += jump;
}

// Substreams: stream first + m takes rings[m] (its ring after m * 2^q words
// of the seeded sequence), the Weyl word w0 + m 2^q omega and position m 2^q.
__global__ void substream_scatter_kernel(State st, uint32_t first, uint32_t n, const uint32_t* __restrict__ rings,
                                         const uint32_t* __restrict__ w0, int q, uint32_t omega)
{
    const uint32_t m = blockIdx.x;
    if (m >= n) return;
    const uint32_t s = first + m;
    uint32_t* dst = st.win + (size_t)s * kWin + kRingBase;
    for (int w = threadIdx.x; w < kR; w += blockDim.x) dst[w] = rings[(size_t)m * kR + w];
    if (threadIdx.x == 0) {
        const uint64_t off = (uint64_t)m << q;
        st.weyl[s] = *w0 + (uint32_t)off * omega;
        st.pend[s] = 0;
        st.pos[s] = off;
    }
}

// ---------------------------------------------------------------------------

template <int NV>
static cudaError_t launch_pairs(const MatSet& mats, int n_mats, uint32_t* out, uint32_t n, const uint32_t* d_src,
                                const uint32_t* d_dst, int sm_count, cudaStream_t s, bool dependent, bool early)
{
    const uint32_t groups = (n + NV - 1) / NV;
    // enough blocks for about 8 per SM, splitting the 4096 columns if needed
    // (down to one 32-column input word per block: with few states the
    // matrix read is the cost, spread over up to 128 blocks)
    int chunks = 1;
    while (chunks < kBits / 32 && (uint64_t)groups * chunks * n_mats < (uint64_t)8 * sm_count) chunks *= 2;
    return launch_dependent(dependent, dim3(groups, chunks, n_mats), dim3(128), s, gf2_apply_pairs_kernel<NV>, mats,
                            d_src, d_dst, out, kBits / chunks, early);
}

// Matrix j applied to the states in[j] (null lists: state i to state j n + i;
// counts: to the first counts[j]).
static cudaError_t apply_sets(const uint64_t* const* C, int n_mats, const uint32_t* const* in, uint32_t* out, uint32_t n,
                              const uint32_t* d_src, const uint32_t* d_dst, int sm_count, cudaStream_t s, bool dependent,
                              bool early, const uint32_t* counts = nullptr)
{
    if (n == 0 || n_mats == 0) return cudaSuccess;
    if (n_mats > kMaxMats) return cudaErrorInvalidValue;
    MatSet mats{};
    uint32_t at = 0;
    for (int j = 0; j < n_mats; ++j) {
        mats.C[j] = reinterpret_cast<const uint32_t*>(C[j]);
        mats.in[j] = in[j];
        mats.n[j] = counts ? counts[j] : n;
        mats.at[j] = at;
        at += mats.n[j];
    }
    if (n >= 4 * 48) return launch_pairs<48>(mats, n_mats, out, n, d_src, d_dst, sm_count, s, dependent, early);
    if (n > 4) return launch_pairs<16>(mats, n_mats, out, n, d_src, d_dst, sm_count, s, dependent, early);
    return launch_pairs<4>(mats, n_mats, out, n, d_src, d_dst, sm_count, s, dependent, early);
}

cudaError_t launch_gf2_apply_multi(const uint64_t* const* C, int n_mats, const uint32_t* in, uint32_t* out, uint32_t n,
                                   const uint32_t* d_src, const uint32_t* d_dst, int sm_count, cudaStream_t s,
                                   bool dependent, bool early, const uint32_t* counts)
{
    const uint32_t* all[kMaxMats];
    for (const uint32_t*& p : all) p = in;
    return apply_sets(C, n_mats, all, out, n, d_src, d_dst, sm_count, s, dependent, early, counts);
}

// C = M^J from the newest word's columns Y_b = M^J E_b (states, consecutive
// rings); seq: 2 * kBits * kMaxNewest / 8 bytes of scratch.
constexpr size_t kSeqBytes = (size_t)2 * kBits / 8 * kMaxNewest;

template <class F>
static cudaError_t build_columns(const uint32_t* states, uint8_t* seq, uint64_t* C, cudaStream_t s, bool dependent)
{
    using Word = typename F::Word;
    Word* sq = reinterpret_cast<Word*>(seq);
    cudaError_t e = launch_dependent(dependent, dim3(F::BITS), dim3(128), s, continue_kernel<F>,
                                     reinterpret_cast<const Word*>(states), sq);
    if (e == cudaSuccess)
        e = launch_dependent(true, dim3(kBits * F::R / 256), dim3(256), s, columns_kernel<F>,
                             static_cast<const Word*>(sq), reinterpret_cast<Word*>(C));
    return e;
}

// dependent: as in launch_gf2_apply_pairs.
static cudaError_t launch_build_columns(int family, const uint32_t* states, uint8_t* seq, uint64_t* C, cudaStream_t s,
                                        bool dependent = false)
{
    if (family == kJumpSetW64) return build_columns<Ring64>(states, seq, C, s, dependent);
    if (family == 1) return build_columns<Ring32<ParamsPaper>>(states, seq, C, s, dependent);
    return build_columns<Ring32<ParamsDefault>>(states, seq, C, s, dependent);
}

// Columns of the newest ring word: the last ones of a matrix in column form.
static int newest_columns(int family) { return family == kJumpSetW64 ? 64 : 32; }
static const uint32_t* newest_of(const uint64_t* C, int family)
{
    return reinterpret_cast<const uint32_t*>(C) + (size_t)(kBits - newest_columns(family)) * kR;
}

namespace {
struct Tables {
    uint64_t* mat[kMaxPow] = {};  // C_k: 4096 columns x 64 uint64 (2 MiB), allocated when built
    int built = 0;                // C_0 .. C_{built-1} are valid
    uint64_t* odd[3][kMaxPow] = {};  // M^(j 2^k) for j = 3, 5, 7
    uint8_t* scratch = nullptr;   // squaring: kMaxNewest states, sequences, identity list
};
std::mutex g_tab_mu;
Tables g_tabs[64][3];  // per device, per matrix family

// Device memory of the odd multiples and the FP4 copies.  64 exponents of three
// families would take 7 GiB; a server of the default size needs 0.6 GiB of one
// family, so the limit leaves each of them as many exponents as calls of up to
// 2^37 words have.
std::atomic<size_t> g_derived[64];

size_t derived_limit()
{
    const char* v = std::getenv("XG_JUMP_TABLE_MIB");
    return v ? (size_t)std::strtoull(v, nullptr, 10) << 20 : size_t(3) << 30;
}

cudaError_t derived_alloc(int device, void** p, size_t bytes)
{
    cudaError_t e = cudaErrorMemoryAllocation;
    if (g_derived[device].fetch_add(bytes) + bytes <= derived_limit()) e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) g_derived[device].fetch_sub(bytes);
    return e;
}

void derived_free(int device, void* p, size_t bytes)
{
    cudaFree(p);
    g_derived[device].fetch_sub(bytes);
}
}  // namespace

// out = A B (powers of one matrix): A applied to B's newest columns.
static cudaError_t multiply_matrices(int device, int family, Tables& T, const uint64_t* A, const uint64_t* B,
                                     uint64_t* out, cudaStream_t s)
{
    const int nb = newest_columns(family);
    uint32_t* states = reinterpret_cast<uint32_t*>(T.scratch);
    uint8_t* seq = T.scratch + (size_t)kMaxNewest * kR * 4;
    uint32_t* ids = reinterpret_cast<uint32_t*>(seq + kSeqBytes);
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = launch_jump_index(ids, (uint32_t)nb, 0u, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(states, 0, (size_t)nb * kR * 4, s);
    if (e == cudaSuccess)
        e = launch_gf2_apply_pairs(A, newest_of(B, family), states, (uint32_t)nb, ids, ids, sms, s);
    if (e == cudaSuccess) e = launch_build_columns(family, states, seq, out, s);
    return e;
}

const uint64_t* jump_matrix(int device, int param_set, int k, cudaStream_t s, xg_status* st)
{
    *st = XG_OK;
    if (device < 0 || device >= 64 || k < 0 || k >= kMaxPow || param_set < 0 || param_set > kJumpSetW64) {
        *st = fail(XG_EINVAL, "jump power %d out of range", k);
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(g_tab_mu);
    Tables& T = g_tabs[device][param_set];
    const size_t mat_bytes = (size_t)kBits * kWords64 * 8;
    bool built_now = false;
    while (T.built <= k) {
        const int b = T.built;
        cudaError_t e = cudaMalloc(&T.mat[b], mat_bytes);
        if (e == cudaSuccess && !T.scratch) {
            void* p = nullptr;
            e = cudaMalloc(&p, (size_t)kMaxNewest * kR * 4 + kSeqBytes + (size_t)3 * kMaxNewest * 4);
            if (e == cudaSuccess) T.scratch = static_cast<uint8_t*>(p);
            else cudaFree(T.mat[b]);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            T.mat[b] = nullptr;
            *st = fail(XG_ENOMEM, "jump tables: cudaMalloc(2 MiB) failed for power %d", b);
            return nullptr;
        }
        if (b == 0) {
            if (param_set == kJumpSetW64)
                e = xg64::launch_step_columns(T.mat[0], s);
            else if (param_set == 1)
                step_columns_kernel<ParamsPaper><<<kBits / 128, 128, 0, s>>>(reinterpret_cast<uint32_t*>(T.mat[0]));
            else
                step_columns_kernel<ParamsDefault><<<kBits / 128, 128, 0, s>>>(reinterpret_cast<uint32_t*>(T.mat[0]));
        } else {
            e = multiply_matrices(device, param_set, T, T.mat[b - 1], T.mat[b - 1], T.mat[b], s);
        }
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) {
            *st = cuda_fail(e, "jump table build");
            return nullptr;
        }
        T.built = b + 1;
        built_now = true;
    }
    // other CUDA streams may use the tables next: make the build complete
    if (built_now && cudaStreamSynchronize(s) != cudaSuccess) {
        *st = cuda_fail(cudaGetLastError(), "jump table build");
        return nullptr;
    }
    return T.mat[k];
}

const uint64_t* jump_matrix_multiple(int device, int param_set, int j, int k, cudaStream_t s, xg_status* st)
{
    while (j > 1 && j % 2 == 0) {
        j /= 2;
        ++k;
    }
    if (j == 1) return jump_matrix(device, param_set, k, s, st);
    // j = 3, 5, 7: M^(2^k) times M^((j - 1) 2^k), itself an even multiple
    const uint64_t* a = jump_matrix(device, param_set, k, s, st);
    const uint64_t* b = a ? jump_matrix_multiple(device, param_set, j - 1, k, s, st) : nullptr;
    if (!b) return nullptr;
    std::lock_guard<std::mutex> lk(g_tab_mu);
    Tables& T = g_tabs[device][param_set];
    uint64_t*& C = T.odd[(j - 3) / 2][k];
    if (C) return C;
    void* p = nullptr;
    const size_t bytes = (size_t)kBits * kWords64 * 8;
    cudaError_t e = derived_alloc(device, &p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *st = fail(XG_ENOMEM, "jump tables: no 2 MiB for %d times power %d", j, k);
        return nullptr;
    }
    e = multiply_matrices(device, param_set, T, a, b, static_cast<uint64_t*>(p), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // other CUDA streams may use it next
    if (e != cudaSuccess) {
        derived_free(device, p, bytes);
        *st = cuda_fail(e, "jump table build");
        return nullptr;
    }
    return C = static_cast<uint64_t*>(p);
}

namespace {
// FP4 copies of the powers for the tensor-core path: 8 MiB each, built on
// first use and kept until exit.
std::mutex g_tc_mu;
uint8_t* g_tc_mats[64][3][4][kMaxPow] = {};   // [.. j = 1, 3, 5, 7][k]
}  // namespace

const uint8_t* jump_matrix_tc(int device, int family, int j, int k, cudaStream_t s, xg_status* st)
{
    while (j > 1 && j % 2 == 0) {
        j /= 2;
        ++k;
    }
    const uint64_t* C = jump_matrix_multiple(device, family, j, k, s, st);
    if (!C) return nullptr;
    std::lock_guard<std::mutex> lk(g_tc_mu);
    uint8_t*& A = g_tc_mats[device][family][j / 2][k];
    if (A) return A;
    void* p = nullptr;
    cudaError_t e = derived_alloc(device, &p, kGf2TcMatrixBytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *st = fail(XG_ENOMEM, "jump tables: no 8 MiB for the FP4 copy of %d times power %d", j, k);
        return nullptr;
    }
    e = gf2_tc_expand_matrix(C, static_cast<uint8_t*>(p), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // other CUDA streams may use it next
    if (e != cudaSuccess) {
        derived_free(device, p, kGf2TcMatrixBytes);
        *st = cuda_fail(e, "jump tables: FP4 expansion");
        return nullptr;
    }
    A = static_cast<uint8_t*>(p);
    return A;
}

bool gf2_use_tc(int device, uint32_t n, uint32_t from)
{
    // read on every call (a few hundred nanoseconds against a matrix application)
    const char* off = std::getenv("XG_JUMP_TENSOR_CORES");
    if (off && std::strcmp(off, "0") == 0) return false;
    const char* v = std::getenv("XG_GF2_TC_MIN_STATES");
    const uint32_t min_states = v ? (uint32_t)std::strtoul(v, nullptr, 10) : from;
    return n >= std::max(1u, min_states) && gf2_tc_available(device);
}

size_t gf2_apply_scratch(int device, uint32_t n)
{
    return gf2_use_tc(device, n) ? gf2_tc_scratch_bytes(n) : 0;
}

cudaError_t gf2_apply(int device, int family, int k, uint32_t* rings, uint32_t n, const uint32_t* d_src,
                      const uint32_t* d_dst, uint8_t* scratch, TcStatus& tc, int sm_count, cudaStream_t s, xg_status* st,
                      bool dst_zeroed)
{
    *st = XG_OK;
    if (n == 0) return cudaSuccess;
    if (scratch && gf2_use_tc(device, n) && tc.device()) {
        const uint8_t* A = jump_matrix_tc(device, family, 1, k, s, st);
        if (!A && *st != XG_ENOMEM) return cudaErrorUnknown;   // with *st
        if (A) return gf2_tc_apply(device, &A, 1, TcStates{rings, kGf2Words, d_src, nullptr, 0}, n, rings, kGf2Words, d_dst, scratch,
                            tc, s);
    }
    const uint64_t* C = jump_matrix(device, family, k, s, st);   // *st is XG_OK again
    if (!C) return cudaErrorMemoryAllocation;
    cudaError_t e = dst_zeroed ? cudaSuccess : zero_rings(rings, d_dst, n, s);
    if (e == cudaSuccess) e = launch_gf2_apply_pairs(C, rings, rings, n, d_src, d_dst, sm_count, s);
    return e;
}

// With several set bits the powers are multiplied first: one chain of
// applications to 32 (64) states, or two at half the length, instead of one to
// all states.  From 2 bits on for more than kMaxNewest states; fewer states
// cost hardly more than the columns do, so there the product has to save
// launches: us per jump power by power / by the product, 16 streams 4 bits 60 /
// 54, 8 bits 101 / 67, 1 stream 4 bits 44 / 50, 8 bits 68 / 60.
static bool jump_combines(uint64_t words, uint32_t n)
{
    const int bits = __builtin_popcountll(words);
    return bits >= (n > (uint32_t)kMaxNewest ? 2 : n > 4 ? 4 : 7);
}

// Work area of a product: one group of newest columns per set bit, the
// sequences, the product and one factor in column form.
static size_t product_bytes(uint64_t words)
{
    return (size_t)__builtin_popcountll(words) * kMaxNewest * kR * 4 + kSeqBytes + (size_t)2 * kBits * kR * 4;
}

// The tensor cores beside the table kernel in jumps by one power: us per jump
// of 8 / 64 / 160 / 256 streams 23.4 / 23.4 / 24.2 / 24.4 in place against 27.8
// / 30.4 / 33.8 / 42.9 (gather, table kernel, scatter); by a product of 8 powers
// 61 / 62 / 62 / 63 against 65 / 66 / 70 / 80.
constexpr uint32_t kInPlaceStreams = 8;

size_t gf2_jump_work_bytes(int device, uint32_t n, uint64_t words, bool in_place)
{
    const size_t product = jump_combines(words, n) ? product_bytes(words) : 0;
    if (!in_place) return product ? product : gf2_apply_scratch(device, n);
    // the tensor-core operand, then the product's work area and its FP4 copy
    return (gf2_tc_scratch_bytes(n) + 255) / 256 * 256 + (product ? product + kGf2TcMatrixBytes : 0);
}

// The product of the powers in `words` in column form (in w, product_bytes):
// its newest columns by one application per further set bit to 32 (64) states,
// then all columns from them.  For 16384 streams and 8 set bits this took the
// jump from 0.615 ms (seven tensor-core products of 4096 columns each) to
// 0.311 ms.  The applications are one dependent chain, 3 us each (the launch
// that waits for the one before it, the states, 8 rounds of tables), so from
// kTwoChains bits on the powers form two chains that share their launches; one
// of them then gets all its columns (5 us) and is applied to the other.  300
// streams, 8 / 16 / 30 bits: 78 / 113 / 180 -> 66 / 91 / 144 us.
// Last launch: a dependent one may follow.
constexpr int kTwoChains = 6;

static cudaError_t power_product(int device, int family, uint64_t words, uint8_t* w, int sm_count, cudaStream_t s,
                                 const uint64_t** product, xg_status* st)
{
    const uint32_t nb = (uint32_t)newest_columns(family);
    const size_t group = (size_t)nb * kR;   // 32-bit words of one group of columns
    uint32_t* cols = reinterpret_cast<uint32_t*>(w);
    const int bits = __builtin_popcountll(words);
    uint8_t* seq = w + (size_t)bits * kMaxNewest * kR * 4;
    uint64_t* prod = reinterpret_cast<uint64_t*>(seq + kSeqBytes);
    uint64_t* factor = prod + (size_t)kBits * kWords64;
    const uint64_t* C[64];
    int n = 0;
    for (int k = 0; k < 64; ++k) {
        if (!((words >> k) & 1)) continue;
        C[n] = jump_matrix(device, family, k, s, st);
        if (!C[n++]) return cudaErrorMemoryAllocation;
    }
    cudaError_t e = cudaMemsetAsync(cols, 0, (size_t)(bits - 1) * group * 4, s);
    // chain c starts with the newest columns of its first power
    const int chains = bits >= kTwoChains ? 2 : 1;
    const int len[2] = {(bits + chains - 1) / chains, chains == 2 ? bits / 2 : 0};
    const uint64_t* const* power[2] = {C, C + len[0]};
    const uint32_t* have[2] = {newest_of(C[0], family), chains == 2 ? newest_of(C[len[0]], family) : nullptr};
    uint32_t* to = cols;
    bool dependent = false;   // the launch before is one of this chain's
    for (int i = 1; i < len[0] && e == cudaSuccess; ++i) {
        const int now = i < len[1] ? 2 : 1;
        const uint64_t* m[2] = {power[0][i], now == 2 ? power[1][i] : nullptr};
        e = apply_sets(m, now, have, to, nb, nullptr, nullptr, sm_count, s, dependent, true);
        dependent = true;
        for (int c = 0; c < now; ++c, to += group) have[c] = to;
    }
    if (chains == 2) {
        if (e == cudaSuccess) e = launch_build_columns(family, have[1], seq, factor, s, dependent);
        // an ordinary launch: a dependent one would read the factor's first
        // columns before the kernel that writes them has ended
        const uint64_t* f = factor;
        if (e == cudaSuccess) e = apply_sets(&f, 1, have, to, nb, nullptr, nullptr, sm_count, s, false, true);
        dependent = true;
        have[0] = to;
    }
    if (e == cudaSuccess) e = launch_build_columns(family, have[0], seq, prod, s, dependent);
    *product = prod;
    return e;
}

bool gf2_jump_in_place(int device, int family, uint32_t n, uint64_t words, TcStatus& tc, cudaStream_t s)
{
    if (!gf2_use_tc(device, n, kInPlaceStreams) || !tc.device()) return false;
    xg_status st = XG_OK;
    if (__builtin_popcountll(words) == 1) return jump_matrix_tc(device, family, 1, __builtin_ctzll(words), s, &st) != nullptr;
    return jump_combines(words, n);
}

cudaError_t gf2_jump_windows(int device, int family, uint64_t words, const JumpWindows& win, uint32_t n, uint8_t* work,
                             TcStatus& tc, int sm_count, cudaStream_t s, xg_status* st)
{
    *st = XG_OK;
    const uint8_t* A = nullptr;
    if (__builtin_popcountll(words) == 1) {
        A = jump_matrix_tc(device, family, 1, __builtin_ctzll(words), s, st);
        if (!A) return cudaErrorMemoryAllocation;
    } else {
        uint8_t* w = work + (gf2_tc_scratch_bytes(n) + 255) / 256 * 256;
        uint8_t* abuf = w + product_bytes(words);
        const uint64_t* P = nullptr;
        cudaError_t e = power_product(device, family, words, w, sm_count, s, &P, st);
        if (e == cudaSuccess) e = gf2_tc_expand_matrix(P, abuf, s, true);
        if (e != cudaSuccess) return e;
        A = abuf;
    }
    // the windows were last written before the product's first launch
    uint32_t* ring = win.win + kRingBase;
    return gf2_tc_apply(device, &A, 1, TcStates{ring, kWin, nullptr, win.pend, win.word, true}, n, ring, kWin, nullptr,
                        work, tc, s, __builtin_popcountll(words) > 1);
}

cudaError_t gf2_jump_states(int device, int family, uint64_t words, uint32_t* rings, uint32_t n,
                            const uint32_t* d_idx, uint8_t* work, TcStatus& tc, int sm_count, cudaStream_t s, xg_status* st,
                            bool* result_hi)
{
    *st = XG_OK;
    *result_hi = false;
    const uint32_t* lo = d_idx;       // 0 .. n-1
    const uint32_t* hi = d_idx + n;   // n .. 2n-1
    if (!jump_combines(words, n)) {
        uint8_t* scratch = gf2_apply_scratch(device, n) ? work : nullptr;
        bool in_lo = true;
        for (int k = 0; k < 64; ++k) {
            if (!((words >> k) & 1)) continue;
            cudaError_t e = gf2_apply(device, family, k, rings, n, in_lo ? lo : hi, in_lo ? hi : lo, scratch, tc, sm_count, s,
                                      st);
            if (e != cudaSuccess) return e;
            in_lo = !in_lo;
        }
        *result_hi = !in_lo;
        return cudaSuccess;
    }
    const uint64_t* P = nullptr;
    cudaError_t e = power_product(device, family, words, work, sm_count, s, &P, st);
    if (e == cudaSuccess) e = zero_rings(rings, hi, n, s);
    if (e == cudaSuccess) e = launch_gf2_apply_pairs(P, rings, rings, n, lo, hi, sm_count, s);
    *result_hi = true;
    return e;
}

// ids[i] = first + i for i < n, then ids[n + j] = j for j < 2n.
__global__ void jump_index_kernel(uint32_t* __restrict__ ids, uint32_t n, uint32_t first)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ids[i] = first + (uint32_t)i;
    else if (i < (uint64_t)3 * n) ids[i] = (uint32_t)(i - n);
}

cudaError_t launch_jump_index(uint32_t* ids, uint32_t n, uint32_t first, cudaStream_t s)
{
    const uint64_t total = (uint64_t)3 * n;
    jump_index_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(ids, n, first);
    return cudaGetLastError();
}

cudaError_t launch_gf2_apply_pairs(const uint64_t* C, const uint32_t* in, uint32_t* out, uint32_t n,
                                   const uint32_t* d_src, const uint32_t* d_dst, int sm_count, cudaStream_t s,
                                   bool dependent)
{
    return launch_gf2_apply_multi(&C, 1, in, out, n, d_src, d_dst, sm_count, s, dependent);
}

cudaError_t zero_rings(uint32_t* rings, const uint32_t* d_idx, uint32_t n, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    zero_listed_kernel<<<n, kR, 0, s>>>(rings, d_idx, n);
    return cudaGetLastError();
}

cudaError_t launch_gather_rings(const State& st, const uint32_t* d_streams, uint32_t n, uint32_t* d_rings,
                                const uint64_t* d_skip, uint32_t* d_weyl0, uint32_t weyl0_stride, uint32_t omega,
                                cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    gather_rings_kernel<<<n, 128, 0, s>>>(st, d_streams, n, d_rings, d_skip, d_weyl0, weyl0_stride, omega);
    return cudaGetLastError();
}

}  // namespace xg

extern "C" xg_status xg_jump(xg_ctx* ctx, uint32_t first, uint32_t nstreams, uint64_t words)
{
    using namespace xg;
    if (!ctx) return fail(XG_EINVAL, "null context");
    if ((uint64_t)first + nstreams > ctx->n) return fail(XG_EINVAL, "streams out of range");
    if (ctx->server) return fail(XG_EINVAL, "the request server owns this context; stop it first");
    if (nstreams == 0 || words == 0) return XG_OK;
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (xg_status f = ctx->earlier_failure()) return f;
    cudaStream_t s = ctx->stream;
    int top = 63;
    while (!((words >> top) & 1)) --top;
    xg_status st = XG_OK;
    for (int k = 0; k <= top; ++k)
        if (((words >> k) & 1) && !jump_matrix(ctx->device, (int)ctx->param_set, k, s, &st)) return st;
    const uint32_t omega = ctx->weyl_on ? 0x9E3779B9u : 0u;
    const bool in_place = gf2_jump_in_place(ctx->device, (int)ctx->param_set, nstreams, words, ctx->tc, s) &&
                          ctx->ensure_jump_ws(gf2_jump_work_bytes(ctx->device, nstreams, words, true)) == XG_OK;
    cudaError_t e;
    if (in_place) {
        e = gf2_jump_windows(ctx->device, (int)ctx->param_set, words,
                             JumpWindows{ctx->st.win + (size_t)first * kWin, ctx->st.pend + first, 1}, nstreams,
                             static_cast<uint8_t*>(ctx->jump_ws), ctx->tc, ctx->sm_count, s, &st);
        if (e == cudaSuccess) {
            finish_jump_kernel<<<(nstreams + 255) / 256, 256, 0, s>>>(ctx->st, first, nstreams, words, omega);
            e = cudaGetLastError();
        }
    } else {
        // workspace kept in the context (grow-only): rings[0, n) hold the
        // states, rings[n, 2n) receive the results; index lists (stream ids for
        // the gather, then 0 .. 2n-1); the jump's own work area
        const size_t rings_bytes = (size_t)2 * nstreams * kR * 4;
        const size_t ids_off = rings_bytes;
        const size_t work_off = (ids_off + (size_t)3 * nstreams * 4 + 255) / 256 * 256;
        const size_t wbytes = gf2_jump_work_bytes(ctx->device, nstreams, words, false);
        if (xg_status g = ctx->ensure_jump_ws(work_off + wbytes)) return g;
        char* ws = static_cast<char*>(ctx->jump_ws);
        uint32_t* rings = reinterpret_cast<uint32_t*>(ws);
        uint32_t* ids = reinterpret_cast<uint32_t*>(ws + ids_off);
        const uint32_t* lo_idx = ids + nstreams;  // 0 .. 2n-1
        e = launch_jump_index(ids, nstreams, first, s);
        if (e == cudaSuccess) e = launch_gather_rings(ctx->st, ids, nstreams, rings, nullptr, nullptr, 0, 0, s);
        bool hi = false;
        if (e == cudaSuccess)
            e = gf2_jump_states(ctx->device, (int)ctx->param_set, words, rings, nstreams, lo_idx,
                                reinterpret_cast<uint8_t*>(ws + work_off), ctx->tc, ctx->sm_count, s, &st, &hi);
        if (e == cudaSuccess) {
            const uint32_t* res = hi ? rings + (size_t)nstreams * kR : rings;
            scatter_rings_kernel<<<nstreams, 128, 0, s>>>(ctx->st, first, nstreams, res, words, omega);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (st != XG_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "xg_jump");
    return ctx->earlier_failure();
}

extern "C" xg_status xg_seed_substreams(xg_ctx* ctx, uint32_t first, uint32_t count, uint32_t seed,
                                        uint32_t log2_spacing)
{
    using namespace xg;
    if (!ctx) return fail(XG_EINVAL, "null context");
    if ((uint64_t)first + count > ctx->n) return fail(XG_EINVAL, "streams out of range");
    if (count == 0) return XG_OK;
    if (ctx->server) return fail(XG_EINVAL, "the request server owns this context; stop it first");
    // the last stream starts at (count - 1) * 2^q, which must fit in 64 bits
    int steps = 0;   // doubling steps: bits of count - 1
    while (steps < 32 && ((uint64_t)(count - 1) >> steps)) ++steps;
    if (log2_spacing > 63 || (count > 1 && (int)log2_spacing + steps > 64))
        return fail(XG_EINVAL, "(count - 1) * 2^%u does not fit in 64 bits", log2_spacing);
    if (xg_status s = xg_seed(ctx, first, 1, &seed)) return s;
    std::lock_guard<std::mutex> lk(ctx->mu);
    cudaStream_t s = ctx->stream;
    const int q = (int)log2_spacing;
    xg_status st = XG_OK;
    for (int b = 0; b < steps; ++b)
        if (!jump_matrix(ctx->device, (int)ctx->param_set, q + b, s, &st)) return st;
    // step b takes the states m - 2^b to the states m, m in [2^b, min(2^(b+1), count)):
    // its sources are the identity list from 0 and its destinations the same
    // list from 2^b, so one device-built list 0 .. 2 count - 1 serves every step
    uint32_t most = 0;
    for (int b = 0; b < steps; ++b) {
        const uint32_t lo = 1u << b, hi = (uint32_t)std::min<uint64_t>((uint64_t)lo << 1, count);
        most = std::max(most, hi - lo);
    }
    // workspace kept in the context (grow-only): rings of all count states;
    // the index lists (first + i, then 0 .. 2 count - 1); the gathered Weyl
    // word; the tensor-core operand (when used)
    const size_t rings_bytes = (size_t)count * kR * 4;
    const size_t ids_off = rings_bytes;
    const size_t w0_off = ids_off + (size_t)3 * count * 4;
    const size_t scratch_off = (w0_off + 4 + 255) / 256 * 256;
    const size_t sbytes = gf2_apply_scratch(ctx->device, most);
    if (xg_status g = ctx->ensure_jump_ws(scratch_off + sbytes)) return g;
    char* ws = static_cast<char*>(ctx->jump_ws);
    uint32_t* rings = reinterpret_cast<uint32_t*>(ws);
    uint32_t* ids = reinterpret_cast<uint32_t*>(ws + ids_off);
    const uint32_t* iota = ids + count;
    uint32_t* d_w0 = reinterpret_cast<uint32_t*>(ws + w0_off);
    uint8_t* scratch = sbytes ? reinterpret_cast<uint8_t*>(ws + scratch_off) : nullptr;
    cudaError_t e = launch_jump_index(ids, count, first, s);
    if (e == cudaSuccess) e = launch_gather_rings(ctx->st, ids, 1, rings, nullptr, d_w0, 1, 0u, s);
    // the destinations 1 .. count - 1, zeroed once for all the steps
    if (e == cudaSuccess && count > 1) e = cudaMemsetAsync(rings + kR, 0, (size_t)(count - 1) * kR * 4, s);
    for (int b = 0; b < steps && e == cudaSuccess; ++b) {
        const uint32_t lo = 1u << b, hi = (uint32_t)std::min<uint64_t>((uint64_t)lo << 1, count);
        e = gf2_apply(ctx->device, (int)ctx->param_set, q + b, rings, hi - lo, iota, iota + lo, scratch, ctx->tc,
                      ctx->sm_count, s, &st, true);
    }
    if (e == cudaSuccess) {
        substream_scatter_kernel<<<count, 128, 0, s>>>(ctx->st, first, count, rings, d_w0, q,
                                                       ctx->weyl_on ? 0x9E3779B9u : 0u);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (st != XG_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "xg_seed_substreams");
    return ctx->earlier_failure();
}

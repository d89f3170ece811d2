// GF(2) matrix applications on the tensor cores (tcgen05, sm_103a).
//
// The recurrence of Sec. 2 is linear over GF(2) on the 4096-bit state, so a
// jump-ahead applies a 4096 x 4096 bit matrix C to many states: y = C x.
// Over the integers, with 0/1 entries, (C x)_i counts the set bits of row i
// of C that meet set bits of x; the GF(2) result is that count's parity.  The
// counts are at most 4096, which an FP32 accumulator holds exactly, and 0/1
// are exact in FP4 E2M1, so the product of the matrix and a batch of states
// is a block-scaled FP4 GEMM whose scales are all 1 (mxf4: UE8M0 127):
//   D[i][s] = sum_k A[i][k] B[s][k],  A[i][k] = C[i][k],  B[s][k] = bit k of x_s
// (M = 4096 output bits, N = states, K = 4096 input bits, both operands
// K-major), followed by a parity epilogue that packs bits back into 32-bit
// ring words.  FP4 halves the bytes per operand of the same kernel in FP8
// (kind::f8f6f4): one application to 16384 states 150 -> 86 us.  Bound by
// shared memory: 47 KB per 128 x 240 x 256 block are written and read once,
// about 130 B per clock and SM; the tensor pipe is 66% active.
//
// Order of K: both operands hold the 32 bits of an input word as 32 nibbles
// in the order that three shifts and masks give (spread32); a dot product
// does not depend on it.
//
// Kernel: persistent, one CTA per SM, output tiles of 128 bits by bn states, bn
// up to 240 (gf2_tc_tile; two FP32 accumulators of 240 columns and 32 columns
// of scales fill the 512 TMEM columns).  Warp 0 (one lane) streams 128-byte-wide K blocks (256 bits) of A
// and B into a 4-stage shared-memory ring with TMA (128B swizzle, mbarrier
// transaction counts); warp 1 (one lane) issues tcgen05.mma (kind::mxf4,
// E2M1 x E2M1 -> F32, 128 x bn x 64 each) into one of two TMEM accumulators
// and frees each stage with tcgen05.commit; four epilogue warps read the
// other accumulator with tcgen05.ld (32 TMEM lanes = 32 output bits each),
// take each count's parity and pack the 32 lanes' bits with a warp ballot:
// one ballot is one ring word of one state.  The scales are written once: every byte of their
// columns is 127, so no layout of them matters.  The set-up runs beside the end
// of the kernel before it; the launch after it starts when it ends: kernels that
// were resident earlier would crowd onto the SMs that have no tile.
//
// Every wait is bounded (2 s of %globaltimer); a wait that gives up records
// a failure in its owner's status word (TcStatus), the CTA waits (bounded) for its
// own TMA copies still in flight, frees its TMEM and returns.  To test that
// path, XG_TC_TEST_STALL=1 in the environment makes CTA 0 arm its first
// stage's barrier without starting the stage's copies: the waits on that
// stage run out (no fault, no unbounded wait) and the call reports it.
#include <cuda.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <mutex>
#include <utility>
#include <vector>

#include "xg_gf2_tc.h"
#include "xg_runtime.h"

namespace xg {
namespace {

constexpr int kBM = 128;                  // output bits per tile (TMEM lanes)
constexpr int kBN = 240;                  // most states per tile (TMEM columns)
constexpr int kRowBytes = kGf2Bits / 2;   // 4096 nibbles
constexpr int kBK = 128;                  // bytes of K per stage: one 128-byte swizzle row
constexpr int kKBlocks = kRowBytes / kBK; // 16
constexpr int kTmemCols = 512;
constexpr int kScaleA = 2 * kBN, kScaleB = 2 * kBN + 16;   // TMEM columns of the scales
static_assert(kScaleB + 16 <= kTmemCols, "TMEM columns");
constexpr int kStages = 4;
constexpr int kABytes = kBM * kBK;        // 16 KiB
constexpr int kBBytes = kBN * kBK;        // 30 KiB
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kSmemBytes = kStages * kStageBytes + 1024 /* barriers */ + 1024 /* alignment */;
constexpr int kEpilogueWarps = 4;
constexpr int kThreads = 32 * (2 + kEpilogueWarps);
constexpr uint64_t kWaitLimitNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// Wait for the phase with the given parity to complete; false if it has not
// after the deadline.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t deadline)
{
    const uint32_t a = smem_addr(bar);
    for (uint32_t it = 0;; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 255u) == 255u && global_ns() > deadline) return false;
    }
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::
            "r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_addr(bar)), "r"(x), "r"(y)
        : "memory");
}

// Shared-memory matrix descriptor (tcgen05): K-major, 128B swizzle, rows of
// 128 bytes, 8-row groups 1024 bytes apart, version 1.
__device__ __forceinline__ uint64_t smem_desc(const void* p)
{
    const uint64_t addr = smem_addr(p);
    return ((addr & 0x3FFFFull) >> 4)        // start address, bits 0-13
           | (1ull << 16)                    // leading byte offset (unused for swizzled K-major)
           | ((1024ull >> 4) << 32)          // stride byte offset: 8 rows x 128 B
           | (1ull << 46)                    // descriptor version
           | (2ull << 61);                   // layout: 128-byte swizzle
}

// Instruction descriptor, kind::mxf4: A and B E2M1, both K-major, UE8M0
// scales (data id 0), K = 64, N = bn (a multiple of 16), M = kBM.
__device__ __forceinline__ uint32_t instr_desc(uint32_t bn)
{
    return (1u << 7) | (1u << 10)   // A, B: E2M1
           | (1u << 23)             // scale type UE8M0
           | ((bn >> 3) << 17) | ((uint32_t)(kBM >> 7) << 27);
}

__device__ __forceinline__ void mma_f4(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t sa_tmem, uint32_t sb_tmem, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sa_tmem), "r"(sb_tmem)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive columns of this warp's 32 TMEM lanes: v[j] = column col + j.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The same word to 16 consecutive columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_fill16(uint32_t taddr, uint32_t x)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr),
        "r"(x)
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ bool failed(const volatile int* flag) { return *flag != 0; }

struct TcMaps {
    CUtensorMap a[kGf2TcMaxMats];
    CUtensorMap b;
    uint32_t n[kGf2TcMaxMats];    // matrix j applies to the first n[j] states
    uint32_t at[kGf2TcMaxMats];   // its destinations in the list
    uint32_t end[kGf2TcMaxMats];  // tiles of the matrices up to j
};

// Matrix and state tile of tile t.
struct TcTile {
    uint32_t j, nt;
};
__device__ __forceinline__ TcTile tc_tile(const TcMaps& maps, uint32_t t)
{
    uint32_t j = 0, from = 0;
    while (t >= maps.end[j]) from = maps.end[j++];
    return TcTile{j, (t - from) / (uint32_t)(kGf2Bits / kBM)};
}

// out[dst[at_j + s]] = C_j x_s for the first n_j states of the B operand (rows
// past them count for nothing).  Persistent: CTA b takes tiles b, b +
// gridDim.x, ... of the matrices' (4096 / kBM) x (n_j / bn) tiles, M fastest
// (consecutive tiles share a B tile in L2).  bn states per tile: 240 for many
// states; fewer states take the width that gives the shortest waves (see
// gf2_tc_tile), whose smaller B tiles are loaded and multiplied faster.  A few hundred states fill a part
// of the SMs with one matrix, and a launch costs as much as its first tile
// (14 us, each further wave 4), so several matrices share one: 500 states by 7
// matrices 35 us, in three doubling launches 75 us.  192 threads: warp 0 = TMA producer, warp 1 = TMEM owner and
// MMA issuer, warps 2-5 = epilogue (warp w reads TMEM lanes 32 (w mod 4) ..).
// Two accumulators of kBN columns alternate, so that the epilogue of one
// tile overlaps the MMAs of the next.
__global__ void __launch_bounds__(kThreads, 1) gf2_tc_kernel(const __grid_constant__ TcMaps maps, uint32_t total, uint32_t bn,
                                                              const uint32_t* __restrict__ dst, uint32_t* out,
                                                              uint32_t out_stride, uint32_t* status, uint32_t stall)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sa = smem;
    uint8_t* sb = smem + kStages * kABytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(sb + kStages * kBBytes);
    uint64_t* empty = full + kStages;
    uint64_t* tfull = empty + kStages;   // [2] accumulator ready (MMA commit)
    uint64_t* tempty = tfull + 2;        // [2] accumulator drained (4 epilogue warps)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
    __shared__ volatile int s_failed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kMTiles = kGf2Bits / kBM;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], kEpilogueWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_failed = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"((uint32_t)kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp >= 2) {
        const uint32_t lanes = tmem + ((uint32_t)(warp & 3) * 32 << 16);
        tmem_fill16(lanes + kScaleA, 0x7F7F7F7Fu);
        tmem_fill16(lanes + kScaleB, 0x7F7F7F7Fu);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cudaGridDependencySynchronize();   // B, and the rings that an earlier kernel still reads

    uint32_t issued = 0;  // producer: K blocks whose copies were started
    if (warp == 0) {
        if (lane == 0) {
            for (uint32_t t = blockIdx.x; t < total && !failed(&s_failed); t += gridDim.x) {
                const TcTile tile = tc_tile(maps, t);
                const int mt = (int)(t % kMTiles), nt = (int)tile.nt;
                const CUtensorMap* ma = &maps.a[tile.j];
                for (int kb = 0; kb < kKBlocks; ++kb, ++issued) {
                    const uint32_t s = issued % kStages, u = issued / kStages;
                    if (issued >= (uint32_t)kStages && !mbar_wait(&empty[s], (u & 1) ^ 1, global_ns() + kWaitLimitNs)) {
                        s_failed = 1;
                        break;
                    }
                    mbar_expect_tx(&full[s], kABytes + bn * kBK);
                    if (stall && blockIdx.x == 0 && issued == 0) continue;   // the failure-path test
                    tma_load_2d(sa + s * kABytes, ma, &full[s], kb * kBK, mt * kBM);
                    tma_load_2d(sb + s * kBBytes, &maps.b, &full[s], kb * kBK, nt * (int)bn);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = instr_desc(bn);
            uint32_t it = 0, lt = 0;
            for (uint32_t t = blockIdx.x; t < total && !failed(&s_failed); t += gridDim.x, ++lt) {
                const uint32_t acc = lt & 1, v = lt >> 1;
                if (lt >= 2 && !mbar_wait(&tempty[acc], (v & 1) ^ 1, global_ns() + kWaitLimitNs)) {
                    s_failed = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + acc * kBN;
                for (int kb = 0; kb < kKBlocks; ++kb, ++it) {
                    const uint32_t s = it % kStages, u = it / kStages;
                    if (!mbar_wait(&full[s], u & 1, global_ns() + kWaitLimitNs)) {
                        s_failed = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t ad = smem_desc(sa + s * kABytes);
                    const uint64_t bd = smem_desc(sb + s * kBBytes);
#pragma unroll
                    for (int kk = 0; kk < kBK / 32; ++kk)  // K = 32 bytes per instruction: +2 in 16-byte units
                        mma_f4(d, ad + 2 * kk, bd + 2 * kk, idesc, tmem + kScaleA, tmem + kScaleB, (kb | kk) != 0);
                    mma_commit(&empty[s]);
                }
                mma_commit(&tfull[acc]);  // arrives once this tile's MMAs have completed
            }
        }
        __syncwarp();
    } else {
        // epilogue: this warp's 32 TMEM lanes = output bits 32 q .. 32 q + 31 of a tile
        const uint32_t q = (uint32_t)(warp & 3);
        uint32_t lt = 0;
        for (uint32_t t = blockIdx.x; t < total; t += gridDim.x, ++lt) {
            const uint32_t acc = lt & 1, v = lt >> 1;
            if (!mbar_wait(&tfull[acc], v & 1, global_ns() + kWaitLimitNs)) {
                s_failed = 1;
                break;
            }
            tc_fence_after();
            if (failed(&s_failed)) break;
            const TcTile tile = tc_tile(maps, t);
            const uint32_t mt = t % kMTiles, nt = tile.nt, n = maps.n[tile.j];
            const uint32_t* to = dst ? dst + maps.at[tile.j] : nullptr;
            const uint32_t word = mt * (kBM / 32) + q;  // ring word of these 32 bits
            static_assert(kBN % 16 == 0, "columns are read 16 at a time");
            for (uint32_t c = 0; c < bn; c += 32) {
                uint32_t vals[32];
                const uint32_t col = tmem + ((q * 32) << 16) + acc * kBN + c;
                tmem_ld16(col, vals);
                if (c + 16 < bn) tmem_ld16(col + 16, vals + 16);
                tmem_ld_wait();
                uint32_t mine = 0;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    if (j >= 16 && c + 16 >= bn) break;
                    // the count is an integer <= 4096: adding 2^23 puts its parity in the last bit
                    const uint32_t bit = __float_as_uint(__uint_as_float(vals[j]) + 8388608.0f) & 1u;
                    const uint32_t b = __ballot_sync(0xFFFFFFFFu, bit);
                    if (lane == j) mine = b;
                }
                const uint32_t st = nt * bn + c + (uint32_t)lane;
                if (st < n && c + lane < bn) {
                    const uint32_t d = to ? to[st] : st;
                    if (d != kNoState) out[(size_t)d * out_stride + word] = mine;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[acc]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (failed(&s_failed)) {
        if (warp == 0 && lane == 0) {
            // the copies of the last (at most kStages) started K blocks may still be in flight
            for (uint32_t kb = issued > (uint32_t)kStages ? issued - kStages : 0u; kb < issued; ++kb)
                (void)mbar_wait(&full[kb % kStages], (kb / kStages) & 1, global_ns() + kWaitLimitNs);
        }
        if (threadIdx.x == 0) {
            *reinterpret_cast<volatile uint32_t*>(status) = 1u;
            __threadfence_system();
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kTmemCols)
                     : "memory");
    }
}

// 32 bits to 32 nibbles of 0 or 1.0 (E2M1: 2): nibble n of word j is bit 4 n + j.
__device__ __forceinline__ uint4 spread32(uint32_t x)
{
    return make_uint4((x << 1) & 0x22222222u, x & 0x22222222u, (x >> 1) & 0x22222222u, (x >> 2) & 0x22222222u);
}

// A[i][k] = bit i of column k of C (column form: column k = 128 ring words).
// A warp transposes 32 x 32 bits: lane l holds output word w of column
// 32 kw + l, and the ballot of bit b is row 32 w + b over those columns.
// Neighbouring warps of a block take neighbouring kw, so a row's 16-byte
// pieces are written by one block.
__global__ void __launch_bounds__(256) expand_matrix_kernel(const uint32_t* __restrict__ cols,
                                                            uint8_t* __restrict__ A)
{
    const uint32_t lane = threadIdx.x & 31u, kw = blockIdx.x * 8 + (threadIdx.x >> 5), w = blockIdx.y;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const uint32_t word = cols[(size_t)(32 * kw + lane) * kGf2Words + w];
    uint32_t row = 0;
#pragma unroll
    for (int b = 0; b < 32; ++b) {
        const uint32_t v = __ballot_sync(0xFFFFFFFFu, (word >> b) & 1u);
        if (lane == (uint32_t)b) row = v;
    }
    *reinterpret_cast<uint4*>(A + (size_t)(32 * w + lane) * kRowBytes + 16 * kw) = spread32(row);
}

// B[s][k] = bit k of state s of `in` (s < n; TMA fills rows past n with 0).  A warp
// takes a state, a lane four of its words (16 bytes of B each), so that four
// reads are under way: 16384 states 11.4 us with one word per thread, 7.1 us so.
__global__ void __launch_bounds__(256) expand_states_kernel(TcStates in, uint32_t n, uint8_t* __restrict__ B)
{
    const uint32_t s = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x & 31u;
    cudaTriggerProgrammaticLaunchCompletion();
    if (!in.settled) cudaGridDependencySynchronize();
    if (s < n) {
        const uint32_t* ring = in.base + (size_t)(in.list ? in.list[s] : s) * in.stride;
        if (in.pend) ring -= in.pend[s] * in.word;
        uint32_t x[4];
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) x[i] = ring[32 * i + lane];
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i)
            *reinterpret_cast<uint4*>(B + (size_t)s * kRowBytes + 16 * (32 * i + lane)) = spread32(x[i]);
    }
    // the product waits for this kernel only: it ends after the one before it
    if (in.settled) cudaGridDependencySynchronize();
}

// ---- host side -------------------------------------------------------------

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

std::mutex g_mu;
EncodeTiled g_encode = nullptr;
bool g_probed = false;
bool g_attr_set[64] = {};
std::vector<std::pair<uint32_t*, uint32_t*>> g_status_free;   // status words without an owner (host, device)

bool init_locked()
{
    if (g_probed) return g_encode != nullptr;
    g_probed = true;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return false;
    }
    g_encode = reinterpret_cast<EncodeTiled>(fn);
    return true;
}

bool make_map(CUtensorMap* m, const uint8_t* base, uint64_t rows, uint32_t box_rows)
{
    const cuuint64_t dims[2] = {(cuuint64_t)kRowBytes, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)kRowBytes};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool gf2_tc_available(int device)
{
    std::lock_guard<std::mutex> lk(g_mu);
    if (!init_locked()) return false;
    int major = 0, minor = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, device) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return major == 10 && minor == 3;
}

size_t gf2_tc_scratch_bytes(uint32_t n) { return (size_t)n * kRowBytes; }

// A tile's time grows with its bytes into shared memory, (kBM + bn) kRowBytes,
// beside the latency of a stage and what the matrices take from HBM.  500
// states by 7 matrices, 5 waves of 240 or of 176 states: 36.4 and 35.2 us; a
// jump of 300 streams by one power, one wave of 240 or 80: 25.1 and 23.3 us; a
// cut call of 400 x 131072 words 66.6 and 62.2 us.
uint32_t gf2_tc_tile(const uint32_t* counts, int n_mats, int sms, uint32_t* waves)
{
    const bool equal = counts[0] == counts[n_mats - 1];   // they never increase
    uint32_t best = kBN;
    uint64_t best_cost = ~uint64_t(0);
    for (uint32_t bn = kBN; bn >= 16; bn -= 16) {
        uint32_t tiles = 0;
        if (equal) tiles = (counts[0] + bn - 1) / bn * (uint32_t)n_mats;
        else
            for (int j = 0; j < n_mats; ++j) tiles += (counts[j] + bn - 1) / bn;
        const uint32_t w = (tiles * (kGf2Bits / kBM) + sms - 1) / sms;
        const uint64_t cost = (uint64_t)w * (kBM + bn);
        if (cost < best_cost) {
            best_cost = cost;
            best = bn;
            *waves = w;
        }
        if (w > 64) break;   // many states: the widest tile
    }
    return best;
}

cudaError_t gf2_tc_expand_matrix(const uint64_t* C, uint8_t* A, cudaStream_t s, bool dependent)
{
    return launch_dependent(dependent, dim3(kGf2Words / 8, kGf2Words), dim3(256), s, expand_matrix_kernel,
                            reinterpret_cast<const uint32_t*>(C), A);
}

cudaError_t gf2_tc_apply(int device, const uint8_t* const* A, int n_mats, const TcStates& in, uint32_t n, uint32_t* out,
                         uint32_t out_stride, const uint32_t* dst, uint8_t* scratch, TcStatus& status, cudaStream_t s,
                         bool dependent, const uint32_t* counts)
{
    if (n == 0 || n_mats == 0) return cudaSuccess;
    if (n_mats < 0 || n_mats > kGf2TcMaxMats) return cudaErrorInvalidValue;
    uint32_t* const word = status.device();
    if (!word) return cudaErrorMemoryAllocation;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms <= 0) sms = 1;
    TcMaps maps{};
    uint32_t at = 0, tiles = 0, waves = 0;
    for (int j = 0; j < n_mats; ++j) maps.n[j] = counts ? counts[j] : n;
    const uint32_t bn = gf2_tc_tile(maps.n, n_mats, sms, &waves);
    for (int j = 0; j < n_mats; ++j) {
        maps.at[j] = at;
        at += maps.n[j];
        tiles += (maps.n[j] + bn - 1) / bn * (kGf2Bits / kBM);
        maps.end[j] = tiles;
    }
    if (tiles == 0) return cudaSuccess;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!init_locked()) return cudaErrorNotSupported;
        for (int j = 0; j < n_mats; ++j)
            if (!make_map(&maps.a[j], A[j], kGf2Bits, kBM)) return cudaErrorInvalidValue;
        if (!make_map(&maps.b, scratch, n, bn)) return cudaErrorInvalidValue;
        if (device >= 0 && device < 64 && !g_attr_set[device]) {
            cudaError_t e = cudaFuncSetAttribute(gf2_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
            if (e != cudaSuccess) return e;
            g_attr_set[device] = true;
        }
    }
    cudaError_t e = launch_dependent(dependent, dim3((n + 7) / 8), dim3(256), s, expand_states_kernel, in, n, scratch);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<uint32_t>(tiles, (uint32_t)sms);
    const char* stall = std::getenv("XG_TC_TEST_STALL");
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gf2_tc_kernel, maps, tiles, bn, dst, out, out_stride, word,
                              (stall && stall[0] == '1') ? 1u : 0u);
}

uint32_t* TcStatus::device()
{
    if (dev_) return dev_;
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_status_free.empty()) {
        constexpr size_t kWords = 1024;   // one page
        void *h = nullptr, *d = nullptr;
        cudaError_t e = cudaHostAlloc(&h, kWords * 4, cudaHostAllocMapped | cudaHostAllocPortable);
        if (e == cudaSuccess) e = cudaHostGetDevicePointer(&d, h, 0);
        if (e != cudaSuccess) {
            cudaGetLastError();
            if (h) cudaFreeHost(h);
            return nullptr;
        }
        for (size_t i = kWords; i-- > 0;)
            g_status_free.emplace_back(static_cast<uint32_t*>(h) + i, static_cast<uint32_t*>(d) + i);
    }
    host_ = g_status_free.back().first;
    dev_ = g_status_free.back().second;
    g_status_free.pop_back();
    *host_ = 0;
    return dev_;
}

TcStatus::~TcStatus()
{
    if (!dev_) return;
    std::lock_guard<std::mutex> lk(g_mu);
    g_status_free.emplace_back(const_cast<uint32_t*>(host_), dev_);
}

bool TcStatus::take()
{
    if (!host_ || !*host_) return false;
    *host_ = 0;
    return true;
}

}  // namespace xg

// GF(2) matrix applications on the tensor cores (see xg_gf2_tc.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "xg_launch.h"

namespace xg {

constexpr int kGf2Bits = 4096;             // state bits = matrix order
constexpr int kGf2Words = kGf2Bits / 32;   // 32-bit ring words per state

// A destination index that takes no result.
constexpr uint32_t kNoState = 0xFFFFFFFFu;

// True on sm_103 with the driver's tensor-map encoder available.
bool gf2_tc_available(int device);

// Bytes of the B operand of n states.
size_t gf2_tc_scratch_bytes(uint32_t n);

// States per output tile (16 .. 240) that a launch of n_mats matrices on
// counts[j] states each takes, and its waves of tiles over the SMs: the
// smallest product of waves and bytes per tile (plain C++).
uint32_t gf2_tc_tile(const uint32_t* counts, int n_mats, int sms, uint32_t* waves);

// Bytes of a matrix as the A operand.
constexpr size_t kGf2TcMatrixBytes = (size_t)kGf2Bits * kGf2Bits / 2;

// A (4096 x 2048 bytes, 8 MiB) = C in FP4 E2M1, row i over input bits k, from
// C in column form (column k = the 128 ring words of C e_k).
// dependent: as in launch_gf2_apply_pairs.
cudaError_t gf2_tc_expand_matrix(const uint64_t* C, uint8_t* A, cudaStream_t s, bool dependent = false);

// Most matrices applied by one launch.
constexpr int kGf2TcMaxMats = 7;

// The word that a tensor-core launch sets when one of its waits gives up: its
// results are then not valid.  One per owner of such launches (a context, a
// batch launcher), so that a failure reaches its owner and no other.  The word
// is mapped host memory from a process-wide list, taken at the owner's first
// launch and given back with the owner, whose launches have finished by then.
class TcStatus {
public:
    TcStatus() = default;
    TcStatus(const TcStatus&) = delete;
    TcStatus& operator=(const TcStatus&) = delete;
    ~TcStatus();
    uint32_t* device();                                    // null: no memory for the word
    const volatile uint32_t* host() const { return host_; }   // null before the first launch
    bool take();                                           // a wait gave up since the last call

private:
    volatile uint32_t* host_ = nullptr;
    uint32_t* dev_ = nullptr;
};

// The states that are read: state i is the 128 words at base + list[i] stride
// (list null: i), or, with pend, at base + i stride - pend[i] word (the ring in
// a stream's window, base its position without pending words).  settled: no
// kernel since the last ordinary launch writes them, so that a dependent launch
// may read them beside the kernels before it.
struct TcStates {
    const uint32_t* base;
    uint32_t stride;
    const uint32_t* list;
    const uint32_t* pend;
    uint32_t word;
    bool settled = false;
};

// out[dst[j n + i] out_stride ..] = C_j (state i) for i < n and j < n_mats (<=
// kGf2TcMaxMats; dst null: one matrix, i), with A[j] from gf2_tc_expand_matrix.
// counts (host, n_mats entries, each <= n, not increasing): matrix j applies to
// the first counts[j] states, and the destinations of the matrices follow one
// another in dst.
// All states are read before the first is written: out may overlap the states
// with one matrix, else if no destination is a source.  kNoState destinations
// are skipped.  scratch: gf2_tc_scratch_bytes(n) bytes, 16-byte aligned, reused
// once the launch has finished.  Asynchronous on s.  dependent: as in
// launch_gf2_apply_pairs.
cudaError_t gf2_tc_apply(int device, const uint8_t* const* A, int n_mats, const TcStates& in, uint32_t n, uint32_t* out,
                         uint32_t out_stride, const uint32_t* dst, uint8_t* scratch, TcStatus& status, cudaStream_t s,
                         bool dependent = false, const uint32_t* counts = nullptr);

}  // namespace xg

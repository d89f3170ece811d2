// Jump-ahead: powers of the GF(2) transition matrix and their application.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "xg_launch.h"
#include "xorgens_gb300.h"

namespace xg {

class TcStatus;

constexpr int kMaxPow = 64;  // C_k = M^(2^k), k < 64
// Matrix families: the 32-bit parameter sets 0 (default) and 1 (paper), and
// the 64-bit-word generator.
constexpr int kJumpSetW64 = 2;

// Most matrices applied by one launch of the table kernel.
constexpr int kMaxMats = 7;

// C_k for a device and matrix family, built on first use (on stream s, each
// from the one before; 2 MiB each, kept until the process exits).  Null on failure.
const uint64_t* jump_matrix(int device, int param_set, int k, cudaStream_t s, xg_status* st);

// out[d_dst[i]] ^= C in[d_src[i]] for n pairs of 128-word states.  in and out
// may be one array; destinations are distinct, not among the sources, and
// zeroed beforehand.  dependent: the kernel before it on the stream is one of
// this file's or of the cut calls' set-up, so the launch may overlap its end
// (both wait for each other where it matters).
cudaError_t launch_gf2_apply_pairs(const uint64_t* C, const uint32_t* in, uint32_t* out, uint32_t n,
                                   const uint32_t* d_src, const uint32_t* d_dst, int sm_count, cudaStream_t s,
                                   bool dependent = false);

// The same for several matrices in one launch: out[d_dst[j n + i]] ^=
// C[j] in[d_src[i]] for j < n_mats (<= kMaxMats); kNoState destinations are
// skipped.  early: a dependent launch after it may become resident while it
// runs.  Wrong for long kernels of many blocks, which would be spread over the
// SMs by what this one has left free: 16 streams of 2^18 words in 128 pieces
// 45 us early, 33 us not.  counts as in gf2_tc_apply.
cudaError_t launch_gf2_apply_multi(const uint64_t* const* C, int n_mats, const uint32_t* in, uint32_t* out, uint32_t n,
                                   const uint32_t* d_src, const uint32_t* d_dst, int sm_count, cudaStream_t s,
                                   bool dependent = false, bool early = true,
                                   const uint32_t* counts = nullptr);

// M^(j 2^k) for 1 <= j <= 7, built on first use like jump_matrix.  The odd
// multiples and the FP4 copies of a device take at most 3 GiB in all
// (XG_JUMP_TABLE_MIB sets another limit); past it, and where the device has no
// memory left, a new one is XG_ENOMEM, and the callers do without: jumps and
// batches with the powers and the table kernel, cut calls as whole calls.
const uint64_t* jump_matrix_multiple(int device, int param_set, int j, int k, cudaStream_t s, xg_status* st);

// The same as the A operand of gf2_tc_apply.
const uint8_t* jump_matrix_tc(int device, int family, int j, int k, cudaStream_t s, xg_status* st);

// Whether an application with n results runs on the tensor cores (sm_103 and
// n >= XG_GF2_TC_MIN_STATES, default `from`; XG_JUMP_TENSOR_CORES=0 turns the
// tensor-core path off), and the device scratch it then needs (0 otherwise).
// A launch for 192 results costs 13 us on the tensor cores and 15 by the table
// kernel (0.05 us per result), whose launches overlap better.
constexpr uint32_t kTcMinResults = 192;
bool gf2_use_tc(int device, uint32_t n, uint32_t from = kTcMinResults);
size_t gf2_apply_scratch(int device, uint32_t n);

// rings[d_dst[i]] = C_k rings[d_src[i]] for n pairs, C_k the power 2^k of
// the matrix family (destinations distinct and not among the sources).  On
// the tensor cores when gf2_use_tc(device, n), scratch (gf2_apply_scratch
// bytes) is given and the FP4 copy is to be had, else with the table kernel.
// Asynchronous on s, except
// that a power's first use builds it.  After synchronising, a caller that
// may have used the tensor cores checks the status.  The table
// kernel XORs into the destinations, so it zeroes them first unless the
// caller says they are zero already (dst_zeroed).
cudaError_t gf2_apply(int device, int family, int k, uint32_t* rings, uint32_t n, const uint32_t* d_src,
                      const uint32_t* d_dst, uint8_t* scratch, TcStatus& tc, int sm_count, cudaStream_t s, xg_status* st,
                      bool dst_zeroed = false);

// Advance n states by `words` positions: M^words applied to rings[0, n),
// with rings[n, 2n) as the second buffer (*result_hi: the result ended there)
// and d_idx the identity list 0 .. 2n - 1.  With several set bits (2, 4 or 7 by
// the number of states) the powers are multiplied first and the product applied
// once.  work: gf2_jump_work_bytes bytes of device memory, 256-byte aligned
// (the tensor-core operand or the product's work area).
size_t gf2_jump_work_bytes(int device, uint32_t n, uint64_t words, bool in_place);
cudaError_t gf2_jump_states(int device, int family, uint64_t words, uint32_t* rings, uint32_t n,
                            const uint32_t* d_idx, uint8_t* work, TcStatus& tc, int sm_count, cudaStream_t s, xg_status* st,
                            bool* result_hi);

// Whether a jump applies one matrix (a power, or the product of several) on
// the tensor cores (false too where there is no memory for a power's FP4 copy,
// which is built here); then gf2_jump_windows reads the rings of n consecutive
// streams in their windows and writes them back there, without pending words:
// for 16384 streams it saves the copies of all rings out of the windows and
// back (25 of 229 us).  The caller resets pend and advances the Weyl words.
// work as for gf2_jump_states.
struct JumpWindows {
    uint32_t* win;    // the first stream's window, kWin 32-bit words each
    uint32_t* pend;   // of the first stream
    uint32_t word;    // 32-bit words per generator word
};
bool gf2_jump_in_place(int device, int family, uint32_t n, uint64_t words, TcStatus& tc, cudaStream_t s);
cudaError_t gf2_jump_windows(int device, int family, uint64_t words, const JumpWindows& win, uint32_t n, uint8_t* work,
                             TcStatus& tc, int sm_count, cudaStream_t s, xg_status* st);

// ids[i] = first + i for i < n, then ids[n + j] = j for j < 2n (3n entries).
cudaError_t launch_jump_index(uint32_t* ids, uint32_t n, uint32_t first, cudaStream_t s);

// rings[d_idx[i]] = 0 for n listed 128-word rings.
cudaError_t zero_rings(uint32_t* rings, const uint32_t* d_idx, uint32_t n, cudaStream_t s);

// rings[k] = current ring of stream d_streams[k]; weyl0[k * weyl0_stride] =
// its Weyl word advanced by d_skip[k] words (weyl0 may be null).
cudaError_t launch_gather_rings(const State& st, const uint32_t* d_streams, uint32_t n, uint32_t* d_rings,
                                const uint64_t* d_skip, uint32_t* d_weyl0, uint32_t weyl0_stride, uint32_t omega,
                                cudaStream_t s);

}  // namespace xg

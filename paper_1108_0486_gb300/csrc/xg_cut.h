// Cut calls: a plain generation call on few streams, generated as pieces of
// 2^q outputs per stream that different warps run at once.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "xg_gf2_tc.h"
#include "xg_launch.h"
#include "xorgens_gb300.h"

namespace xg {

// Output kinds of cut_choose: those of xg_launch.h, and the 64-bit words'.
constexpr int kCutU64 = 4;
constexpr int kCutUniform64 = 5;

// The piece length 2^q that a call of n outputs (of any kind) on nstreams
// streams is predicted to run fastest with, or 0 when the whole call is (plain
// C++, no device access).  forced: a piece length set by the caller (a power
// of two >= 64), or 0.
int cut_choose(int kind, uint32_t nstreams, uint64_t n, int sm_count, uint64_t forced);

// Predicted time of the prologue in us (the same).
double cut_prologue_us(uint32_t nstreams, uint64_t pieces, int sm_count);

// A context's workspace for cut calls (grow-only, freed with the context).
// Used on the context's stream of the moment: the event follows the last use,
// and a use on another stream waits for it.  Streams are told apart by their
// ids: a handle may name another stream later (one made after it was
// destroyed, or another thread's per-thread default stream).
struct CutWorkspace {
    void* mem = nullptr;
    size_t bytes = 0;
    cudaEvent_t event = nullptr;
    unsigned long long stream_id = 0;   // of the last use
    bool used = false;                  // the event has been recorded

    xg_status ensure(size_t want);
    xg_status acquire(cudaStream_t s);   // before the first launch that uses it
    xg_status release(cudaStream_t s);   // after the last one that was enqueued
    void destroy();
};

// The streams of a context as the prologue reads them: windows of kWin 32-bit
// words, `word` of them (1 or 2) per generator word.
struct CutStreams {
    int device;
    int sm_count;
    int family;             // matrix family (xg_jump.h)
    const uint32_t* win;
    const uint32_t* pend;
    const uint32_t* weyl;
    uint32_t word;
    TcStatus* tc;           // the context's
};

// What the prologue leaves in the workspace: 128-word rings [nstreams][pieces],
// the streams' Weyl words [nstreams], extra bytes (256-byte aligned).
struct CutRings {
    uint32_t* rings;
    uint32_t* weyl0;
    char* extra;
};

// Enqueue the prologue of a call on streams [first, first + nstreams) cut into
// pieces of 2^q words on stream s.  The kernel that follows may be launched as
// a dependent one; then ws.release().  *ran = false (and XG_OK) when the
// workspace or a matrix could not be had: nothing was enqueued.
xg_status cut_prologue(CutWorkspace& ws, const CutStreams& streams, uint32_t first, uint32_t nstreams, uint32_t pieces,
                       int q, size_t extra_bytes, cudaStream_t s, CutRings* out, bool* ran);

// Generate the call cut into pieces of 2^q outputs.  Asynchronous on the
// context's stream; the outputs and the stream states are exactly those of
// the whole call (kNormalSum, out = one sum per stream and ld unused: the same
// normals, added up in another order).  *ran as for cut_prologue.
xg_status cut_generate(xg_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* out, uint64_t ld,
                       int q, bool* ran);

}  // namespace xg

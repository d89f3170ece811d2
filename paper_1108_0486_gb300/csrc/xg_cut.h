// Cut calls: a plain generation call on few streams, generated as pieces of
// 2^q outputs per stream that different warps run at once.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "xorgens_gb300.h"

namespace xg {

// The piece length 2^q that a call of n outputs (of any kind) on nstreams
// streams is predicted to run fastest with, or 0 when the whole call is (plain
// C++, no device access).  forced: a piece length set by the caller (a power
// of two >= 64), or 0.
int cut_choose(int kind, uint32_t nstreams, uint64_t n, int sm_count, uint64_t forced);

// Generate the call cut into pieces of 2^q outputs.  Asynchronous on the
// context's stream; the outputs and the stream states are exactly those of
// the whole call (kNormalSum, out = one sum per stream and ld unused: the same
// normals, added up in another order).  *ran = false (and XG_OK) when the
// workspace could not be had: nothing was enqueued.
xg_status cut_generate(xg_ctx* c, int kind, uint32_t first, uint32_t nstreams, uint64_t n, void* out, uint64_t ld,
                       int q, bool* ran);

}  // namespace xg

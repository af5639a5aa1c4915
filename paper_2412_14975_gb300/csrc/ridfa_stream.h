// Host interface of the stream kernels (ridfa_stream.cu): recognition of one text by automata with
// a merge graph.  Not part of the public ABI.
#pragma once

#include <cuda_runtime_api.h>

#include "ridfa_internal.h"

namespace ridfa {

struct StreamShape {
    uint32_t per_chunk = 1;      // pieces a chunk is cut into
    uint64_t pieces = 0;
    bool walk_only = false;      // short pieces: one-byte steps only, no main table to set up
    uint32_t block = 32, grid = 1, warps = 1;   // warps of a block that take pieces
    uint32_t join_chunks = 256;  // chunks per join block
    uint32_t join_blocks = 1;
    bool fused = false;          // the join runs in the last block of the reach launch
    uint32_t group = 0, groups = 0;  // pieces a group, groups a chunk is joined by; 0: its pieces themselves
    size_t smem = 0;
};

// Buffers of one call.  ticket (two words) and work are zero before and after every call.
struct StreamCall {
    const HostAutomaton *H = nullptr;
    const DeviceAutomaton *D = nullptr;
    const uint8_t *text = nullptr;
    uint64_t len = 0;
    uint32_t c = 0;
    uint32_t *res = nullptr;         // [pieces]
    uint32_t *groups = nullptr;      // [c * groups], with groups
    uint16_t *tables = nullptr;      // [c * groups][n]
    uint16_t *maps = nullptr;        // [c][k]
    uint32_t *dinfo = nullptr;       // [c]
    uint32_t *partials = nullptr;    // [join_blocks][kPartialWords]
    uint32_t *ticket = nullptr, *work = nullptr, *status = nullptr;
    uint8_t *accept = nullptr;
    uint8_t *h_accept = nullptr;     // page-locked host copies of the results, or null
    uint32_t *h_status = nullptr;
    ridfa_shard_summary *summary = nullptr;
    cudaEvent_t between = nullptr;   // recorded between the two launches when set
};

bool stream_takes(const HostAutomaton &H, uint64_t len, uint32_t c);
StreamShape stream_shape(const HostAutomaton &H, uint64_t len, uint32_t c, int sms);
ridfa_kernel_report stream_report(const HostAutomaton &H, const StreamShape &S);
cudaError_t stream_launch(const StreamCall &C, const StreamShape &S, cudaStream_t st);

}  // namespace ridfa

// Host interface of the set kernels (ridfa_set.cu): recognition of one text by automata whose runs stay
// apart, over an alphabet of at most four bytes.  Not part of the public ABI.
#pragma once

#include <cuda_runtime_api.h>

#include "ridfa_internal.h"

namespace ridfa {

struct SetCall {
    const HostAutomaton *H = nullptr;
    const DeviceAutomaton *D = nullptr;
    const uint8_t *text = nullptr;
    uint64_t len = 0;
    uint32_t c = 0, spc = 0;         // chunks, pieces of each (set_pieces)
    uint8_t *scratch = nullptr;      // set_scratch(c, spc) bytes, aligned to 256
    uint16_t *maps = nullptr;        // [c][k], or null
    uint32_t *ticket = nullptr, *status = nullptr;   // ticket: zero before and after every call
    uint8_t *accept = nullptr;
    uint8_t *h_accept = nullptr;     // page-locked host copies of the results, or null
    uint32_t *h_status = nullptr;
    cudaEvent_t between = nullptr;   // recorded between the two launches when set
};

// Pieces the set kernels cut each chunk into; 0: the call is not theirs.
uint32_t set_pieces(const HostAutomaton &H, uint64_t len, uint32_t c, int sms);
size_t set_scratch(uint32_t c, uint32_t spc);
cudaError_t set_launch(const SetCall &C, int sms, cudaStream_t st);

}  // namespace ridfa

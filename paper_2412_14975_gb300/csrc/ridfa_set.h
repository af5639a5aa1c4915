// Host interface of the set kernels (ridfa_set.cu): recognition of one text by automata whose runs stay
// apart, over an alphabet of at most four bytes.  Not part of the public ABI.
#pragma once

#include <cuda_runtime_api.h>

#include <vector>

#include "ridfa_internal.h"
#include "ridfa_stream_batch.h"

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
ridfa_kernel_report set_report(const HostAutomaton &H, uint32_t c, uint32_t spc, int sms);
cudaError_t set_launch(const SetCall &C, int sms, cudaStream_t st);

// The texts of one program of a batch, each of kSetBatchText bytes or more, on `grid` SMs: only accept
// bits are asked for, so a piece is entered through the interface slots, as a chunk is.
constexpr uint64_t kSetBatchText = 32;         // (as deep as the graph may be)
constexpr uint64_t kSetBatchPiece = 512;       // bytes a piece has at least, but a text's last
constexpr size_t kSetBatchResult = kSetRuns * 2 + 8 + 4;     // bytes of scratch a piece
// Text a batch's launch has to have.  (50 texts of 16 KB against 3 REs, one of them the codon RE: 242 us
// with its texts in the general kernel, 58 us in this one; 30 texts of 2 KB: 181 and 56.)
constexpr uint64_t kSetBatchBytes = 4096;
constexpr uint32_t kSetBatchProgs = 16;
struct SetBatchPlan {
    const HostAutomaton *H = nullptr;
    const DeviceAutomaton *D = nullptr;
    std::vector<StreamBatchText> texts;
    std::vector<uint32_t> bases;
    uint32_t pieces = 0, grid = 0;
    size_t image_bytes = 0, result_bytes = 0, o_bases = 0;
};
double set_batch_weight(const HostAutomaton &H);         // time per byte, a two-byte stream table's being 1
void plan_set_batch(SetBatchPlan &P, const StreamBatchSource &src, uint32_t sms);
void set_batch_image(const SetBatchPlan &P, uint8_t *img);
cudaError_t set_batch_launch(const SetBatchPlan &P, const uint8_t *dev_image, uint8_t *dev_results, uint8_t *d_accept, cudaStream_t st);

}  // namespace ridfa

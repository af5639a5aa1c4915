// Host interface of the batched stream kernels (ridfa_stream_batch.cu): the texts of a batch whose
// programs have a merge graph.  Not part of the public ABI.
#pragma once

#include <cuda_runtime_api.h>

#include <vector>

#include "ridfa_internal.h"

namespace ridfa {

constexpr uint32_t kStreamBatchProgs = 64;       // programs of one plan at most
constexpr uint64_t kStreamBatchPiece = 96;       // bytes a piece has at least, but a text of one piece
// Shared memory that launches which run side by side take at least: over half of an SM's, so that each
// of their blocks has an SM to itself (blocks of small tables otherwise met on one SM while others
// stood idle).
constexpr size_t kStreamBatchSmem = 116 * 1024;

struct StreamBatchText {         // one text as the kernels see it
    const uint8_t *text;
    uint64_t len;
    uint64_t step;               // bytes per piece, 16 fraction bits
    uint32_t base, pieces;       // its pieces in its program's numbering (0 for an empty text)
    uint32_t prog, item;         // prog: index into the stream programs
};
struct StreamBatchPart {         // tasks (32 pieces each) [task0, task1) of one program, for one block
    uint32_t prog, task0, task1, pad;
};

// One launch: the programs of one table form (or all of them, in one-byte steps).
struct StreamBatchLaunch {
    uint32_t form = 0, first = 0;                    // first: its entry in first_part
    uint32_t grid = 0, block = 0;
    size_t smem = 0;
    uint32_t text0 = 0, n_texts = 0, most = 0;       // its texts, joined right after it; pieces of the longest
};

// Plan of a batch's stream part.  The descriptors of plan_stream_image() go to the device as they
// are; res (results_words words) is device scratch.
struct StreamBatchPlan {
    std::vector<const HostAutomaton *> H;
    std::vector<const DeviceAutomaton *> D;
    std::vector<uint32_t> text0, np, res0;           // per program: first text, pieces, first result
    std::vector<StreamBatchText> texts;              // grouped by program
    std::vector<uint32_t> bases;                     // texts[i].base, packed for the search
    std::vector<StreamBatchPart> parts;
    std::vector<uint32_t> first_part;                // per launch: grid + 1 entries
    std::vector<StreamBatchLaunch> launches;         // to run side by side
    std::vector<uint8_t> tables;                     // the reach launches' table arguments
    uint64_t bytes = 0;
    bool walk_only = false;
    size_t image_bytes = 0, result_words = 0;
    size_t o_progs = 0, o_texts = 0, o_bases = 0, o_parts = 0, o_first = 0;
    bool empty() const { return texts.empty(); }
};

// Texts of one program in the order of its items; `item` indexes the batch's accept bytes.
struct StreamBatchItem {
    const uint8_t *text;
    uint64_t len;
    uint32_t item;
};

struct StreamBatchSource {       // one program with its texts
    const HostAutomaton *H;
    const DeviceAutomaton *D;
    std::vector<StreamBatchItem> items;
};

// Plan the sources (reordered by table form) on `blocks` blocks (one per SM).
void plan_stream_batch(StreamBatchPlan &P, std::vector<StreamBatchSource> &src, uint32_t blocks);
void stream_batch_image(const StreamBatchPlan &P, uint8_t *dev_image, uint32_t *dev_results, uint8_t *img);
cudaError_t stream_batch_reach(const StreamBatchPlan &P, const StreamBatchLaunch &L, const uint8_t *dev_image, cudaStream_t st);
cudaError_t stream_batch_join(const StreamBatchPlan &P, const StreamBatchLaunch &L, const uint8_t *dev_image, uint8_t *d_accept, cudaStream_t st);

}  // namespace ridfa

// Internal structures shared by the host compiler (ridfa_compile.cpp) and the device code
// (ridfa_device.cu).  Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cstddef>
#include <cuda_runtime_api.h>
#include <nvtx3/nvToolsExt.h>
#include <mutex>
#include <string>
#include <vector>

#include "ridfa.h"

namespace ridfa {

// A named NVTX range over a host scope (compile, reach launches, join launch, batch and server
// launches), for timeline tools such as Nsight Systems; free when no tool is attached.
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// The merge graph of an automaton: what becomes of the runs from all of its states at once.
// A node is a function f from the states to the states (or undefined) that some byte sequence
// performs; the root is the identity.  Functions with two or more distinct defined values are
// inner nodes; a function with one value v is a leaf, and the run goes on alone from v.  A function
// is kept as (partition, images): part[pid][x] = the block of state x (kNoBlock: its run died),
// images[b] = the state of block b's runs.  A chunk (or any piece of one) is then read by one lane:
// down the graph until a leaf, on with the leaf's single run to the end.  What is left of the
// piece's function is one word: (pid, state) -- x goes to state if part[pid][x] is a block -- or an
// inner node.  Only built where the graph is small (most automata of practical REs: all runs merge
// within tens of bytes); ok = false otherwise.
struct HostMerge {
    bool ok = false;
    uint32_t inner = 0, parts = 0;
    std::vector<uint16_t> next;       // [inner][C]: an inner node, or kLeafBit | leaf
    std::vector<uint16_t> walk;       // [n_states + 1 + inner][C]: one-byte steps of the states (as
                                      // trans), then of the nodes (node u as n_states + 1 + u; an
                                      // edge to a leaf goes to the leaf's state)
    std::vector<uint16_t> edge_pid;   // [inner][C]: the leaf's partition, for edges to leaves
    std::vector<uint32_t> leaf;       // [leaves]: pid << 16 | state; leaf 0: every run dead
    std::vector<uint16_t> node_part;  // [inner]
    std::vector<uint32_t> node_img;   // [inner]: offset into images
    std::vector<uint16_t> images;
    std::vector<uint16_t> part;       // [parts][n_states]; partition 0: all dead
    std::vector<uint32_t> slot_alive; // [parts][kw]: slots whose start state has a block
};
constexpr uint16_t kLeafBit = 0x8000;
constexpr uint16_t kNoBlock = 0xFFFF;

// Main-loop table of the stream kernels (ridfa_stream.cu), chosen per automaton on the host.
//   kStreamField: the live bytes (those some position reads) differ in a field of `width` <= 2 bits
//     at bit `shift`; codes come from the field by arithmetic, `canon` holds the byte of each code
//     (a byte that is not its code's is not in the alphabet and kills the run), one lookup takes
//     `group` bytes: column = the codes, first byte lowest.
//   kStreamPair / kStreamSingle: two / one bytes a lookup; byte_code[b] = the column offset of b as
//     first byte (low half) and second byte (high half) of a pair, whose sum is the column.
// Entries are next states of `entry` bytes (1 when all ids and the dead state fit 8 bits, else 2);
// row s, column col: word s * row_words + col / (4 / entry), each word in `copies` lane copies.
enum StreamKind : uint32_t { kStreamNone = 0, kStreamField = 1, kStreamPair = 2, kStreamSingle = 3 };
struct HostStream {
    uint32_t kind = kStreamNone;
    uint32_t entry = 1, copies = 32, row_words = 0, group = 1, shift = 0, width = 0;
    uint32_t canon = 0;
    uint32_t warps = 0;               // warps a block holds beside the table (and its staging)
    float cost = 0;                   // estimated shared-memory cycles per 32 text bytes
    std::vector<uint32_t> byte_code;  // [256] (kStreamPair, kStreamSingle)
    std::vector<uint32_t> words;      // [(n_states + 1) * row_words]
};

// Automata whose runs stay apart, over an alphabet of at most four bytes (set kernels, ridfa_set.cu): the
// functions that the first `depth` bytes perform on the interface slots, all of which have fewer than
// kSetRuns distinct values, so that a lane takes up a chunk's runs after walking `depth` edges.
struct HostSet {
    bool ok = false;
    uint32_t depth = 0, inner = 0, parts = 0;
    std::vector<uint16_t> next;       // [inner][C]: an inner node, or kLeafBit | leaf (leaf 0: all dead)
    std::vector<uint32_t> leaf;       // [leaves][2]: partition, offset into images
    std::vector<uint16_t> images;     // states of a leaf's blocks, kSetRuns each (unused ones: n_states)
    std::vector<uint8_t> part;        // [parts][k]: block of each slot, 0xFF: dead
    std::vector<uint32_t> block_mask; // [parts][kw][kSetRuns]: slots of each block
    HostStream table;                 // kStreamField, entries of 2 bytes
    uint32_t back_depth = 0;          // 0: not built.  The sets the bytes before a piece leave of all states;
                                      // every string of back_depth bytes comes to a leaf:
    std::vector<uint16_t> back_next;  // [inner sets][C]: an inner set, or kLeafBit | leaf (leaf 0: all dead)
    std::vector<uint16_t> back_images;// [leaves][kSetRuns]: states (unused ones: n_states)
};
constexpr uint32_t kSetRuns = 16;     // places; at most 15 are taken (15 marks a dead run in 4 bits)

// One speculative automaton as the device sees it: the RI-DFA B with its interface
// (Sec. 3.1-3.4) or the minimal DFA with every state initial (Sec. 2).
struct HostAutomaton {
    uint32_t n_states = 0;            // |P| (or |Q|); the dead state has id n_states
    uint32_t n_classes = 0;           // byte classes C
    uint32_t k = 0;                   // interface slots
    uint32_t kw = 0;                  // 32-bit words per interface-set row: ceil(k / 32)
    uint32_t q0_slot = 0;             // slot whose start state is {q0} (or the DFA start)
    std::vector<uint16_t> trans;      // [(n_states + 1) * n_classes], dead row / moves = n_states
    std::vector<uint8_t> classmap;    // [256]
    std::vector<uint8_t> final_flag;  // [n_states]
    std::vector<uint32_t> final_bits; // [ceil((n_states + 1) / 32)]
    std::vector<uint32_t> ifmask;     // [(n_states + 1) * kw]: slots of if_min({p}); dead row = 0
    std::vector<uint16_t> slot_state; // [k]: start state of each slot
    uint32_t merges = 0;              // 1: runs from every slot merge on random text (merge_hint)
    HostMerge merge;
    HostStream stream;
    HostSet set;                      // only where merge is not built
};

// Build H.merge with H.stream, or H.set, where they are small enough (ridfa_merge.cpp).
void build_stream(HostAutomaton &H);
// Shared memory of a stream kernel's block besides the staging buffers: tables and the compact
// copies for the ragged ends.
size_t stream_table_bytes(const HostAutomaton &H);
size_t stream_walk_bytes(const HostAutomaton &H);      // the one-byte tables alone
size_t set_rest_bytes(const HostAutomaton &H);         // of a set kernel's block besides the table
constexpr size_t kStreamSmem = 226 * 1024;        // shared memory a stream block may take
constexpr size_t kStreamWalkSmem = 24 * 1024;     // a walk table up to this size sits in shared memory,
                                                  // a larger one is read through L1
constexpr size_t kStreamStaging = 4096;           // per-warp staging (kStreamPair, kStreamSingle)

// The tables of an automaton that go to the device, in the order they have there: f(table, data, bytes).
// kTabAll (state s for every state s) has no data of its own.
enum DeviceTable : uint32_t {
    kTabTrans, kTabClass, kTabFinal, kTabIfmask, kTabSlots, kTabAll,
    kTabWalk, kTabEdge, kTabNodePart, kTabNodeImg, kTabImages, kTabPart, kTabAlive, kTabCode, kTabWords,
    kTabSetNext, kTabSetLeaf, kTabSetImages, kTabSetPart, kTabSetMask, kTabSetWords, kTabBackNext, kTabBackImages,
    kTables
};
template <class F>
void each_table(const HostAutomaton &H, F f) {
    auto vec = [&](DeviceTable t, const auto &v) { f(t, static_cast<const void *>(v.data()), v.size() * sizeof(v[0])); };
    vec(kTabTrans, H.trans);
    vec(kTabClass, H.classmap);
    vec(kTabFinal, H.final_bits);
    vec(kTabIfmask, H.ifmask);
    vec(kTabSlots, H.slot_state);
    f(kTabAll, static_cast<const void *>(nullptr), static_cast<size_t>(H.n_states) * 2);
    if (H.stream.kind != kStreamNone) {
        vec(kTabWalk, H.merge.walk);
        vec(kTabEdge, H.merge.edge_pid);
        vec(kTabNodePart, H.merge.node_part);
        vec(kTabNodeImg, H.merge.node_img);
        vec(kTabImages, H.merge.images);
        vec(kTabPart, H.merge.part);
        vec(kTabAlive, H.merge.slot_alive);
        vec(kTabCode, H.stream.byte_code);
        vec(kTabWords, H.stream.words);
    }
    if (H.set.ok) {
        vec(kTabSetNext, H.set.next);
        vec(kTabSetLeaf, H.set.leaf);
        vec(kTabSetImages, H.set.images);
        vec(kTabSetPart, H.set.part);
        vec(kTabSetMask, H.set.block_mask);
        vec(kTabSetWords, H.set.table.words);
        vec(kTabBackNext, H.set.back_next);
        vec(kTabBackImages, H.set.back_images);
    }
}
// Every table begins on a 256-byte boundary of one block of this many bytes.
inline size_t table_room(size_t bytes) { return (bytes + 255) & ~static_cast<size_t>(255); }
inline size_t device_table_bytes(const HostAutomaton &H) {
    size_t total = 0;
    each_table(H, [&](DeviceTable, const void *, size_t n) { total += table_room(n); });
    return total;
}

// Device copy of one automaton (one per device it was uploaded to).
struct DeviceAutomaton {
    int device = -1;
    uint16_t *trans = nullptr;
    uint8_t *classmap = nullptr;
    uint32_t *final_bits = nullptr;
    uint32_t *ifmask = nullptr;
    uint16_t *slot_state = nullptr;
    uint16_t *all_states = nullptr;   // [n_states]: state s (every state as a start, for pieces)
    // merge graph and stream table (HostMerge, HostStream); null when not built
    uint16_t *mg_walk = nullptr, *mg_edge_pid = nullptr, *mg_node_part = nullptr, *mg_images = nullptr, *mg_part = nullptr;
    uint32_t *mg_node_img = nullptr, *mg_slot_alive = nullptr;
    uint32_t *st_code = nullptr, *st_words = nullptr;
    // set tables (HostSet)
    uint16_t *set_next = nullptr, *set_images = nullptr, *set_back_next = nullptr, *set_back_images = nullptr;
    uint32_t *set_leaf = nullptr, *set_block_mask = nullptr, *set_words = nullptr;
    uint8_t *set_part = nullptr;
    size_t bytes = 0;
};

// The position NFA over byte classes, for the NFA variant of the classic algorithm (the
// comparator of Sec. 2 / Table 3): follow rows, class rows (positions reading the class) and the
// final set as bitsets of nw 32-bit words (bit q of word q / 32 = NFA state q; 0 = q0).  Kept
// only when n <= 128 (nw <= 4); n = 0 otherwise.
struct HostNfa {
    uint32_t n = 0, nw = 0, n_classes = 0;
    std::vector<uint8_t> classmap;    // [256]
    std::vector<uint32_t> follow;     // [n][nw]
    std::vector<uint32_t> cls;        // [n_classes][nw]
    std::vector<uint32_t> finals;     // [nw]
};

// Device copy of a HostNfa (one per device it was uploaded to): one allocation.
struct DeviceNfa {
    int device = -1;
    void *base = nullptr;
    const uint8_t *classmap = nullptr;
    const uint32_t *follow = nullptr, *cls = nullptr, *finals = nullptr;
    void *scratch = nullptr;          // the call's relations (grown on demand)
    size_t scratch_bytes = 0;
    uint8_t *h_accept_pinned = nullptr;
};

// What one join scan works in: two result words and working space on the device, two page-locked words.
struct ScanSpace {
    void *base = nullptr;             // the words, then (256 bytes on) the working space
    size_t bytes = 0;
    uint64_t *host = nullptr;
};

// Per-device scratch of a program: chunk maps when the caller passes none, per-chunk summaries,
// the join's partial products, a block ticket, the status word and the accept byte.
struct DeviceScratch {
    int device = -1;
    void *base = nullptr;
    size_t bytes = 0;
    uint8_t *h_accept_pinned = nullptr;
    uint32_t *h_status_pinned = nullptr;
    void *ev[3] = {nullptr, nullptr, nullptr};   // cudaEvent_t: before reach, before join, after
    bool profiled = false;
    ridfa_plan_report last_plan{};               // the reach plan of the last call on this device
    ridfa_kernel_report last_kernel{};           // what it ran in
    bool planned = false;
    bool stream_call = false;                    // the last call took the stream kernels: its plan on the
    bool stream_dfa = false;                     // general path is worked out when asked for
    const uint8_t *stream_text = nullptr;        // (only its alignment is looked at)
    uint64_t stream_len = 0;
    uint32_t stream_chunks = 0;
    ScanSpace scan;                              // of the last join scan, while none runs
};

}  // namespace ridfa

struct ridfa_program {
    std::string re;
    uint32_t n_nfa = 0;
    std::vector<std::vector<uint32_t>> state_sets;   // NFA states of each RI-DFA state
    std::vector<uint32_t> slots;                      // representative NFA state per slot
    std::vector<uint32_t> delegate_slot;              // NFA state -> slot of its representative
    ridfa::HostAutomaton rid;
    ridfa::HostAutomaton dfa;
    bool has_dfa = false;
    ridfa::HostNfa nfa;                               // the NFA variant's tables (n <= 128)
    // device side (filled lazily by the device code)
    mutable std::mutex mu;
    mutable std::vector<ridfa::DeviceAutomaton> dev_rid, dev_dfa;
    mutable std::vector<ridfa::DeviceScratch> scratch;
    mutable std::vector<ridfa::DeviceNfa> dev_nfa;
};

namespace ridfa {
void release_device(const ridfa_program *prog);   // defined in the device code
void release_nfa(const ridfa_program *prog);      // ridfa_nfa.cu

// Device buffers supplied by the caller of launch_with_buffers: the automaton's tables and every
// piece of scratch the reach and join kernels use.  Nothing is allocated by the launch.
struct PreparedBuffers {
    const uint16_t *trans;
    const uint8_t *classmap;
    const uint32_t *final_bits;
    const uint32_t *ifmask;
    const uint16_t *slot_state;
    uint16_t *maps;        // [c][k]
    uint32_t *dinfo;       // [c]
    uint32_t *partials;    // [kMaxJoinBlocks][33]
    uint32_t *ticket;      // zero before the launch
    uint32_t *status;      // zero before the launch
    uint8_t *accept;
};
// Host helpers of the device code (ridfa_device.cu), shared with the batched path.
int cuda_fail(cudaError_t e);
int upload(const HostAutomaton &H, DeviceAutomaton &D, int dev);
const DeviceAutomaton *device_copy(const ridfa_program *P, bool dfa, int dev, int *err);
int smem_optin_limit();
// The space of one join scan, taken from the program (or made) and given back, so that prog->mu need not be
// held while the scan runs: scans that overlap have one each, of which the program keeps one a device.
// Callers of take and give hold prog->mu; grow makes room for `bytes` of working space.
int scan_take(const ridfa_program *prog, int dev, ScanSpace *out);
int scan_grow(ScanSpace *sp, size_t bytes);
void scan_give(const ridfa_program *prog, int dev, const ScanSpace &sp);
// Raise a kernel's dynamic shared-memory cap on the current device to at least `bytes`.  The cap
// is never lowered, so a launch sized by another thread (or an earlier plan) stays valid.
cudaError_t ensure_smem_cap(const void *kern, size_t bytes);

constexpr uint32_t kMaxJoinBlocks = 1024;
constexpr uint32_t kPartialWords = 33;

// Enqueue the reach and join kernels of the RID path (automatic tuning) on `stream`, on buffers
// that are already resident.  Returns a RIDFA_* status; performs no allocation.
int launch_with_buffers(const HostAutomaton &H, const PreparedBuffers &B, const uint8_t *d_text,
                        uint64_t len, uint32_t n_chunks, void *stream);
}

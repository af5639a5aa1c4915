// Set kernels: automata whose runs stay apart (the codon RE's three reading frames), over an alphabet
// of at most four bytes, a chunk per lane from its first byte to its last.
//
// The lane walks the first bytes of its chunk through the graph of functions on the interface slots
// (HostSet) and takes up the distinct runs it finds there, fewer than 16; from then on every byte is
// stepped once for all of them: the column of four bytes comes from arithmetic on their bit fields, and
// each run pays one lookup per four bytes into a table of one copy that fills the SM's shared memory
// (no staging: text comes by 32-byte loads of each lane's own chunk, the next 64 bytes under way; one
// 32-byte load ahead hid too little, 558 -> 586 us at 65,536 chunks of 1 GiB and 566 -> 768 us at
// 77,824, whose chunks begin between blocks).  Every 256 bytes the lane's runs are compacted and the
// warp's loop respecialised to its largest count.
// Bound by the table's bank conflicts, about 3.1 wavefronts a gather (the shared memory pipe is 78 %
// busy).  The general kernel spends 1 + M/2 lookups per byte on M runs, and a warp's time on its chunks'
// first 16 bytes one after another: 1 GiB of codon text in 65,536 chunks 797 -> 559 us, in 1,048,576
// chunks 2863 -> 1334 us with the join, 128 MiB in 65,536 chunks 226 -> 127 us.
//
// The join works on the lane's places: chunk i's function is block of the slot -> place of the block's
// run -> the place's end state, and the transfer from a place of chunk i - 1 that ended in y to the
// places of chunk i comes from the blocks that if_min({y}) meets.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "ridfa_set.h"
#include "ridfa_stream.cuh"

namespace ridfa {
namespace {

constexpr int kSetBlock = 512;
constexpr int kHalf = kSetRuns / 2;

struct SetArgs {
    const uint8_t *text;
    uint64_t len, q, frac;        // chunk i begins at i * q + (i * frac >> 64)
    uint32_t c, depth, spc, back_depth;
    uint64_t pieces;              // c * spc; pieces of a chunk are equal up to 64 bytes
    const uint16_t *next, *images, *back_next, *back_images;
    const uint32_t *leaf;
    uint16_t *ends;               // [pieces][kSetRuns]: distinct end states, dead beyond them
    uint64_t *reps;               // [pieces]: place of each run of the graph's leaf (4 bits; 15: dead)
    uint16_t *entry;              // [pieces][kSetRuns]: states a later piece's runs begin in
    uint32_t *pids;               // [c]: the leaf's partition
    const StreamBatchText *texts; // a batch's texts (null: one text), every piece of them a chunk
    const uint32_t *bases;        // their first pieces
    uint32_t n_texts;
    StreamTables t;
};

__device__ __forceinline__ uint64_t set_chunk_at(const SetArgs &p, uint32_t i) { return i * p.q + __umul64hi(i, p.frac); }

// Drop dead runs and runs in the same state as an earlier one of the places [0, N), pack the others
// to the front, and follow them in `rep` (4 bits per original run: its place, 15 once dead).  As
// compact_runs, by select networks only.
template <int N>
__device__ __forceinline__ uint32_t compact_set(uint32_t (&s)[kSetRuns], uint64_t &rep, uint32_t dead) {
    uint64_t place = 0;
    uint32_t cnt = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        uint32_t at = 15;
        if (s[j] != dead) {
#pragma unroll
            for (int i = 0; i < j; ++i)
                if (at == 15 && s[i] == s[j]) at = static_cast<uint32_t>(place >> (4 * i)) & 15;
            if (at == 15) at = cnt++;
        }
        place |= static_cast<uint64_t>(at) << (4 * j);
    }
    uint32_t t[N];
#pragma unroll
    for (int j = 0; j < N; ++j) t[j] = dead;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const uint32_t at = static_cast<uint32_t>(place >> (4 * j)) & 15;
#pragma unroll
        for (int i = 0; i <= j; ++i)
            if (at == static_cast<uint32_t>(i)) t[i] = s[j];
    }
#pragma unroll
    for (int j = 0; j < N; ++j) s[j] = t[j];
    uint64_t nrep = 0;
#pragma unroll
    for (int g = 0; g < static_cast<int>(kSetRuns); ++g) {
        const uint32_t r = static_cast<uint32_t>(rep >> (4 * g)) & 15;
        nrep |= (r == 15 ? 15ull : (place >> (4 * r)) & 15) << (4 * g);
    }
    rep = nrep;
    return cnt;
}

// One word of text for the first m places (m is the same in the whole warp).
template <int G>
__device__ __forceinline__ void set_word(const StreamTables &p, uint32_t lt, uint32_t w, uint32_t (&s)[kSetRuns], uint32_t m_runs) {
    const uint32_t f = w >> p.shift;
    const uint32_t m1 = f & 0x01010101u, m2 = (w >> (p.shift + 1)) & p.second;
    const uint32_t m = m1 + 2 * m2;
    const bool bad = (m1 * p.d1 + m2 * p.d2 + (m1 & m2) * p.d12 + p.canon0) != w;
#pragma unroll
    for (int h = 0; h < 4 / G; ++h) {
        const uint32_t col = __umulhi(m * (h ? p.mul_h : p.mul), p.take_bits);
        const uint32_t x = col * p.col_mul + (col & p.part_mask) * p.part_mul + lt;
#pragma unroll
        for (int g = 0; g < static_cast<int>(kSetRuns); ++g)
            if (static_cast<uint32_t>(g) < m_runs) s[g] = lds_u16(s[g] * p.row + x);
    }
    if (bad) {
#pragma unroll
        for (int g = 0; g < static_cast<int>(kSetRuns); ++g) s[g] = p.n;
    }
}

// Places that are stepped without asking whether the lane has so many: those beyond are few lanes', and
// a lookup of the dead state takes its banks as any other does (1 GiB in 4,096 chunks 658 -> 635 us).
constexpr uint32_t kSetAlways = 3;

// Eight words of text for the first M runs of places [B, B + 8), of which the lane has cnt in all.
// Returns whether all bytes were in the alphabet.
template <int G, int M, int B>
__device__ __forceinline__ bool set_block(const StreamTables &p, uint32_t lt, const uint32_t (&w)[8], uint32_t (&s)[kSetRuns], uint32_t cnt) {
    uint32_t bad = 0;
    bool on[M];
#pragma unroll
    for (int g = 0; g < M; ++g) on[g] = B + g < kSetAlways || B + g < cnt;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t f = w[i] >> p.shift;
        const uint32_t m1 = f & 0x01010101u, m2 = (w[i] >> (p.shift + 1)) & p.second;
        const uint32_t m = m1 + 2 * m2;
        bad |= (m1 * p.d1 + m2 * p.d2 + (m1 & m2) * p.d12 + p.canon0) ^ w[i];
#pragma unroll
        for (int h = 0; h < 4 / G; ++h) {
            const uint32_t col = __umulhi(m * (h ? p.mul_h : p.mul), p.take_bits);
            const uint32_t x = col * p.col_mul + (col & p.part_mask) * p.part_mul + lt;
#pragma unroll
            for (int g = 0; g < M; ++g)
                if (on[g]) s[B + g] = lds_u16(s[B + g] * p.row + x);
        }
    }
    return bad == 0;
}

template <int G, int B>
__device__ __forceinline__ bool set_block_m(const StreamTables &p, uint32_t lt, const uint32_t (&w)[8], uint32_t (&s)[kSetRuns], uint32_t cnt, uint32_t M) {
    switch (M) {
        case 1: return set_block<G, 1, B>(p, lt, w, s, cnt);
        case 2: return set_block<G, 2, B>(p, lt, w, s, cnt);
        case 3: return set_block<G, 3, B>(p, lt, w, s, cnt);
        case 4: return set_block<G, 4, B>(p, lt, w, s, cnt);
        case 5: return set_block<G, 5, B>(p, lt, w, s, cnt);
        case 6: return set_block<G, 6, B>(p, lt, w, s, cnt);
        case 7: return set_block<G, 7, B>(p, lt, w, s, cnt);
        default: return set_block<G, 8, B>(p, lt, w, s, cnt);
    }
}

// Byte i of 32.
__device__ __forceinline__ uint32_t byte_of(const uint32_t (&w)[8], uint32_t i) {
    uint32_t v = w[0];
#pragma unroll
    for (int k = 1; k < 8; ++k)
        if (i >> 2 == static_cast<uint32_t>(k)) v = w[k];
    return v >> (8 * (i & 3)) & 0xFF;
}

template <int G>
__global__ void __launch_bounds__(kSetBlock, 1) rid_set_kernel(const __grid_constant__ SetArgs p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t base = smem_addr(smem);
    load_tables<Steps<kStreamField, G, 2, 2>>(p.t, smem);        // (the walk table is the one-byte table)
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, dead = p.t.n;
    const uint32_t lt = base + p.t.off_table + (lane & (p.t.copies - 1)) * 4;
    const uint32_t cls = base + p.t.off_cls, one = base + p.t.off_walk;
    const uint64_t t0 = reinterpret_cast<uint64_t>(p.text);
    for (uint64_t task = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; task * 32 < p.pieces; task += gridDim.x * (kSetBlock / 32)) {
        const uint64_t pc = task * 32 + lane;
        const bool have = pc < p.pieces;
        uint32_t ch = static_cast<uint32_t>(pc), j = 0;
        uint64_t pos = t0, end = t0;
        if (have && p.texts) {
            uint32_t lo = 0, hi = p.n_texts - 1;             // the last text that begins at pc or before
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) / 2;
                if (__ldg(p.bases + mid) <= ch) lo = mid;
                else hi = mid - 1;
            }
            const StreamBatchText td = p.texts[lo];
            const uint32_t t = ch - td.base;
            const uint64_t s0 = reinterpret_cast<uint64_t>(td.text);
            pos = t ? (s0 + (t * td.step >> 16)) & ~63ull : s0;
            end = t + 1 < td.pieces ? (s0 + ((t + 1) * td.step >> 16)) & ~63ull : s0 + td.len;
        } else if (have) {
            if (p.spc > 1) {
                ch = static_cast<uint32_t>(pc / p.spc);
                j = static_cast<uint32_t>(pc - static_cast<uint64_t>(ch) * p.spc);
            }
            pos = t0 + set_chunk_at(p, ch);
            end = t0 + set_chunk_at(p, ch + 1);
            if (p.spc > 1) {
                // (cuts on 64-byte boundaries of the text: no ragged ends but the chunk's)
                const uint64_t s0 = pos, per = (end - s0) / p.spc, rem = (end - s0) - per * p.spc;
                if (j) pos = (s0 + j * per + min(static_cast<uint64_t>(j), rem)) & ~63ull;
                if (j + 1 < p.spc) end = (s0 + (j + 1) * per + min(static_cast<uint64_t>(j + 1), rem)) & ~63ull;
            }
        }
        // ---- the first bytes through the graph (chunks are longer than its depth); for a later piece,
        // the bytes before it, from all states (pieces are longer than back_depth)
        uint32_t leaf = 0;
        uint32_t before[8];                      // the 32 bytes before a later piece
        uint32_t taken = 32;
        if (j) {
            load32(reinterpret_cast<const uint8_t *>(pos - 32), before);
            uint32_t node = 0;
            taken = 32 - p.back_depth;
            for (; taken < 32; ++taken) {
                const uint32_t e = __ldg(p.back_next + node * p.t.C + lds_u8(cls + byte_of(before, taken)));
                node = e;
                if (e & kLeafBit) break;
            }
            ++taken;
            leaf = node & kLeafBit ? node & 0x7FFF : 0;      // (always a leaf: back_depth is the longest way to one)
        } else if (have) {
            uint32_t node = 0;
            for (uint32_t d = 0; d < p.depth; ++d) {
                const uint32_t e = __ldg(p.next + node * p.t.C + lds_u8(cls + __ldg(reinterpret_cast<const uint8_t *>(pos++))));
                node = e;
                if (e & kLeafBit) break;
            }
            leaf = node & 0x7FFF;
        }
        const uint32_t pid = j ? 0u : __ldg(p.leaf + 2 * leaf);
        const uint16_t *img = j ? p.back_images + leaf * kSetRuns : p.images + __ldg(p.leaf + 2 * leaf + 1);
        uint32_t s[kSetRuns];
        uint64_t rep = ~0ull;
        uint32_t cnt = 0;
#pragma unroll
        for (int g = 0; g < static_cast<int>(kSetRuns); ++g) {
            s[g] = __ldg(img + g);
            if (s[g] != dead) {
                rep = (rep & ~(15ull << (4 * g))) | static_cast<uint64_t>(g) << (4 * g);
                ++cnt;
            }
        }
        // ---- one-byte steps for all runs up to a 64-byte boundary
        const uint32_t most = __reduce_max_sync(kFull, cnt);
        auto step_byte = [&](uint32_t m, uint32_t byte) {
            const uint32_t c = lds_u8(cls + byte);
#pragma unroll
            for (int g = 0; g < static_cast<int>(kSetRuns); ++g)
                if (static_cast<uint32_t>(g) < m) s[g] = lds_u16(one + 2 * (s[g] * p.t.C + c));
        };
        auto step_all = [&](uint32_t m) { step_byte(m, __ldg(reinterpret_cast<const uint8_t *>(pos++))); };
        auto store = [&](uint16_t *to) {
            uint32_t w[kHalf];
#pragma unroll
            for (int g = 0; g < kHalf; ++g) w[g] = s[2 * g] | s[2 * g + 1] << 16;
            uint4 *out = reinterpret_cast<uint4 *>(to + pc * kSetRuns);
            out[0] = make_uint4(w[0], w[1], w[2], w[3]);
            out[1] = make_uint4(w[4], w[5], w[6], w[7]);
        };
        if (j) {
            for (; taken < 32; ++taken) step_byte(most, byte_of(before, taken));
            store(p.entry);                      // (states may repeat: those runs end in one place)
        }
        // (by words once those are aligned: a lookup a run for four bytes)
        while (cnt && pos < end && (pos & 3)) step_all(most);
        while (cnt && pos + 4 <= end && (pos & 63)) {
            set_word<G>(p.t, lt, __ldg(reinterpret_cast<const uint32_t *>(pos)), s, most);
            pos += 4;
        }
        cnt = compact_set<kSetRuns>(s, rep, dead);
        // ---- blocks of 64 bytes, the next one under way
        uint32_t blocks = cnt && pos < end ? static_cast<uint32_t>((end - pos) >> 6) : 0;
        const uint32_t rounds = __reduce_max_sync(kFull, blocks);
        uint32_t M = __reduce_max_sync(kFull, cnt);
        uint32_t a[8], b[8], na[8], nb[8];
        if (blocks) {
            load32(reinterpret_cast<const uint8_t *>(pos), a);
            load32(reinterpret_cast<const uint8_t *>(pos + 32), b);
        }
        for (uint32_t r = 0; r < rounds; ++r) {
            if (r + 1 < blocks) {
                load32(reinterpret_cast<const uint8_t *>(pos + 64), na);
                load32(reinterpret_cast<const uint8_t *>(pos + 96), nb);
            }
            if (r < blocks) {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    bool ok = set_block_m<G, 0>(p.t, lt, a, s, cnt, min(M, 8u));
                    if (M > kHalf) ok = set_block_m<G, kHalf>(p.t, lt, a, s, cnt, M - kHalf);
                    if (!ok) {
#pragma unroll
                        for (int g = 0; g < static_cast<int>(kSetRuns); ++g) s[g] = dead;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) a[i] = b[i];
                }
                pos += 64;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    a[i] = na[i];
                    b[i] = nb[i];
                }
            }
            if (r < 3 || (r & 3) == 3) {         // (the most runs die in the first bytes)
                // (M is the most runs of the lanes that had a block: a lane that ended its own earlier may
                // hold more, beyond the places a narrow compaction looks at, and waits for the one at the end)
                if (r < blocks) {
                    if (M > kHalf) cnt = compact_set<kSetRuns>(s, rep, dead);
                    else cnt = compact_set<kHalf>(s, rep, dead);
                }
                M = __reduce_max_sync(kFull, r + 1 < blocks ? cnt : 0u);
                if (M == 0) break;
            }
        }
        // ---- ragged end
        uint32_t used = 0;                       // places up to the last live run
#pragma unroll
        for (int g = 0; g < static_cast<int>(kSetRuns); ++g)
            if (s[g] != dead) used = g + 1;
        M = __reduce_max_sync(kFull, used);
        while (used && !(pos & 3) && pos + 4 <= end) {
            set_word<G>(p.t, lt, __ldg(reinterpret_cast<const uint32_t *>(pos)), s, M);
            pos += 4;
        }
        while (used && pos < end) step_all(M);
        compact_set<kSetRuns>(s, rep, dead);
        if (!have) continue;
        store(p.ends);
        p.reps[pc] = rep;
        if (j == 0) p.pids[ch] = pid;
    }
}

// Up to kComposeSet consecutive pieces of a chunk as one: a half-warp follows the places of the first
// through the others, whose runs it finds by the states they begin in.  Bound by latency: the words of
// four pieces are loaded at a time.
constexpr uint32_t kComposeSet = 32, kComposeOne = 64;       // (up to kComposeOne pieces in one launch)
struct SetComposeArgs {
    uint32_t c, in, out, group, n;                           // pieces a chunk, before and after
    const uint16_t *ends, *entry;
    const uint64_t *reps;
    uint16_t *to_ends, *to_entry;
    uint64_t *to_reps;
};

__global__ void __launch_bounds__(256) rid_set_compose_kernel(const __grid_constant__ SetComposeArgs p) {
    const uint32_t lane = threadIdx.x & 31, x = lane & 15, half = lane & 16;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint64_t all = static_cast<uint64_t>(p.c) * p.out;
    const uint64_t id = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 4;
    const uint64_t mine = min(id, all - 1);
    const uint64_t ch = mine / p.out;
    const uint32_t g0 = static_cast<uint32_t>(mine - ch * p.out) * p.group;
    const uint32_t n_in = min(p.group, p.in - g0);
    const uint64_t at = ch * p.in + g0;
    uint32_t y = __ldg(p.ends + at * kSetRuns + x);
    uint32_t ew[4] = {}, z[4] = {}, ne[4] = {}, nz[4] = {};
    uint64_t rp[4] = {}, nr[4] = {};
    auto fetch = [&](uint32_t j0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j0 + u >= n_in) continue;
            const uint64_t o = at + j0 + u;
            ne[u] = __ldg(reinterpret_cast<const uint32_t *>(p.entry + o * kSetRuns) + (x & 7));
            nz[u] = __ldg(p.ends + o * kSetRuns + x);
            nr[u] = __ldg(reinterpret_cast<const unsigned long long *>(p.reps) + o);
        }
    };
    fetch(1);
    for (uint32_t j0 = 1; j0 < p.group; j0 += 4) {           // (the whole warp takes p.group pieces)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            ew[u] = ne[u];
            z[u] = nz[u];
            rp[u] = nr[u];
        }
        fetch(j0 + 4);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool on = j0 + u < n_in;
            uint32_t place = 15;
#pragma unroll
            for (int g = 0; g < kHalf; ++g) {
                const uint32_t w = __shfl_sync(kFull, ew[u], half + g);
                if (y == (w & 0xFFFFu)) place = static_cast<uint32_t>(rp[u] >> (8 * g)) & 15;
                if (y == w >> 16) place = static_cast<uint32_t>(rp[u] >> (8 * g + 4)) & 15;
            }
            if (y >= p.n) place = 15;
            const uint32_t to = __shfl_sync(kFull, z[u], half + place);     // (place 15 stays dead)
            if (on) y = to;
        }
    }
    if (id >= all) return;
    p.to_ends[mine * kSetRuns + x] = static_cast<uint16_t>(y);
    if (p.out > 1) p.to_entry[mine * kSetRuns + x] = __ldg(p.entry + at * kSetRuns + x);
    if (x == 0) p.to_reps[mine] = __ldg(reinterpret_cast<const unsigned long long *>(p.reps) + at);
}

// ------------------------------------------------------------------------------- join
struct SetJoinArgs {
    uint32_t c, k, kw, n, q0_slot, per_warp;
    const uint16_t *ends;
    const uint64_t *reps;
    const uint32_t *pids, *block_mask, *ifmask, *final_bits;
    const uint8_t *part;
    uint16_t *maps;               // null: not asked for
    uint32_t *partials, *ticket, *status;
    uint8_t *accept, *h_accept;
    uint32_t *h_status;
    const StreamBatchText *texts; // a batch's texts, a block each (null: one text)
};

constexpr uint32_t kSetJoinWarps = 16;
constexpr uint32_t kSetTile = 16;                // chunks a warp stages at a time

// rows <- rows · M in each half-warp: lane h * 16 + x has row x of both (at most 15 places).  `from`
// is added to the lane M's row z is read from (z + from): the own half's, or a fixed half's.
__device__ __forceinline__ uint32_t set_times(uint32_t row, uint32_t m, uint32_t from) {
    if (__all_sync(kFull, m == 1u << (threadIdx.x & 15))) return row;       // (identities would be the longest)
    const uint32_t any = __ballot_sync(kFull, m != 0);
    uint32_t out = 0;
    for (uint32_t nz = (any | any >> 16) & 0xFFFFu; nz; nz &= nz - 1) {
        const uint32_t z = __ffs(nz) - 1, mz = __shfl_sync(kFull, m, z + from);
        if ((row >> z) & 1) out |= mz;
    }
    return out;
}

// Chunk maps, and the product over all boundaries.  A warp takes per_warp consecutive chunks by tiles
// of 16 that it stages in shared memory, a tile ahead in registers; each half-warp forms the product of
// eight boundaries, a place of the chunk before per lane, so that a boundary costs a quarter of the
// loads and half of the serial steps that a warp per boundary takes (46 -> 26 us at 65,536 chunks, 409
// -> 232 us at 1,048,576; the general join took 65 and about 500 us).  Bound by latency: tables through
// L1 and the products' shuffles.  A block takes the product of its warps', the last block that of all;
// of a batch's texts each has one block.
__global__ void __launch_bounds__(32 * kSetJoinWarps) rid_set_join_kernel(const __grid_constant__ SetJoinArgs a) {
    __shared__ __align__(16) uint16_t s_end[kSetJoinWarps][kSetTile + 1][kSetRuns];  // row 0: the chunk before
    __shared__ uint64_t s_rep[kSetJoinWarps][kSetTile];
    __shared__ uint32_t s_pid[kSetJoinWarps][kSetTile];
    __shared__ uint32_t s_prod[2 * kSetJoinWarps][kSetRuns];
    __shared__ uint32_t s_last;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, x = lane & 15, half = lane & 16;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    SetJoinArgs p = a;
    uint32_t first_block = blockIdx.x;
    if (a.texts) {
        const StreamBatchText td = a.texts[blockIdx.x];
        p.c = td.pieces;
        p.ends += static_cast<uint64_t>(td.base) * kSetRuns;
        p.reps += td.base;
        p.pids += td.base;
        p.accept += td.item;
        p.per_warp = ((td.pieces + kSetJoinWarps - 1) / kSetJoinWarps + kSetTile - 1) / kSetTile * kSetTile;
        first_block = 0;
    }
    const uint64_t i0 = (static_cast<uint64_t>(first_block) * kSetJoinWarps + warp) * p.per_warp;
    const uint64_t i1 = min(static_cast<uint64_t>(p.c), i0 + p.per_warp);
    uint32_t row = 1u << x;
    uint4 e{};
    uint64_t rep = 0;
    uint32_t pid = 0;
    // lane l: half a row of ends; the first 16 lanes: a chunk's places and partition
    auto fetch = [&](uint64_t i) {
        if (i + (lane >> 1) < i1) e = __ldg(reinterpret_cast<const uint4 *>(p.ends + i * kSetRuns) + lane);
        if (lane < kSetTile && i + lane < i1) {
            rep = __ldg(reinterpret_cast<const unsigned long long *>(p.reps) + i + lane);
            pid = __ldg(p.pids + i + lane);
        }
    };
    if (i0 < i1) {
        if (lane < kSetRuns) s_end[warp][kSetTile][lane] = i0 ? __ldg(p.ends + (i0 - 1) * kSetRuns + lane) : static_cast<uint16_t>(p.n);
        fetch(i0);
    }
    for (uint64_t i = i0; i < i1; i += kSetTile) {
        const uint32_t cnt = static_cast<uint32_t>(min(static_cast<uint64_t>(kSetTile), i1 - i));
        if (lane < kSetRuns) s_end[warp][0][lane] = s_end[warp][kSetTile][lane];
        __syncwarp();
        reinterpret_cast<uint4 *>(s_end[warp][1])[lane] = e;
        if (lane < kSetTile) {
            s_rep[warp][lane] = rep;
            s_pid[warp][lane] = pid;
        }
        __syncwarp();
        if (i + kSetTile < i1) fetch(i + kSetTile);
        // boundaries before chunks i + u, i + 8 + u
        uint32_t prod = 1u << x;
#pragma unroll 2
        for (uint32_t u = 0; u < 8; ++u) {
            const uint32_t at = (half >> 1) + u;
            uint32_t m = 1u << x;                            // (no boundary before chunk 0 or beyond the end)
            if (at < cnt && i + at != 0) {
                m = 0;
                const uint32_t y = s_end[warp][at][x], id = s_pid[warp][at];
                const uint64_t rp = s_rep[warp][at];
                for (uint32_t w = 0; w < p.kw; ++w) {
                    const uint32_t in = y < p.n ? __ldg(p.ifmask + static_cast<uint64_t>(y) * p.kw + w) : 0u;
                    const uint4 *bm = reinterpret_cast<const uint4 *>(p.block_mask + (static_cast<uint64_t>(id) * p.kw + w) * kSetRuns);
#pragma unroll
                    for (int q = 0; q < static_cast<int>(kSetRuns) / 4; ++q) {
                        const uint4 v = __ldg(bm + q);
                        const uint32_t b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            if (in & b[t]) m |= 1u << (static_cast<uint32_t>(rp >> (4 * (4 * q + t))) & 15);
                    }
                }
                m &= 0x7FFFu;                                // (place 15: the run died)
            }
            prod = set_times(prod, m, half);
        }
        row = set_times(row, prod, 0);
        row = set_times(row, prod, 16);
        if (p.maps) {
            for (uint32_t j = lane; j < cnt * p.k; j += 32) {
                const uint32_t u = j / p.k, a = j - u * p.k;
                const uint32_t b = __ldg(p.part + static_cast<uint64_t>(s_pid[warp][u]) * p.k + a);
                const uint32_t at = b == 0xFF ? 15u : static_cast<uint32_t>(s_rep[warp][u] >> (4 * (b & 15))) & 15;
                const uint32_t v = s_end[warp][u + 1][at];   // (place 15 stays dead)
                p.maps[i * p.k + j] = static_cast<uint16_t>(v >= p.n ? kUndef : v);
            }
        }
        __syncwarp();
    }
    if (lane < kSetRuns) s_prod[warp][lane] = row;
    __syncthreads();
    auto accepts = [&](uint32_t products) {                  // (one warp)
        // the place of q0's slot in chunk 0, through all boundaries, to a final state
        const uint32_t q0 = __ldg(p.part + static_cast<uint64_t>(__ldg(p.pids)) * p.k + p.q0_slot);
        const uint32_t at = q0 == 0xFF ? 15u : static_cast<uint32_t>(__ldg(reinterpret_cast<const unsigned long long *>(p.reps)) >> (4 * q0)) & 15;
        uint32_t v = at == 15 ? 0u : 1u << at;
        for (uint32_t w = 0; w < products; ++w) v = __reduce_or_sync(kFull, (v >> x) & 1 ? s_prod[w][x] : 0u);
        const uint32_t z = lane < kSetRuns ? __ldg(p.ends + static_cast<uint64_t>(p.c - 1) * kSetRuns + lane) : p.n;
        const bool fin = ((v >> x) & 1) && z < p.n && ((__ldg(p.final_bits + (z >> 5)) >> (z & 31)) & 1);
        return __any_sync(kFull, fin) ? 1u : 0u;
    };
    if (p.texts) {
        if (warp) return;
        const uint32_t acc = accepts(kSetJoinWarps);
        if (lane == 0) *p.accept = static_cast<uint8_t>(acc);
        return;
    }
    if (warp == 0) {
        // the upper half its eight warps, then both
        row = 1u << x;
        for (uint32_t w = 0; w < kSetJoinWarps / 2; ++w) row = set_times(row, s_prod[(half ? kSetJoinWarps / 2 : 0) + w][x], half);
        const uint32_t all = set_times(row, row, 16);        // (lower half: first · second)
        if (lane < kSetRuns) p.partials[static_cast<uint64_t>(blockIdx.x) * kSetRuns + lane] = all;
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            s_last = atomicAdd(p.ticket, 1) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // ---- last block: each half-warp its share of the blocks' products
    const uint32_t per = (gridDim.x + 2 * kSetJoinWarps - 1) / (2 * kSetJoinWarps), hw = 2 * warp + (half >> 4);
    const uint32_t b0 = min(gridDim.x, hw * per), b1 = min(gridDim.x, b0 + per);
    row = 1u << x;
    for (uint32_t b = 0; b < per; b += 4) {
        uint32_t m[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) m[u] = b0 + b + u < b1 ? __ldcg(p.partials + static_cast<uint64_t>(b0 + b + u) * kSetRuns + x) : 1u << x;
#pragma unroll
        for (int u = 0; u < 4; ++u) row = set_times(row, m[u], half);
    }
    s_prod[hw][x] = row;
    __syncthreads();
    if (warp) return;
    const uint32_t acc = accepts(2 * kSetJoinWarps);
    if (lane == 0) {
        *p.accept = static_cast<uint8_t>(acc);
        *p.status = 0;
        *p.ticket = 0;
        if (p.h_accept) {
            *p.h_accept = static_cast<uint8_t>(acc);
            *p.h_status = 0;
        }
    }
}

// Whole tiles, for a few blocks on each of about 150 SMs: 256 blocks' products are short work for the
// last block, and a warp's chain is short up to 65,536 chunks.
uint32_t join_per_warp(uint32_t c) { return std::max<uint32_t>(kSetTile, (c / 8192 + kSetTile - 1) / kSetTile * kSetTile); }

uint32_t set_join_blocks(uint32_t c) {
    const uint64_t per = static_cast<uint64_t>(join_per_warp(c)) * kSetJoinWarps;
    return static_cast<uint32_t>((c + per - 1) / per);
}

}  // namespace

namespace {
// The parts of the kernels' arguments that depend on the automaton alone; returns the shared memory.
size_t set_args(const HostAutomaton &H, const DeviceAutomaton &D, SetArgs &a, SetJoinArgs &j) {
    const HostStream &T = H.set.table;
    a.depth = H.set.depth;
    a.back_depth = H.set.back_depth;
    a.next = D.set_next;
    a.images = D.set_images;
    a.back_next = D.set_back_next;
    a.back_images = D.set_back_images;
    a.leaf = D.set_leaf;
    a.t = stream_field_tables(T);
    a.t.walk = D.trans;
    a.t.classmap = D.classmap;
    a.t.words = D.set_words;
    a.t.n = H.n_states;
    a.t.C = H.n_classes;
    a.t.n_walk = static_cast<uint32_t>(H.trans.size() + 1) & ~1u;      // (whole words; the upload is padded)
    const uint32_t off = a.t.n_words * 4 * T.copies;
    a.t.off_table = 0;
    a.t.off_cls = (off + 15) & ~15u;
    a.t.off_walk = a.t.off_cls + 256;
    j.k = H.k;
    j.kw = H.kw;
    j.n = H.n_states;
    j.q0_slot = H.q0_slot;
    j.block_mask = D.set_block_mask;
    j.ifmask = D.ifmask;
    j.final_bits = D.final_bits;
    j.part = D.set_part;
    return set_rest_bytes(H) + static_cast<size_t>(off);
}

cudaError_t set_reach(const HostAutomaton &H, const SetArgs &a, uint32_t grid, size_t smem, cudaStream_t st) {
    auto kern = H.set.table.group == 4 ? rid_set_kernel<4> : rid_set_kernel<2>;
    cudaError_t e = ensure_smem_cap(reinterpret_cast<const void *>(kern), smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, kSetBlock, smem, st>>>(a);       // (all warps load the table)
    return cudaGetLastError();
}
}  // namespace

uint32_t set_pieces(const HostAutomaton &H, uint64_t len, uint32_t c, int sms) {
    if (!H.set.ok || c > (1u << 26) || len > (1ull << 40) || len / c < 32) return 0;
    // (32 bytes: a chunk is no shorter than the graph is deep.  5 KB in 80 chunks: 186 us in the
    // general kernels, 55 us here; 64 MiB in 1,000,000 chunks 2,086 and 607 us.)
    const uint64_t lanes = static_cast<uint64_t>(sms) * kSetBlock;
    // Without the sets of what a piece is entered with, a chunk is one lane's work: at least half of the
    // lanes have to have one (at a quarter the general path was as fast).
    if (!H.set.back_depth) return static_cast<uint64_t>(c) * 2 > lanes ? 1 : 0;
    // As many pieces as the lanes take at once, of 256 bytes or more: a second round costs its pieces'
    // first bytes, with the most runs, again (1 GiB in 20,000 chunks: 721 us in 3 pieces each, 883 in 7;
    // in 40,000 chunks 782 in one, 978 in 3), and a shorter piece is mostly such bytes.
    return static_cast<uint32_t>(std::max<uint64_t>(1, std::min<uint64_t>(len / c / 256, lanes / c)));
}

size_t set_scratch(uint32_t c, uint32_t spc) {
    size_t n = 0;
    for (uint64_t s = spc; s > 1; s = (s + kComposeSet - 1) / kComposeSet) n += c * s;       // each level's pieces
    return (n + c) * (2 * kSetRuns * 2 + 8) + static_cast<size_t>(c) * 4 + static_cast<size_t>(set_join_blocks(c)) * kSetRuns * 4 + 64 * 256;
}

namespace {
uint32_t set_grid(uint64_t pieces, int sms) { return static_cast<uint32_t>(std::min<uint64_t>(sms, (pieces + 31) / 32)); }
}  // namespace

ridfa_kernel_report set_report(const HostAutomaton &H, uint32_t c, uint32_t spc, int sms) {
    const HostStream &T = H.set.table;
    return {RIDFA_KERNEL_SET, T.group, 0, T.entry, T.copies, spc, kSetBlock, set_grid(static_cast<uint64_t>(c) * spc, sms)};
}

cudaError_t set_launch(const SetCall &C, int sms, cudaStream_t st) {
    const HostAutomaton &H = *C.H;
    const DeviceAutomaton &D = *C.D;
    const uint64_t pieces = static_cast<uint64_t>(C.c) * C.spc;
    uint8_t *next = C.scratch;
    auto take = [&](size_t bytes) {
        uint8_t *r = next;
        next += (bytes + 255) & ~static_cast<size_t>(255);
        return r;
    };
    auto u16 = [&](uint64_t n) { return reinterpret_cast<uint16_t *>(take(n * kSetRuns * 2)); };
    auto u64 = [&](uint64_t n) { return reinterpret_cast<uint64_t *>(take(n * 8)); };
    uint32_t *pids = reinterpret_cast<uint32_t *>(take(C.c * 4ull));
    uint32_t *partials = reinterpret_cast<uint32_t *>(take(static_cast<size_t>(set_join_blocks(C.c)) * kSetRuns * 4));
    SetArgs a{};
    a.text = C.text;
    a.len = C.len;
    a.q = C.len / C.c;
    const uint64_t rem = C.len % C.c;
    a.frac = rem ? static_cast<uint64_t>((static_cast<unsigned __int128>(rem) << 64) / C.c) + 1 : 0;   // (as the stream kernels)
    a.c = C.c;
    a.spc = C.spc;
    a.pieces = pieces;
    a.ends = u16(pieces);
    a.reps = u64(pieces);
    a.entry = C.spc > 1 ? u16(pieces) : nullptr;
    a.pids = pids;
    SetJoinArgs j{};
    const size_t smem = set_args(H, D, a, j);
    cudaError_t e = set_reach(H, a, set_grid(pieces, sms), smem, st);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    SetComposeArgs m{};
    m.c = C.c;
    m.n = H.n_states;
    m.ends = a.ends;
    m.entry = a.entry;
    m.reps = a.reps;
    for (m.in = C.spc; m.in > 1; m.in = m.out) {
        m.group = m.in <= kComposeOne ? m.in : kComposeSet;
        m.out = (m.in + m.group - 1) / m.group;
        const uint64_t n = static_cast<uint64_t>(C.c) * m.out;
        m.to_ends = u16(n);
        m.to_reps = u64(n);
        m.to_entry = m.out > 1 ? u16(n) : nullptr;
        cfg.gridDim = dim3(static_cast<unsigned>((n + 15) / 16));
        cfg.blockDim = dim3(256);
        e = cudaLaunchKernelEx(&cfg, rid_set_compose_kernel, m);
        if (e != cudaSuccess) return e;
        m.ends = m.to_ends;
        m.entry = m.to_entry;
        m.reps = m.to_reps;
    }
    if (C.between) {
        e = cudaEventRecord(C.between, st);
        if (e != cudaSuccess) return e;
    }
    j.c = C.c;
    j.per_warp = join_per_warp(C.c);
    j.ends = m.ends;
    j.reps = m.reps;
    j.pids = pids;
    j.maps = C.maps;
    j.partials = partials;
    j.ticket = C.ticket;
    j.status = C.status;
    j.accept = C.accept;
    j.h_accept = C.h_accept;
    j.h_status = C.h_status;
    cfg.gridDim = dim3(set_join_blocks(C.c));
    cfg.blockDim = dim3(32 * kSetJoinWarps);
    cfg.numAttrs = C.between ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, rid_set_join_kernel, j);
}

// (measured on the batch of 2,000 texts against 16 REs: 4 bytes a clock of an SM, a two-byte stream
// table 10 to 12)
double set_batch_weight(const HostAutomaton &H) { return H.set.table.group == 4 ? 2.5 : 4.0; }

constexpr uint64_t kSetBatchPieces = 4096;

void plan_set_batch(SetBatchPlan &P, const StreamBatchSource &src, uint32_t sms) {
    P = SetBatchPlan{};
    P.H = src.H;
    P.D = src.D;
    uint64_t bytes = 0;
    for (const auto &it : src.items) bytes += it.len;
    // one round of pieces for the SMs' lanes, none longer than the others
    const uint64_t piece = std::max<uint64_t>(kSetBatchPiece, bytes / (static_cast<uint64_t>(sms) * kSetBlock) + 1);
    for (const auto &it : src.items) {
        StreamBatchText t{it.text, it.len, 0, P.pieces, 0, 0, it.item};
        // (one block joins a text's pieces, 23 ns each: longer ones for a text of very many, 64 MB in two
        // texts 1,002 us without the bound)
        t.pieces = static_cast<uint32_t>(std::min<uint64_t>(kSetBatchPieces, (it.len + piece - 1) / piece));
        t.step = static_cast<uint64_t>((static_cast<unsigned __int128>(it.len) << 16) / t.pieces);
        P.pieces += t.pieces;
        P.texts.push_back(t);
        P.bases.push_back(t.base);
    }
    P.grid = std::min<uint32_t>(sms, (P.pieces + 31) / 32);
    P.o_bases = (P.texts.size() * sizeof(StreamBatchText) + 255) & ~static_cast<size_t>(255);
    P.image_bytes = P.o_bases + P.bases.size() * 4;
    P.result_bytes = static_cast<size_t>(P.pieces) * kSetBatchResult;
}

void set_batch_image(const SetBatchPlan &P, uint8_t *img) {
    std::memcpy(img, P.texts.data(), P.texts.size() * sizeof(StreamBatchText));
    std::memcpy(img + P.o_bases, P.bases.data(), P.bases.size() * 4);
}

cudaError_t set_batch_launch(const SetBatchPlan &P, const uint8_t *dev, uint8_t *res, uint8_t *d_accept, cudaStream_t st) {
    SetArgs a{};
    SetJoinArgs j{};
    const size_t smem = set_args(*P.H, *P.D, a, j);
    a.texts = reinterpret_cast<const StreamBatchText *>(dev);
    a.bases = reinterpret_cast<const uint32_t *>(dev + P.o_bases);
    a.n_texts = static_cast<uint32_t>(P.texts.size());
    a.spc = 1;
    a.pieces = P.pieces;
    a.ends = reinterpret_cast<uint16_t *>(res);
    a.reps = reinterpret_cast<uint64_t *>(res + static_cast<size_t>(P.pieces) * kSetRuns * 2);
    a.pids = reinterpret_cast<uint32_t *>(a.reps + P.pieces);
    cudaError_t e = set_reach(*P.H, a, P.grid, smem, st);
    if (e != cudaSuccess) return e;
    j.texts = a.texts;
    j.ends = a.ends;
    j.reps = a.reps;
    j.pids = a.pids;
    j.accept = d_accept;
    rid_set_join_kernel<<<a.n_texts, 32 * kSetJoinWarps, 0, st>>>(j);
    return cudaGetLastError();
}

}  // namespace ridfa

// Stream kernels: the reach phase of automata whose runs merge, one lane per chunk (or per piece
// of a chunk) from its first byte to its last.
//
// The merge graph (HostMerge) tells what becomes of the runs from every state at once: the lane
// walks it until one run is left, usually within some ten bytes, and goes on with that run through
// the table of HostStream.  The piece's function is then one word (StreamArgs::res).  Against the
// lockstep speculation of the general reach kernel (a warp stepping every slot's run of one chunk
// after another), nothing here is serial over a warp's chunks and nothing is written per slot; and
// because the graph covers every state, not only the interface slots, a chunk can be cut into any
// number of pieces at no extra lookups.
//
// The join kernel composes a chunk's pieces, writes the chunk maps and evaluates the join.  A
// chunk whose pieces all merged has at most one end state, so a boundary's transfer matrix is one
// bit: does if_min of the previous chunk's end state meet the slots alive in this chunk?
#include <cuda_runtime.h>

#include <algorithm>

#include "ridfa_join.cuh"
#include "ridfa_stream.h"

namespace ridfa {
namespace {

constexpr uint32_t kNoNode = 0xFFFFFFFFu;
constexpr uint32_t kNodeResult = 0x80000000u;   // a piece that ended in an inner node
constexpr uint32_t kGlobal = 0xFFFFFFFFu;       // a ragged-end table left in global memory
constexpr int kStreamBlock = 1024;

struct StreamArgs {
    const uint8_t *text;
    uint64_t len, np, q, r;       // np pieces; q = len / np, r = len % np
    uint32_t *res;                // [np]: kNodeResult | node, or pid << 16 | state
    const uint16_t *trans;
    const uint8_t *classmap;
    const uint16_t *next;
    const uint32_t *leaf, *code, *words;
    uint32_t n, C, inner;
    uint32_t n_words, copies, row;                       // row: bytes per state
    uint32_t shift, mask, mul, sh_w, m_w, sh_q, m_q, canon;   // field codes
    uint32_t off_table, off_trans, off_cls, off_next, off_stage;
};

__device__ __forceinline__ uint64_t piece_begin(const StreamArgs &p, uint64_t i) {
    return i * p.q + (p.r ? i * p.r / p.np : 0);         // floor(i * len / np)
}

// The state of one lane between bytes, and one-byte steps for everything that is not a whole
// granule of a merged run: the graph walk, ragged starts and ends.
struct Walk {
    const uint16_t *trans, *next;
    const uint32_t *leaf;
    const uint8_t *cls;
    uint32_t C;
    uint32_t node, pid, s;
    __device__ __forceinline__ void start() {
        node = 0;
        pid = 0;
        s = 0;
    }
    __device__ __forceinline__ void step(uint32_t b) {
        const uint32_t c = cls[b];
        if (node == kNoNode) {
            s = trans[s * C + c];
            return;
        }
        const uint32_t e = next[node * C + c];
        if (e & kLeafBit) {
            const uint32_t l = __ldg(leaf + (e & 0x7FFF));
            pid = l >> 16;
            s = l & 0xFFFF;
            node = kNoNode;
        } else {
            node = e;
        }
    }
    __device__ __forceinline__ uint32_t result() const {
        return node == kNoNode ? pid << 16 | s : kNodeResult | node;
    }
};

template <int E>
__device__ __forceinline__ uint32_t lds_entry(uint32_t a) {
    return E == 1 ? lds_u8(a) : lds_u16(a);
}

// Table steps of a merged run.  KIND and G (bytes a lookup) as in HostStream, E: bytes per entry.
template <int KIND, int G, int E>
struct Steps {
    static constexpr bool kStaged = KIND != kStreamField;
    uint32_t lc, lt, row;        // this lane's class codes; its copy of the table; bytes per state
    uint32_t shift, mask, mul, sh_w, m_w, sh_q, m_q, canon, dead;
    __device__ __forceinline__ void init(const StreamArgs &p, uint32_t base) {
        const uint32_t lane = threadIdx.x & 31;
        lc = base + lane * 4;
        lt = base + p.off_table + (lane & (p.copies - 1)) * 4;
        row = p.row;
        dead = p.n;
        if (KIND == kStreamField) {
            shift = p.shift; mask = p.mask; mul = p.mul; canon = p.canon;
            sh_w = p.sh_w; m_w = p.m_w; sh_q = p.sh_q; m_q = p.m_q;
        }
    }
    __device__ __forceinline__ uint32_t byte_at(const uint32_t *w, int q) const { return (w[q >> 2] >> (8 * (q & 3))) & 0xFF; }
    // N 32-bit words of text
    template <int N>
    __device__ __forceinline__ uint32_t take(uint32_t s, const uint32_t (&w)[N]) const {
        if constexpr (KIND == kStreamField) {
            // codes: mask the field of all four bytes, gather them with one multiplication (byte 0's
            // code lowest at bit 24), split into word and part of the entry.  A byte that differs
            // from its code's canonical byte is outside the alphabet: the run is dead after it.
            uint32_t bad = 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint32_t m = (w[i] >> shift) & mask;
                const uint32_t y = m | (m >> 4);
                bad |= __byte_perm(canon, 0, __byte_perm(y, 0, 0x4420)) ^ w[i];
                if (G == 4) {
                    const uint32_t g = m * mul;
                    s = lds_entry<E>(s * row + (((g >> sh_w) & m_w) + ((g >> sh_q) & m_q) + lt));
                } else {
                    const uint32_t g = m * mul, h = (m >> 16) * mul;
                    s = lds_entry<E>(s * row + (((g >> sh_w) & m_w) + ((g >> sh_q) & m_q) + lt));
                    s = lds_entry<E>(s * row + (((h >> sh_w) & m_w) + ((h >> sh_q) & m_q) + lt));
                }
            }
            return bad ? dead : s;
        } else if constexpr (KIND == kStreamPair) {
            uint32_t x[2 * N];
#pragma unroll
            for (int i = 0; i < 2 * N; ++i)
                x[i] = lds_u16(lc + (byte_at(w, 2 * i) << 7)) + lds_u16(lc + 2 + (byte_at(w, 2 * i + 1) << 7)) + lt;
#pragma unroll
            for (int i = 0; i < 2 * N; ++i) s = lds_entry<E>(s * row + x[i]);
            return s;
        } else {
            uint32_t x[4 * N];
#pragma unroll
            for (int i = 0; i < 4 * N; ++i) x[i] = lds_u32(lc + (byte_at(w, i) << 7)) + lt;
#pragma unroll
            for (int i = 0; i < 4 * N; ++i) s = lds_entry<E>(s * row + x[i]);
            return s;
        }
    }
};

// Shared-memory tables of a block: class codes (32 lane copies), the main table in its lane copies,
// and the one-byte tables of the ragged ends.
template <class S>
__device__ __forceinline__ void load_tables(const StreamArgs &p, uint8_t *smem, Walk &w) {
    const uint32_t base = smem_addr(smem);
    const uint32_t nt = blockDim.x;
    auto put4 = [&](uint32_t a, uint32_t v) {
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(a), "r"(v) : "memory");
    };
    if (S::kStaged)
        for (uint32_t i = threadIdx.x; i < 256 * 8; i += nt) put4(base + i * 16, __ldg(p.code + (i >> 3)));
    if (p.copies >= 4) {
        const uint32_t lg = __ffs(p.copies) - 3;         // 16-byte stores per word: copies / 4
        for (uint32_t i = threadIdx.x; i < p.n_words << lg; i += nt) put4(base + p.off_table + i * 16, __ldg(p.words + (i >> lg)));
    } else {
        for (uint32_t i = threadIdx.x; i < p.n_words * p.copies; i += nt)
            sts_u32(base + p.off_table + i * 4, __ldg(p.words + i / p.copies));
    }
    w.cls = smem + p.off_cls;
    for (uint32_t i = threadIdx.x; i < 64; i += nt)
        reinterpret_cast<uint32_t *>(smem + p.off_cls)[i] = __ldg(reinterpret_cast<const uint32_t *>(p.classmap) + i);
    w.trans = p.trans;
    if (p.off_trans != kGlobal) {
        uint16_t *t = reinterpret_cast<uint16_t *>(smem + p.off_trans);
        for (uint32_t i = threadIdx.x; i < (p.n + 1) * p.C; i += nt) t[i] = __ldg(p.trans + i);
        w.trans = t;
    }
    w.next = p.next;
    if (p.off_next != kGlobal) {
        uint16_t *t = reinterpret_cast<uint16_t *>(smem + p.off_next);
        for (uint32_t i = threadIdx.x; i < p.inner * p.C; i += nt) t[i] = __ldg(p.next + i);
        w.next = t;
    }
    w.leaf = p.leaf;
    w.C = p.C;
}

// Text through 32-byte loads of each lane's own piece, one block ahead: an L1 line per lane and
// load, so 1.2 LSU cycles per 32 text bytes; worth it where the lookups take less than one.
__device__ __forceinline__ void load32(const uint8_t *a, uint32_t (&w)[8]) {
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(a));
}

// One-byte steps over [pos, end) while the run is not merged or `pos` is not 32-byte aligned (or,
// with `all`, to the end), the text taken in aligned 8-byte loads where they lie inside it.
__device__ __forceinline__ void walk_ragged(Walk &w, uint64_t &pos, uint64_t end, uint64_t t0, uint64_t t1, bool all) {
    while (pos < end && (all || w.node != kNoNode || (pos & 31))) {
        const uint64_t a = pos & ~static_cast<uint64_t>(7);
        uint64_t v;
        uint32_t m = 1;
        if (a >= t0 && a + 8 <= t1) {
            const uint32_t o = static_cast<uint32_t>(pos & 7);
            v = __ldg(reinterpret_cast<const unsigned long long *>(a)) >> (8 * o);
            m = static_cast<uint32_t>(min(static_cast<uint64_t>(8 - o), end - pos));
        } else {
            v = __ldg(reinterpret_cast<const uint8_t *>(pos));
        }
        pos += m;
        for (uint32_t i = 0; i < m; ++i, v >>= 8) w.step(static_cast<uint32_t>(v) & 0xFF);
    }
}

template <class S>
__device__ __forceinline__ void stream_direct(const S &T, Walk &w, uint64_t pos, uint64_t end, uint64_t t0, uint64_t t1) {
    walk_ragged(w, pos, end, t0, t1, false);
    uint32_t blocks = pos < end ? static_cast<uint32_t>((end - pos) >> 5) : 0;
    if (blocks && w.node == kNoNode) {
        uint32_t cur[8], nxt[8];
        load32(reinterpret_cast<const uint8_t *>(pos), cur);
        for (; blocks; --blocks, pos += 32) {
            if (blocks > 1) load32(reinterpret_cast<const uint8_t *>(pos + 32), nxt);
            w.s = T.template take<8>(w.s, cur);
            if (w.s == T.dead) return;
#pragma unroll
            for (int i = 0; i < 8; ++i) cur[i] = nxt[i];
        }
    }
    walk_ragged(w, pos, end, t0, t1, true);
}

// Text staged by the warp: rounds of one 64-byte window per lane, copied with cp.async (L2 to
// shared memory) so that four neighbouring lanes move one window; double-buffered, in the layout of
// coop_unit.  A lane's copies always serve the same four windows, whose places are worked out once
// (offsets from the warp's first window), not passed round by shuffles each time.
template <class S>
__device__ __forceinline__ void stream_staged(const S &T, Walk &w, uint32_t stage, uint64_t pos, uint64_t end, uint64_t t0, uint64_t t1) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t lo = (t0 + 15) & ~static_cast<uint64_t>(15), hi = t1 & ~static_cast<uint64_t>(15);
    // offsets are from the start of the warp's first piece (pieces ascend)
    const uint64_t base = __shfl_sync(kFull, pos, 0) & ~static_cast<uint64_t>(15);
    while (pos < min(end, lo)) w.step(__ldg(reinterpret_cast<const uint8_t *>(pos++)));
    const uint64_t stop64 = min(end, hi);
    const bool have = pos < stop64;
    const uint32_t wrel = have ? static_cast<uint32_t>((pos & ~static_cast<uint64_t>(15)) - base) : 0;
    uint32_t prel = static_cast<uint32_t>(pos - base);
    const uint32_t srel = have ? static_cast<uint32_t>(stop64 - base) : wrel;
    const uint32_t nwin = have ? (srel - wrel + kCoopWin - 1) / kCoopWin : 0;
    const uint32_t rounds = __reduce_max_sync(kFull, nwin);
    const uint32_t g = lane & 3;
    uint32_t src[4], lim[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = u * 8 + (lane >> 2);
        src[u] = __shfl_sync(kFull, wrel, j) + 16 * g;
        lim[u] = __shfl_sync(kFull, srel, j);
    }
    const uint32_t dst = stage + 16 * coop_unit(lane >> 2, g);
    auto issue = [&](uint32_t r) {
        const uint32_t d = dst + (r & 1) * kCoopBufBytes;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (src[u] + kCoopWin * r < lim[u])      // (coop_unit(j + 8, g) is 32 granules on)
                cp_async_16(d + u * 512, reinterpret_cast<const void *>(base + (src[u] + kCoopWin * r)));
        cp_async_commit();
    };
    issue(0);
    const uint32_t sw = (lane >> 1) & 3;
    for (uint32_t r = 0; r < rounds; ++r) {
        if (r + 1 < rounds) issue(r + 1);
        else cp_async_commit();
        cp_async_wait1();
        __syncwarp();
        if (r < nwin && (w.node != kNoNode || w.s != T.dead)) {
            const uint32_t ws = wrel + kCoopWin * r;
            const uint32_t sb = stage + (r & 1) * kCoopBufBytes + 64 * lane;
            const uint32_t stop = min(srel, ws + kCoopWin);
            if (w.node == kNoNode && prel == ws && stop == ws + kCoopWin) {
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q) {
                    const uint4 x = lds_v4(sb + 16 * (q ^ sw));
                    const uint32_t v[4] = {x.x, x.y, x.z, x.w};
                    w.s = T.template take<4>(w.s, v);
                }
            } else {
#pragma unroll 1
                for (uint32_t q = 0; q < 4; ++q) {
                    const uint32_t a = max(prel, ws + 16 * q), b = min(stop, ws + 16 * q + 16);
                    if (a >= b) continue;
                    const uint32_t sa = sb + 16 * (q ^ sw);
                    if (w.node == kNoNode && b - a == 16) {
                        const uint4 x = lds_v4(sa);
                        const uint32_t v[4] = {x.x, x.y, x.z, x.w};
                        w.s = T.template take<4>(w.s, v);
                    } else {
                        for (uint32_t o = a; o < b; ++o) w.step(lds_u8(sa + ((o - ws) & 15)));
                    }
                }
            }
            prel = stop;
        }
        __syncwarp();
    }
    cp_async_wait0();
    __syncwarp();
    if (w.node == kNoNode && w.s == T.dead) return;
    if (have) pos = base + prel;
    while (pos < end) w.step(__ldg(reinterpret_cast<const uint8_t *>(pos++)));
}

template <int KIND, int G, int E>
__global__ void __launch_bounds__(kStreamBlock, 1) rid_stream_kernel(StreamArgs p) {
    extern __shared__ __align__(128) uint8_t smem[];
    using S = Steps<KIND, G, E>;
    Walk w;
    load_tables<S>(p, smem, w);
    S T;
    T.init(p, smem_addr(smem));
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warp0 = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t warps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
    const uint64_t t0 = reinterpret_cast<uint64_t>(p.text), t1 = t0 + p.len;
    for (uint64_t task = warp0; task * 32 < p.np; task += warps) {
        const uint64_t i = task * 32 + lane;
        const bool have = i < p.np;
        const uint64_t pos = t0 + (have ? piece_begin(p, i) : p.len), end = have ? t0 + piece_begin(p, i + 1) : t1;
        w.start();
        if constexpr (S::kStaged)
            stream_staged(T, w, smem_addr(smem) + p.off_stage + (threadIdx.x >> 5) * kWarpCoopBytes, pos, end, t0, t1);
        else
            stream_direct(T, w, pos, end, t0, t1);
        if (have) p.res[i] = w.result();
    }
}

// ------------------------------------------------------------------------------- join
struct StreamJoinArgs {
    JoinArgs j;
    uint16_t *maps;
    uint32_t *dinfo;
    const uint32_t *res;
    const uint16_t *part, *node_part, *images;
    const uint32_t *node_img, *slot_alive;
    uint32_t per_chunk;      // pieces per chunk
    uint32_t chunks;         // chunks per block
    uint32_t k_magic;        // ceil(2^32 / k): e / k = umulhi(e, k_magic) for e < 2^16
    uint32_t *work;          // status bits of this call while it runs
    uint8_t *h_accept;
    uint32_t *h_status;
};

constexpr uint32_t kGeneral = 0xFFFFFFFFu;   // a chunk with a piece that never merged
constexpr uint32_t kBatch = 256;             // chunks a join block handles at a time

// The state that a piece's function takes x to (the dead state n: none).
__device__ __forceinline__ uint32_t apply_piece(const StreamJoinArgs &p, uint32_t f, uint32_t x) {
    const uint32_t n = p.j.A.n;
    if (x >= n) return n;
    if (f & kNodeResult) {
        const uint32_t u = f & ~kNodeResult;
        const uint16_t b = __ldg(p.part + static_cast<uint64_t>(__ldg(p.node_part + u)) * n + x);
        return b == kNoBlock ? n : __ldg(p.images + __ldg(p.node_img + u) + b);
    }
    return __ldg(p.part + static_cast<uint64_t>(f >> 16) * n + x) == kNoBlock ? n : f & 0xFFFF;
}

// Chunk i's function as one word where all of its pieces merged: pid of the first piece and the last
// one's state, or partition 0 and the dead state when some piece's state finds no block in the next
// piece.  By one lane (stride 1), or by a warp, each lane taking every 32nd piece.
__device__ __forceinline__ void chunk_word(const StreamJoinArgs &p, uint64_t i, uint32_t first, uint32_t stride, bool &general,
                                           bool &ok) {
    const uint32_t n = p.j.A.n, s = p.per_chunk;
    const uint32_t *r = p.res + i * s;
    for (uint32_t t = first; t < s; t += stride) {
        const uint32_t f = __ldg(r + t);
        if (f & kNodeResult) {
            general = true;
        } else if (t) {
            const uint32_t y = __ldg(r + t - 1);
            if (!(y & kNodeResult)) {
                const uint32_t x = y & 0xFFFF;
                if (x >= n || __ldg(p.part + static_cast<uint64_t>(f >> 16) * n + x) == kNoBlock) ok = false;
            }
        }
    }
}

__device__ __forceinline__ uint32_t chunk_result(const StreamJoinArgs &p, uint64_t i, bool general, bool ok) {
    const uint32_t n = p.j.A.n;
    if (general) return kGeneral;
    const uint32_t f0 = __ldg(p.res + i * p.per_chunk), fl = __ldg(p.res + (i + 1) * p.per_chunk - 1);
    return ok && (fl & 0xFFFF) != n ? (f0 & 0xFFFF0000u) | (fl & 0xFFFF) : n;
}

// Map row and summary of a chunk some piece of which never merged, by a warp.
__device__ void general_row(const StreamJoinArgs &p, uint64_t i, uint32_t lane) {
    const Automaton &A = p.j.A;
    constexpr int kMaxR = RIDFA_MAX_SLOTS / 32;
    uint32_t v[kMaxR];
#pragma unroll
    for (int r = 0; r < kMaxR; ++r) {
        const uint32_t a = r * 32 + lane;
        v[r] = kUndef;
        if (a < A.k) {
            uint32_t x = A.slot_state[a];
            for (uint32_t t = 0; t < p.per_chunk && x < A.n; ++t) x = apply_piece(p, __ldg(p.res + i * p.per_chunk + t), x);
            if (x < A.n) v[r] = x;
            p.maps[i * A.k + a] = static_cast<uint16_t>(v[r]);
        }
    }
    uint32_t cnt = 0, first = kUndef, cur = 0;
    for (;;) {
        uint32_t m = 0xFFFFFFFFu;
#pragma unroll
        for (int r = 0; r < kMaxR; ++r)
            if (v[r] != kUndef && (cnt == 0 || v[r] > cur)) m = min(m, v[r]);
        m = __reduce_min_sync(kFull, m);
        if (m == 0xFFFFFFFFu) break;
        if (cnt == 0) first = m;
        cur = m;
        if (++cnt > kMaxD) break;
    }
    if (lane == 0) {
        p.dinfo[i] = cnt > kMaxD ? (0xFFu << 16) | first : cnt ? (cnt << 16) | first : static_cast<uint32_t>(kUndef);
        if (cnt > kMaxD) atomicOr(p.work, kStatusWide);
    }
}

// Thread 0 of the last block: accept bit (when `acc` is one) and status to their places, counters
// back to zero for the next call.
__device__ void publish(const StreamJoinArgs &p) {
    const uint32_t st = *reinterpret_cast<volatile uint32_t *>(p.work);
    *p.j.status = st;
    *p.work = 0;
    *p.j.ticket = 0;
    if (p.h_accept) {
        *p.h_accept = *reinterpret_cast<volatile uint8_t *>(p.j.accept);
        *p.h_status = st;
        __threadfence_system();
    }
}

__global__ void __launch_bounds__(kJoinThreads) rid_stream_join_kernel(StreamJoinArgs p) {
    __shared__ Prod s_prod[kJoinThreads];
    __shared__ uint32_t s_info[kBatch + 1];
    __shared__ uint32_t s_vec[RIDFA_MAX_SLOTS / 32], s_nvec[RIDFA_MAX_SLOTS / 32];
    __shared__ uint32_t s_general, s_bits, s_last;
    const Automaton &A = p.j.A;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t c = p.j.c;
    const uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * p.chunks, i1 = min(c, i0 + p.chunks);
    const uint32_t cnt = static_cast<uint32_t>(i1 - i0);
    const uint32_t before = i0 ? 1 : 0;          // the previous chunk is looked at too
    if (tid == 0) {
        s_general = 0;
        s_bits = 1;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    // ---- each chunk's function in one word: s_info[j] = chunk i0 - before + j
    if (p.per_chunk <= 8) {
        for (uint32_t j = tid; j < cnt + before; j += blockDim.x) {
            bool general = false, ok = true;
            chunk_word(p, i0 - before + j, 0, 1, general, ok);
            s_info[j] = chunk_result(p, i0 - before + j, general, ok);
            if (general) s_general = 1;
        }
    } else {
        for (uint32_t j = warp; j < cnt + before; j += blockDim.x / 32) {
            bool general = false, ok = true;
            chunk_word(p, i0 - before + j, lane, 32, general, ok);
            general = __any_sync(kFull, general);
            ok = __all_sync(kFull, ok);
            if (lane == 0) {
                s_info[j] = chunk_result(p, i0 - before + j, general, ok);
                if (general) s_general = 1;
            }
        }
    }
    __syncthreads();
    // ---- map rows and summaries.  A block with an unmerged chunk also writes the row before its
    // first (the same values as the block that owns it), which its transfer matrices read.
    const uint32_t skip = s_general ? 0 : before;
    const uint32_t nrow = cnt + before - skip;
    const uint64_t r0 = i0 - before + skip;
    uint16_t *rows = p.maps + r0 * A.k;
    auto cell = [&](uint32_t info, uint32_t a) -> uint32_t {
        const uint32_t m = __ldg(p.slot_alive + (info >> 16) * A.kw + (a >> 5));
        return (m >> (a & 31)) & 1 ? info & 0xFFFF : kUndef;
    };
    if (!s_general && !(A.k & 1) && !(reinterpret_cast<uint64_t>(rows) & 3)) {
        uint32_t *rows32 = reinterpret_cast<uint32_t *>(rows);
        for (uint32_t e = tid; e < nrow * A.k / 2; e += blockDim.x) {
            const uint32_t j = A.k == 1 ? e : __umulhi(2 * e, p.k_magic), a = 2 * e - j * A.k;
            const uint32_t info = s_info[j + skip];
            const uint32_t m = __ldg(p.slot_alive + (info >> 16) * A.kw + (a >> 5)) >> (a & 31);
            const uint32_t y = info & 0xFFFF;
            rows32[e] = (m & 1 ? y : kUndef) | (m & 2 ? y : kUndef) << 16;
        }
    } else {
        for (uint32_t e = tid; e < nrow * A.k; e += blockDim.x) {
            const uint32_t j = A.k == 1 ? e : __umulhi(e, p.k_magic), a = e - j * A.k;
            const uint32_t info = s_info[j + skip];
            if (info != kGeneral) rows[e] = static_cast<uint16_t>(cell(info, a));
        }
    }
    for (uint32_t j = tid; j < nrow; j += blockDim.x) {
        const uint32_t info = s_info[j + skip];
        if (info == kGeneral) continue;
        uint32_t any = 0;
        for (uint32_t w = 0; w < A.kw; ++w) any |= __ldg(p.slot_alive + (info >> 16) * A.kw + w);
        p.dinfo[r0 + j] = any && (info & 0xFFFF) != A.n ? (1u << 16) | (info & 0xFFFF) : static_cast<uint32_t>(kUndef);
    }
    if (s_general) {
        for (uint32_t j = warp; j < nrow; j += blockDim.x / 32)
            if (s_info[j + skip] == kGeneral) general_row(p, r0 + j, lane);
    }
    // ---- this block's boundaries (chunk i - 1 to i, i0 <= i < i1, i >= 1): their product
    Prod P;
    P.nrows = 0xFFFFFFFFu;
    if (!s_general) {
        const uint32_t j = tid + 1 - before;     // boundary into s_info[j + before]
        bool bit = true;
        for (uint32_t b = j; b < cnt; b += blockDim.x) {
            const uint32_t prev = s_info[b + before - 1], cur = s_info[b + before];
            uint32_t hit = 0;
            if ((prev & 0xFFFF) != A.n && (cur & 0xFFFF) != A.n)
                for (uint32_t w = 0; w < A.kw; ++w)
                    hit |= __ldg(A.ifmask + static_cast<uint64_t>(prev & 0xFFFF) * A.kw + w) & __ldg(p.slot_alive + (cur >> 16) * A.kw + w);
            bit = bit && hit;
        }
        if (!bit) s_bits = 0;
        __syncthreads();
        if (cnt + before > 1) {
            P.nrows = (s_info[0] & 0xFFFF) != A.n ? 1 : 0;
            P.rows[0] = s_bits;
        }
    } else {
        __syncthreads();                         // the rows above are in place
        bool bad = false;
        const uint64_t i = i0 + 1 - before + tid;
        if (i < i1) {
            uint16_t Dp[kMaxD], Dc[kMaxD];
            const uint32_t mp = distinct_of(p.j, static_cast<uint32_t>(i - 1), Dp), mc = distinct_of(p.j, static_cast<uint32_t>(i), Dc);
            if (mp <= static_cast<uint32_t>(kMaxD) && mc <= static_cast<uint32_t>(kMaxD)) {   // (else: the wide path)
                P.nrows = mp;
                for (uint32_t z = 0; z < mp; ++z) P.rows[z] = transfer_row(p.j, static_cast<uint32_t>(i), Dp[z], Dc, mc, &bad);
            }
        }
        if (bad) atomicOr(p.work, kStatusBad);
        s_prod[tid] = P;
        __syncthreads();
        for (uint32_t stride = 1; stride < blockDim.x; stride *= 2) {
            if ((tid % (2 * stride)) == 0 && tid + stride < blockDim.x) compose(s_prod[tid], s_prod[tid + stride]);
            __syncthreads();
        }
        if (tid == 0) P = s_prod[0];
    }
    if (tid == 0) {
        uint32_t *mine = p.j.partials + static_cast<uint64_t>(blockIdx.x) * kPartialWords;
        mine[0] = P.nrows;
        if (P.nrows != 0xFFFFFFFFu)
            for (uint32_t x = 0; x < P.nrows; ++x) mine[1 + x] = P.rows[x];
        __threadfence();
        s_last = atomicAdd(p.j.ticket, 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // ---- last block: the product of all blocks, then lambda_1(q0) and the acceptance test
    if (*reinterpret_cast<volatile uint32_t *>(p.work) & kStatusWide) {
        if (p.j.summary) summary_wide(p.j, s_vec, s_nvec);
        else accept_wide(p.j, s_vec, s_nvec);
        __syncthreads();
        if (tid == 0) publish(p);
        return;
    }
    // while every block's product has at most one row and column, it is the AND of their bits
    if (tid == 0) {
        s_general = 0;
        s_bits = 1;
    }
    __syncthreads();
    {
        bool general = false, bit = true;
        for (uint32_t b = tid; b < gridDim.x; b += blockDim.x) {
            const volatile uint32_t *q = p.j.partials + static_cast<uint64_t>(b) * kPartialWords;
            const uint32_t nr = q[0];
            if (nr == 0xFFFFFFFFu) continue;
            if (nr > 1) general = true;
            else bit = bit && nr == 1 && q[1] == 1;
            if (nr == 1 && q[1] > 1) general = true;
        }
        if (general) s_general = 1;
        if (!bit) s_bits = 0;
    }
    __syncthreads();
    Prod tot;
    tot.nrows = 0xFFFFFFFFu;
    if (!s_general) {
        if (c > 1) {
            tot.nrows = 1;
            tot.rows[0] = s_bits;
        }
    } else {
        for (uint32_t base = 0; base < gridDim.x; base += blockDim.x) {
            Prod x;
            x.nrows = 0xFFFFFFFFu;
            if (base + tid < gridDim.x) {
                const volatile uint32_t *q = p.j.partials + static_cast<uint64_t>(base + tid) * kPartialWords;
                x.nrows = q[0];
                if (x.nrows != 0xFFFFFFFFu)
                    for (uint32_t r = 0; r < x.nrows; ++r) x.rows[r] = q[1 + r];
            }
            __syncthreads();
            s_prod[tid] = x;
            __syncthreads();
            for (uint32_t stride = 1; stride < blockDim.x; stride *= 2) {
                if ((tid % (2 * stride)) == 0 && tid + stride < blockDim.x) compose(s_prod[tid], s_prod[tid + stride]);
                __syncthreads();
            }
            if (tid == 0) compose(tot, s_prod[0]);
            __syncthreads();
        }
    }
    if (tid != 0) return;
    if (p.j.summary) {
        summary_matrix(p.j, tot);
        publish(p);
        return;
    }
    // (chunk 0's row and summary come from another block: read past the caches of this one)
    const uint16_t v0 = *reinterpret_cast<const volatile uint16_t *>(p.maps + A.q0_slot);
    uint8_t acc = 0;
    if (v0 != kUndef) {
        if (c == 1) {
            acc = is_final(A, v0) ? 1 : 0;
        } else {
            uint16_t D0[kMaxD], Dl[kMaxD];
            const uint32_t m0 = distinct_of(p.j, 0, D0), x0 = index_of(D0, m0, v0);
            const uint32_t ml = distinct_of(p.j, static_cast<uint32_t>(c - 1), Dl);
            if (x0 == 0xFFFFFFFFu || tot.nrows == 0xFFFFFFFFu || ml == 0xFFFFFFFFu) {
                atomicOr(p.work, kStatusBad);
            } else if (x0 < tot.nrows) {
                const uint32_t bits = tot.rows[x0];
                for (uint32_t y = 0; y < ml; ++y)
                    if (((bits >> y) & 1) && is_final(A, Dl[y])) acc = 1;
            }
        }
    }
    *p.j.accept = acc;
    publish(p);
}

// --------------------------------------------------------------------------- host side
using StreamKernel = void (*)(StreamArgs);

StreamKernel stream_kernel(const HostStream &T) {
    const bool b = T.entry == 1;
    switch (T.kind) {
        case kStreamField:
            return T.group == 4 ? (b ? rid_stream_kernel<kStreamField, 4, 1> : rid_stream_kernel<kStreamField, 4, 2>)
                                : (b ? rid_stream_kernel<kStreamField, 2, 1> : rid_stream_kernel<kStreamField, 2, 2>);
        case kStreamPair: return b ? rid_stream_kernel<kStreamPair, 2, 1> : rid_stream_kernel<kStreamPair, 2, 2>;
        default: return b ? rid_stream_kernel<kStreamSingle, 1, 1> : rid_stream_kernel<kStreamSingle, 1, 2>;
    }
}

constexpr uint64_t kMinPiece = 64;             // bytes a piece has at least, where chunks are cut

}  // namespace

bool stream_takes(const HostAutomaton &H, uint64_t len, uint32_t c) {
    // (the kernels keep a warp's 32 pieces within 32-bit offsets; stream_shape cuts any text of up
    // to 2^40 bytes into pieces far below that)
    return H.stream.kind != kStreamNone && c <= (1u << 26) && len <= (1ull << 40);
}

StreamShape stream_shape(const HostAutomaton &H, uint64_t len, uint32_t c, int sms) {
    StreamShape S;
    const uint64_t W = H.stream.warps;
    const double L = static_cast<double>(len) / c;
    // Pieces per chunk: the SM with the most warps of pieces decides.  A full round of W warps and a
    // rest of fewer than 16 take about as long as 16 warps do; a piece costs some 80 bytes beside
    // its own (ragged ends, graph walk).
    auto time = [&](uint64_t s) {
        const uint64_t warps = (static_cast<uint64_t>(c) * s + 31) / 32, m = (warps + sms - 1) / sms;
        const uint64_t rest = m % W;
        return static_cast<double>(m / W * W + (rest ? std::max<uint64_t>(rest, std::min<uint64_t>(16, W)) : 0)) *
               (L / static_cast<double>(s) + 80.0);
    };
    uint64_t best = 1;
    double best_t = time(1);
    auto consider = [&](uint64_t s) {
        if (s < 2 || len / c / s < kMinPiece) return;
        const double t = time(s);
        if (t < best_t) {
            best_t = t;
            best = s;
        }
    };
    const uint64_t lanes = static_cast<uint64_t>(sms) * 32;
    for (uint64_t s = 2; s <= 16; ++s) consider(s);
    for (uint64_t m = 1; m <= 2 * W; ++m) consider(m * lanes / c);
    S.per_chunk = static_cast<uint32_t>(best);
    S.pieces = static_cast<uint64_t>(c) * best;
    const uint64_t tasks = (S.pieces + 31) / 32;
    const uint64_t warps = std::min<uint64_t>(W, (tasks + sms - 1) / sms);
    S.block = static_cast<uint32_t>(warps * 32);
    S.grid = static_cast<uint32_t>(std::min<uint64_t>(sms, (tasks + warps - 1) / warps));
    S.smem = stream_table_bytes(H) + (H.stream.kind == kStreamField ? 0 : warps * kStreamStaging);
    // a join block takes 256 chunks, one thread each; where chunks have many pieces, a warp each
    S.join_chunks = S.per_chunk <= 8 ? kBatch : std::min<uint32_t>(kBatch, std::max<uint32_t>(kJoinThreads / 32, (c + 1023) / 1024));
    S.join_blocks = static_cast<uint32_t>((static_cast<uint64_t>(c) + S.join_chunks - 1) / S.join_chunks);
    return S;
}

cudaError_t stream_launch(const StreamCall &C, const StreamShape &S, cudaStream_t st) {
    const HostAutomaton &H = *C.H;
    const DeviceAutomaton &D = *C.D;
    const HostStream &T = H.stream;
    StreamArgs a{};
    a.text = C.text;
    a.len = C.len;
    a.np = S.pieces;
    a.q = C.len / S.pieces;
    a.r = C.len % S.pieces;
    a.res = C.res;
    a.trans = D.trans;
    a.classmap = D.classmap;
    a.next = D.mg_next;
    a.leaf = D.mg_leaf;
    a.code = D.st_code;
    a.words = D.st_words;
    a.n = H.n_states;
    a.C = H.n_classes;
    a.inner = H.merge.inner;
    a.n_words = static_cast<uint32_t>(T.words.size());
    a.copies = T.copies;
    a.row = T.row_words * 4 * T.copies;
    if (T.kind == kStreamField) {
        const uint32_t w = T.width, lgf = static_cast<uint32_t>(__builtin_ctz(T.copies)) + 2;   // log2 of bytes per word
        a.shift = T.shift;
        a.mask = ((1u << w) - 1) * 0x01010101u;
        a.canon = T.canon;
        // byte i's code to bit 24 + w * i
        a.mul = 1u << 24 | 1u << (16 + w);
        if (T.group == 4) a.mul |= 1u << (8 + 2 * w) | 1u << (3 * w);
        // column = the code at bit 24: its low bits are the part of a word, the others the word
        const uint32_t part = T.entry == 1 ? 2 : 1, cols = w * T.group;      // bits
        a.m_q = (1u << std::min(part, cols)) - 1;
        a.sh_q = 24;
        if (T.entry == 2) {
            a.m_q <<= 1;
            a.sh_q = 23;
        }
        a.m_w = cols > part ? ((1u << (cols - part)) - 1) << lgf : 0;
        a.sh_w = 24 + part - lgf;
    }
    uint32_t off = T.kind == kStreamField ? 0 : 256 * 128;
    a.off_table = off;
    off += a.n_words * 4 * T.copies;
    const uint32_t tb = static_cast<uint32_t>(H.trans.size() * 2), nb = static_cast<uint32_t>(H.merge.next.size() * 2);
    off = (off + 15) & ~15u;
    a.off_cls = off;
    off += 256;
    a.off_trans = tb <= kStreamTransSmem ? off : kGlobal;
    off += tb <= kStreamTransSmem ? (tb + 15) & ~15u : 0;
    a.off_next = nb <= kStreamNextSmem ? off : kGlobal;
    off += nb <= kStreamNextSmem ? (nb + 15) & ~15u : 0;
    a.off_stage = (off + 127) & ~127u;
    const StreamKernel kern = stream_kernel(T);
    cudaError_t e = ensure_smem_cap(reinterpret_cast<const void *>(kern), S.smem);
    if (e != cudaSuccess) return e;
    kern<<<S.grid, S.block, S.smem, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (C.between) {
        e = cudaEventRecord(C.between, st);
        if (e != cudaSuccess) return e;
    }
    const Automaton A{D.trans, D.classmap, D.final_bits, D.ifmask, D.slot_state,
                      H.n_states, H.n_classes, H.k, H.kw, H.q0_slot, H.merges};
    StreamJoinArgs j{};
    j.j = JoinArgs{A, C.c, C.maps, C.dinfo, C.status, C.partials, C.ticket, C.accept, 1, C.summary};
    j.maps = C.maps;
    j.dinfo = C.dinfo;
    j.res = C.res;
    j.part = D.mg_part;
    j.node_part = D.mg_node_part;
    j.images = D.mg_images;
    j.node_img = D.mg_node_img;
    j.slot_alive = D.mg_slot_alive;
    j.per_chunk = S.per_chunk;
    j.chunks = S.join_chunks;
    j.k_magic = static_cast<uint32_t>((0xFFFFFFFFull + H.k) / H.k);
    j.work = C.work;
    j.h_accept = C.h_accept;
    j.h_status = C.h_status;
    // the join's blocks may be set up while the last stream blocks run (they wait at their start)
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(S.join_blocks);
    cfg.blockDim = dim3(kJoinThreads);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = C.between ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, rid_stream_join_kernel, j);
}

}  // namespace ridfa

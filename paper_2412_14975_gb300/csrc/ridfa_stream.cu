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
// Bounds, and the reach phase against the general kernels': tables of pairs by the shared-memory pipe
// (two class lookups and one transition for two bytes, and the staged text: 4 GiB of record lines in
// 155,648 chunks 1,290 -> 959 us, 4.5 TB/s); field codes of four bytes by the lanes' text loads and the
// table's bank conflicts (1 GiB, (a|b)*a(a|b){7}: 355 -> 214 us, 5.0 TB/s); short texts by the latency
// of one chain of some 64 steps and of the launches (1 MiB in 64 chunks 36 -> 10 us).
//
// The join kernel composes a chunk's pieces, writes the chunk maps and evaluates the join.  A
// chunk whose pieces all merged has at most one end state, so a boundary's transfer matrix is one
// bit: does if_min of the previous chunk's end state meet the slots alive in this chunk?
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "ridfa_join.cuh"
#include "ridfa_stream.cuh"
#include "ridfa_stream.h"

namespace ridfa {
namespace {

struct StreamArgs {
    const uint8_t *text;
    uint64_t len, q, frac;        // chunk i begins at i * q + (i * frac >> 64): floor(i * len / c)
    uint64_t step;                // bytes per piece of a chunk, 16 fraction bits
    uint32_t np, per_chunk;       // pieces in all, and per chunk
    uint32_t *res;                // [np]: kNodeResult | node, or pid << 16 | state
    StreamTables t;
};

__device__ __forceinline__ uint64_t chunk_at(const StreamArgs &p, uint32_t i) {
    return i * p.q + __umul64hi(i, p.frac);
}

// Piece x as addresses [pos, end).  Inside a chunk the pieces meet at 32-byte boundaries.
__device__ __forceinline__ void piece_range(const StreamArgs &p, uint32_t x, uint64_t t0, uint64_t &pos, uint64_t &end) {
    if (p.per_chunk == 1) {
        pos = t0 + chunk_at(p, x);
        end = t0 + chunk_at(p, x + 1);
        return;
    }
    const uint32_t i = x / p.per_chunk, t = x - i * p.per_chunk;
    const uint64_t b = t0 + chunk_at(p, i);
    pos = t ? (b + (t * p.step >> 16)) & ~static_cast<uint64_t>(31) : b;
    end = t + 1 < p.per_chunk ? (b + ((t + 1) * p.step >> 16)) & ~static_cast<uint64_t>(31) : t0 + chunk_at(p, i + 1);
}

template <int KIND, int G, int E, int W>
__global__ void __launch_bounds__(kStreamBlock, 1) rid_stream_kernel(const __grid_constant__ StreamArgs p) {
    extern __shared__ __align__(128) uint8_t smem[];
    using S = Steps<KIND, G, E, W>;
    load_tables<S>(p.t, smem);
    Walk w(p.t, smem_addr(smem));
    const S T(p.t, smem_addr(smem));
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp >= p.t.warps) return;                 // (only loaded tables)
    const uint64_t t0 = reinterpret_cast<uint64_t>(p.text), t1 = t0 + p.len;
    for (uint32_t task = blockIdx.x * p.t.warps + warp; task * 32 < p.np; task += gridDim.x * p.t.warps) {
        const uint32_t x = task * 32 + lane;
        const bool have = x < p.np;
        uint64_t pos = t1, end = t1;
        if (have) piece_range(p, x, t0, pos, end);
        w.start();
        if constexpr (S::kStaged)
            // (pieces ascend: the warp's first one starts lowest)
            stream_staged(T, w, smem_addr(smem) + p.t.off_stage + warp * kWarpCoopBytes,
                          __shfl_sync(kFull, pos, 0) & ~static_cast<uint64_t>(15), pos, end, t0, t1);
        else
            stream_direct(T, w, pos, end, t0, t1);
        if (have) p.res[x] = w.result();
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
    const uint16_t *tables;  // of the groups that did not merge (kTableResult)
    uint32_t per_chunk;      // pieces (or groups of them) per chunk
    uint32_t chunks;         // chunks per block
    uint32_t k_magic;        // ceil(2^32 / k): e / k = umulhi(e, k_magic) while e * k < 2^32 (e <= 257 k here)
    uint32_t *status;        // the call's status, written once by publish(); while it runs its bits are in j.status
    uint8_t *h_accept;
    uint32_t *h_status;
};

constexpr uint32_t kGeneral = 0xFFFFFFFFu;   // a chunk with a piece that never merged
constexpr uint32_t kTableResult = 0xC0000000u;   // | g: group g's function is row g of the tables (a node
                                                 // id is below 2^15)
constexpr uint32_t kBatch = 256;             // chunks a join block handles at a time

// The state that a piece's function takes x to (the dead state n: none).
__device__ __forceinline__ uint32_t apply_piece(const StreamJoinArgs &p, uint32_t f, uint32_t x) {
    const uint32_t n = p.j.A.n;
    if (x >= n) return n;
    if (f & kNodeResult) {
        if (f >= kTableResult) return __ldcg(p.tables + static_cast<uint64_t>(f & ~kTableResult) * n + x);
        const uint32_t u = f & ~kNodeResult;
        const uint16_t b = __ldg(p.part + static_cast<uint64_t>(__ldg(p.node_part + u)) * n + x);
        return b == kNoBlock ? n : __ldg(p.images + __ldg(p.node_img + u) + b);
    }
    return __ldg(p.part + static_cast<uint64_t>(f >> 16) * n + x) == kNoBlock ? n : f & 0xFFFF;
}

// x through the functions r[0, s), eight words and their tables' places ahead of the states (one after
// another a piece took 0.55 us).
__device__ __forceinline__ uint32_t apply_pieces(const StreamJoinArgs &p, const uint32_t *r, uint32_t s, uint32_t x) {
    const uint32_t n = p.j.A.n;
    if (s < 4) {
        for (uint32_t t = 0; t < s && x < n; ++t) x = apply_piece(p, __ldcg(r + t), x);
        return x;
    }
    for (uint32_t t0 = 0; t0 < s && x < n; t0 += 8) {
        uint32_t f[8], row[8], img[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) f[u] = t0 + u < s ? __ldcg(r + t0 + u) : 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool node = (f[u] & kNodeResult) && f[u] < kTableResult;
            row[u] = node ? __ldg(p.node_part + (f[u] & ~kNodeResult)) : f[u] >> 16;
            img[u] = node ? __ldg(p.node_img + (f[u] & ~kNodeResult)) : 0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (t0 + u >= s || x >= n) continue;
            if (f[u] >= kTableResult) {
                x = apply_piece(p, f[u], x);
            } else {
                const uint16_t b = __ldg(p.part + static_cast<uint64_t>(row[u]) * n + x);
                x = b == kNoBlock ? n : f[u] & kNodeResult ? __ldg(p.images + img[u] + b) : f[u] & 0xFFFF;
            }
        }
    }
    return x;
}

// Chunk i's function as one word where all of its pieces merged: pid of the first piece and the last
// one's state, or partition 0 and the dead state when some piece's state finds no block in the next
// piece; kGeneral when some piece never merged.
__device__ __forceinline__ bool goes_on(const StreamJoinArgs &p, uint32_t y, uint32_t f) {
    const uint32_t x = y & 0xFFFF;
    return x < p.j.A.n && __ldg(p.part + static_cast<uint64_t>(f >> 16) * p.j.A.n + x) != kNoBlock;
}

// One lane, at most 4 pieces (results are read from L2: the fused join reads other blocks' ones).
__device__ __forceinline__ uint32_t chunk_word(const StreamJoinArgs &p, uint64_t i) {
    const uint32_t s = p.per_chunk, *r = p.res + i * s;
    uint32_t f[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) f[t] = t < s ? __ldcg(r + t) : 0;
    uint32_t node = f[0], last = f[0];
    bool ok = true;
#pragma unroll
    for (int t = 1; t < 4; ++t)
        if (t < s) {
            node |= f[t];
            last = f[t];
        }
    if (node & kNodeResult) return kGeneral;
#pragma unroll
    for (int t = 1; t < 4; ++t)
        if (t < s) ok = goes_on(p, f[t - 1], f[t]) && ok;
    return ok && (last & 0xFFFF) != p.j.A.n ? (f[0] & 0xFFFF0000u) | (last & 0xFFFF) : p.j.A.n;
}

// The s pieces at r by a warp: a piece per lane, up to eight at a time so that their loads overlap.
__device__ __forceinline__ uint32_t chunk_word_warp(const StreamJoinArgs &p, const uint32_t *r, uint32_t s, uint32_t lane) {
    uint32_t first = 0, carry = 0;
    bool node = false, ok = true;
    for (uint32_t b = 0; b < s; b += 256) {
        uint32_t f[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) f[u] = b + 32 * u + lane < s ? __ldcg(r + b + 32 * u + lane) : 0;
        if (b == 0) first = __shfl_sync(kFull, f[0], 0);
        bool go[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            uint32_t y = __shfl_up_sync(kFull, f[u], 1);
            const uint32_t end = __shfl_sync(kFull, f[u], 31);
            if (lane == 0) y = carry;
            carry = end;
            const uint32_t t = b + 32 * u + lane;
            node = node || (f[u] & kNodeResult);
            go[u] = true;
            if (t < s && t && !((f[u] | y) & kNodeResult)) go[u] = goes_on(p, y, f[u]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) ok = ok && go[u];
    }
    const uint32_t last = __ldcg(r + s - 1);
    node = __any_sync(kFull, node);
    ok = __all_sync(kFull, ok);
    if (node) return kGeneral;
    return ok && (last & 0xFFFF) != p.j.A.n ? (first & 0xFFFF0000u) | (last & 0xFFFF) : p.j.A.n;
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
            const uint32_t x = apply_pieces(p, p.res + i * p.per_chunk, p.per_chunk, A.slot_state[a]);
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
        if (cnt > kMaxD) atomicOr(p.j.status, kStatusWide);
    }
}

// Thread 0 of the last block: accept bit and status to their places, counters back to zero for the
// next call.
__device__ void publish(const StreamJoinArgs &p, uint8_t acc) {
    const uint32_t st = *reinterpret_cast<volatile uint32_t *>(p.j.status);
    *p.status = st;
    if (st) *p.j.status = 0;
    *p.j.ticket = 0;
    *p.j.accept = acc;
    if (p.h_accept) {
        *p.h_accept = acc;
        *p.h_status = st;                // (visible to the host once the kernel has ended)
    }
}

struct JoinShared {
    Prod prod[kJoinThreads];
    uint32_t info[kBatch + 1];
    uint32_t vec[RIDFA_MAX_SLOTS / 32], nvec[RIDFA_MAX_SLOTS / 32];
    uint32_t general, bits, last;
};

// Words 31 and 32 of a block's partial product hold the words of its first and last chunk while the
// product has at most one row.
constexpr uint32_t kFirstInfo = kPartialWords - 2, kLastInfo = kPartialWords - 1;

// The accept bit when some chunk has more than kMaxD distinct end states, by one block: if_min(PLAS_i)
// as a k-bit set, chunk by chunk, every slot's end state worked out from the pieces.
__device__ uint32_t accept_unmerged(const StreamJoinArgs &p, uint32_t *s_vec, uint32_t *s_nvec) {
    const Automaton &A = p.j.A;
    __shared__ uint32_t s_acc;
    for (uint32_t w = threadIdx.x; w < A.kw; w += blockDim.x) s_vec[w] = (A.q0_slot >> 5) == w ? 1u << (A.q0_slot & 31) : 0u;
    if (threadIdx.x == 0) s_acc = 0;
    for (uint64_t i = 0; i < p.j.c; ++i) {
        for (uint32_t w = threadIdx.x; w < A.kw; w += blockDim.x) s_nvec[w] = 0;
        __syncthreads();
        for (uint32_t a = threadIdx.x; a < A.k; a += blockDim.x) {
            if (!((s_vec[a >> 5] >> (a & 31)) & 1)) continue;
            const uint32_t x = apply_pieces(p, p.res + i * p.per_chunk, p.per_chunk, A.slot_state[a]);
            if (x >= A.n) continue;
            if (i + 1 == p.j.c) {
                if (is_final(A, x)) s_acc = 1;
            } else {
                for (uint32_t w = 0; w < A.kw; ++w) {
                    const uint32_t m = A.ifmask[static_cast<uint64_t>(x) * A.kw + w];
                    if (m) atomicOr(&s_nvec[w], m);
                }
            }
        }
        __syncthreads();
        for (uint32_t w = threadIdx.x; w < A.kw; w += blockDim.x) s_vec[w] = s_nvec[w];
        __syncthreads();
    }
    return s_acc;
}

// The join of chunks [blk * chunks, ...) by one block of kJoinThreads threads, and by the last of
// nblk blocks the whole.
__device__ void stream_join(const StreamJoinArgs &p, uint32_t blk, uint32_t nblk, JoinShared &sh) {
    const Automaton &A = p.j.A;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t c = p.j.c;
    const uint64_t i0 = static_cast<uint64_t>(blk) * p.chunks, i1 = min(c, i0 + p.chunks);
    const uint32_t cnt = static_cast<uint32_t>(i1 - i0);
    const uint32_t before = i0 ? 1 : 0;          // the previous chunk is looked at too
    if (tid == 0) {
        sh.general = 0;
        sh.bits = 1;
    }
    __syncthreads();
    // ---- each chunk's function in one word: info[j] = chunk i0 - before + j
    if (p.per_chunk <= 4) {
        for (uint32_t j = tid; j < cnt + before; j += blockDim.x) {
            const uint32_t v = chunk_word(p, i0 - before + j);
            sh.info[j] = v;
            if (v == kGeneral) sh.general = 1;
        }
    } else {
        for (uint32_t j = warp; j < cnt + before; j += blockDim.x / 32) {
            const uint32_t v = chunk_word_warp(p, p.res + (i0 - before + j) * p.per_chunk, p.per_chunk, lane);
            if (lane == 0) {
                sh.info[j] = v;
                if (v == kGeneral) sh.general = 1;
            }
        }
    }
    __syncthreads();
    // ---- map rows and summaries.  A block with an unmerged chunk also writes the row before its
    // first (the same values as the block that owns it), which its transfer matrices read.  Rows that
    // only the caller reads are written last, beside the other blocks' way to the result.
    const bool unmerged = sh.general, rows_first = unmerged || p.j.summary;
    const uint32_t skip = sh.general ? 0 : before;
    const uint32_t nrow = cnt + before - skip;
    const uint64_t r0 = i0 - before + skip;
    uint16_t *rows = p.maps + r0 * A.k;
    auto write_rows = [&]() {
        if (!unmerged && A.k >= 8 && !(A.k & 1) && !(nrow * A.k & 7) && !(reinterpret_cast<uint64_t>(rows) & 15)) {
            // 8 entries a thread and store, over at most two rows (k >= 8)
            for (uint32_t e = tid * 8; e < nrow * A.k; e += blockDim.x * 8) {
                uint32_t j = __umulhi(e, p.k_magic), a = e - j * A.k, v[4];
                uint32_t info = sh.info[j + skip];
                const uint32_t *alive = p.slot_alive + (info >> 16) * A.kw;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (a >= A.k) {
                        a = 0;
                        info = sh.info[++j + skip];
                        alive = p.slot_alive + (info >> 16) * A.kw;
                    }
                    const uint32_t m = __ldg(alive + (a >> 5)) >> (a & 31), y = info & 0xFFFF;
                    v[q] = (m & 1 ? y : kUndef) | (m & 2 ? y : kUndef) << 16;
                    a += 2;
                }
                *reinterpret_cast<uint4 *>(rows + e) = make_uint4(v[0], v[1], v[2], v[3]);
            }
        } else if (!unmerged && !(A.k & 1) && !(reinterpret_cast<uint64_t>(rows) & 3)) {
            uint32_t *rows32 = reinterpret_cast<uint32_t *>(rows);
            for (uint32_t e = tid; e < nrow * A.k / 2; e += blockDim.x) {
                const uint32_t j = __umulhi(2 * e, p.k_magic), a = 2 * e - j * A.k;
                const uint32_t info = sh.info[j + skip];
                const uint32_t m = __ldg(p.slot_alive + (info >> 16) * A.kw + (a >> 5)) >> (a & 31);
                const uint32_t y = info & 0xFFFF;
                rows32[e] = (m & 1 ? y : kUndef) | (m & 2 ? y : kUndef) << 16;
            }
        } else {
            for (uint32_t e = tid; e < nrow * A.k; e += blockDim.x) {
                const uint32_t j = A.k == 1 ? e : __umulhi(e, p.k_magic), a = e - j * A.k;
                const uint32_t info = sh.info[j + skip];
                if (info == kGeneral) continue;
                const uint32_t m = __ldg(p.slot_alive + (info >> 16) * A.kw + (a >> 5));
                rows[e] = static_cast<uint16_t>((m >> (a & 31)) & 1 ? info & 0xFFFF : kUndef);
            }
        }
    };
    if (rows_first) write_rows();
    for (uint32_t j = tid; j < nrow; j += blockDim.x) {
        const uint32_t info = sh.info[j + skip];
        if (info == kGeneral) continue;
        uint32_t any = 0;
        for (uint32_t w = 0; w < A.kw; ++w) any |= __ldg(p.slot_alive + (info >> 16) * A.kw + w);
        p.dinfo[r0 + j] = any && (info & 0xFFFF) != A.n ? (1u << 16) | (info & 0xFFFF) : static_cast<uint32_t>(kUndef);
    }
    if (sh.general) {
        for (uint32_t j = warp; j < nrow; j += blockDim.x / 32)
            if (sh.info[j + skip] == kGeneral) general_row(p, r0 + j, lane);
    }
    // ---- this block's boundaries (chunk i - 1 to i, i0 <= i < i1, i >= 1): their product
    Prod P;
    P.nrows = 0xFFFFFFFFu;
    if (!sh.general) {
        bool bit = true;
        for (uint32_t b = tid + 1 - before; b < cnt; b += blockDim.x) {      // into info[b + before]
            const uint32_t prev = sh.info[b + before - 1], cur = sh.info[b + before];
            uint32_t hit = 0;
            if ((prev & 0xFFFF) != A.n && (cur & 0xFFFF) != A.n)
                for (uint32_t w = 0; w < A.kw; ++w)
                    hit |= __ldg(A.ifmask + static_cast<uint64_t>(prev & 0xFFFF) * A.kw + w) & __ldg(p.slot_alive + (cur >> 16) * A.kw + w);
            bit = bit && hit;
        }
        if (!bit) sh.bits = 0;
        __syncthreads();
        if (cnt + before > 1) {
            P.nrows = (sh.info[0] & 0xFFFF) != A.n ? 1 : 0;
            P.rows[0] = sh.bits;
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
        if (bad) atomicOr(p.j.status, kStatusBad);
        sh.prod[tid] = P;
        __syncthreads();
        for (uint32_t stride = 1; stride < blockDim.x; stride *= 2) {
            if ((tid % (2 * stride)) == 0 && tid + stride < blockDim.x) compose(sh.prod[tid], sh.prod[tid + stride]);
            __syncthreads();
        }
        if (tid == 0) P = sh.prod[0];
    }
    uint32_t first = sh.info[before ? 1 : 0], last = sh.info[cnt + before - 1];
    bool general = unmerged, bits = sh.bits;
    if (nblk == 1 && !general && !rows_first) write_rows();
    if (nblk > 1 || general) {
        if (tid == 0) {
            uint32_t *mine = p.j.partials + static_cast<uint64_t>(blk) * kPartialWords;
            mine[0] = P.nrows;
            if (P.nrows != 0xFFFFFFFFu)
                for (uint32_t x = 0; x < P.nrows; ++x) mine[1 + x] = P.rows[x];
            if (P.nrows == 0xFFFFFFFFu || P.nrows <= 1) {
                mine[kFirstInfo] = first;
                mine[kLastInfo] = last;
            }
            __threadfence();
            sh.last = atomicAdd(p.j.ticket, 1) == nblk - 1;
        }
        __syncthreads();
        if (!rows_first) write_rows();
        if (!sh.last) return;
        __threadfence();
        // ---- last block: the product of all blocks
        if (*reinterpret_cast<volatile uint32_t *>(p.j.status) & kStatusWide) {
            uint32_t acc = 0;
            if (p.j.summary) summary_wide(p.j, sh.vec, sh.nvec);
            else acc = accept_unmerged(p, sh.vec, sh.nvec);
            __syncthreads();
            if (tid == 0) publish(p, static_cast<uint8_t>(acc));
            return;
        }
        // while every product has at most one row and column, it is the AND of their bits
        if (tid == 0) {
            sh.general = 0;
            sh.bits = 1;
        }
        __syncthreads();
        {
            bool gen = false, bit = true;
            const uint32_t *qf = p.j.partials + kFirstInfo;
            const uint32_t *ql = p.j.partials + static_cast<uint64_t>(nblk - 1) * kPartialWords + kLastInfo;
            first = __ldcg(qf);
            last = __ldcg(ql);
#pragma unroll 4
            for (uint32_t b = tid; b < nblk; b += blockDim.x) {
                const uint32_t *q = p.j.partials + static_cast<uint64_t>(b) * kPartialWords;
                const uint32_t nr = __ldcg(q), row = __ldcg(q + 1);
                if (nr != 0xFFFFFFFFu) {
                    if (nr > 1 || (nr == 1 && row > 1)) gen = true;
                    else bit = bit && nr == 1 && row == 1;
                }
            }
            if (gen || first == kGeneral || last == kGeneral) sh.general = 1;
            if (!bit) sh.bits = 0;
        }
        __syncthreads();
        general = sh.general;
        bits = sh.bits;
    }
    if (!general && !p.j.summary) {
        if (tid == 0) {
            const uint32_t q0 = A.q0_slot;
            const bool enter = (__ldg(p.slot_alive + (first >> 16) * A.kw + (q0 >> 5)) >> (q0 & 31)) & 1;
            publish(p, enter && bits && (first & 0xFFFF) != A.n && is_final(A, last & 0xFFFF) ? 1 : 0);
        }
        return;
    }
    Prod tot;
    tot.nrows = 0xFFFFFFFFu;
    if (!general) {
        if (c > 1) {
            tot.nrows = 1;
            tot.rows[0] = bits;
        }
    } else {
        for (uint32_t base = 0; base < nblk; base += blockDim.x) {
            Prod x;
            x.nrows = 0xFFFFFFFFu;
            if (base + tid < nblk) {
                const volatile uint32_t *q = p.j.partials + static_cast<uint64_t>(base + tid) * kPartialWords;
                x.nrows = q[0];
                if (x.nrows != 0xFFFFFFFFu)
                    for (uint32_t r = 0; r < x.nrows; ++r) x.rows[r] = q[1 + r];
            }
            __syncthreads();
            sh.prod[tid] = x;
            __syncthreads();
            for (uint32_t stride = 1; stride < blockDim.x; stride *= 2) {
                if ((tid % (2 * stride)) == 0 && tid + stride < blockDim.x) compose(sh.prod[tid], sh.prod[tid + stride]);
                __syncthreads();
            }
            if (tid == 0) compose(tot, sh.prod[0]);
            __syncthreads();
        }
    }
    if (tid != 0) return;
    if (p.j.summary) {
        summary_matrix(p.j, tot);
        publish(p, 0);
        return;
    }
    // (chunk 0's row may still be on its way: its entry for q0's slot from the pieces instead)
    const uint32_t x = apply_pieces(p, p.res, p.per_chunk, A.slot_state[A.q0_slot]);
    const uint16_t v0 = x < A.n ? static_cast<uint16_t>(x) : kUndef;
    uint8_t acc = 0;
    if (v0 != kUndef) {
        if (c == 1) {
            acc = is_final(A, v0) ? 1 : 0;
        } else {
            uint16_t D0[kMaxD], Dl[kMaxD];
            const uint32_t m0 = distinct_of(p.j, 0, D0), x0 = index_of(D0, m0, v0);
            const uint32_t ml = distinct_of(p.j, static_cast<uint32_t>(c - 1), Dl);
            if (x0 == 0xFFFFFFFFu || tot.nrows == 0xFFFFFFFFu || ml == 0xFFFFFFFFu) {
                atomicOr(p.j.status, kStatusBad);
            } else if (x0 < tot.nrows) {
                const uint32_t row = tot.rows[x0];
                for (uint32_t y = 0; y < ml; ++y)
                    if (((row >> y) & 1) && is_final(A, Dl[y])) acc = 1;
            }
        }
    }
    publish(p, acc);
}

__global__ void __launch_bounds__(kJoinThreads) rid_stream_join_kernel(const __grid_constant__ StreamJoinArgs p) {
    __shared__ JoinShared sh;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    stream_join(p, blockIdx.x, gridDim.x, sh);
}

// Where a chunk has very many pieces: groups of consecutive ones as one word each, a warp per group.  A group with a piece that did not merge becomes a row of tables, on the states that the piece
// before it (or, for a chunk's first group, the slots) can end in.  Bound by latency.  (64 MiB in one
// chunk: one warp of the join over its 77,824 pieces 292 us in all, and 42.6 ms where runs stay apart.)
struct StreamGroupArgs {
    StreamJoinArgs j;
    uint64_t groups;
    uint32_t per_chunk, size;                // groups per chunk, pieces per group
    uint32_t inner, n_images;                // nodes of the graph and their images
    uint32_t *out;                           // [groups]
    uint16_t *tables;                        // [groups][n]
};

__global__ void __launch_bounds__(kJoinThreads) rid_stream_group_kernel(const __grid_constant__ StreamGroupArgs p) {
    const Automaton &A = p.j.j.A;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t g = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (g >= p.groups) return;
    const uint64_t i = g / p.per_chunk;
    const uint32_t first = static_cast<uint32_t>(g - i * p.per_chunk) * p.size, s = min(p.size, p.j.per_chunk - first);
    const uint32_t *r = p.j.res + i * p.j.per_chunk + first;
    uint32_t word = chunk_word_warp(p.j, r, s, lane);
    if (word == kGeneral) {
        word = kTableResult | static_cast<uint32_t>(g);
        const uint32_t f = first ? __ldcg(r - 1) : 0, u = f & ~kNodeResult;
        const bool slots = first == 0, node = !slots && (f & kNodeResult);
        const uint32_t at = node ? __ldg(p.j.node_img + u) : 0;
        const uint32_t d = slots ? A.k : node ? (u + 1 < p.inner ? __ldg(p.j.node_img + u + 1) : p.n_images) - at : 1;
        for (uint32_t b = lane; b < d; b += 32) {
            const uint32_t x = slots ? A.slot_state[b] : node ? __ldg(p.j.images + at + b) : f & 0xFFFF;
            if (x < A.n) p.tables[g * A.n + x] = static_cast<uint16_t>(apply_pieces(p.j, r, s, x));
        }
    }
    if (lane == 0) p.out[g] = word;
}

// Short pieces: one-byte steps throughout, so a block has only the walk table to set up.  With
// `fused` the last block to finish runs the join of the whole text (one launch in all).
__global__ void __launch_bounds__(kJoinThreads) rid_stream_walk_kernel(const __grid_constant__ StreamArgs p, const __grid_constant__ StreamJoinArgs j, int fused) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ JoinShared sh;
    load_walk(p.t, smem);
    Walk w(p.t, smem_addr(smem));
    __syncthreads();
    const uint64_t t0 = reinterpret_cast<uint64_t>(p.text);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < p.t.warps) {
        for (uint32_t task = blockIdx.x * p.t.warps + warp; task * 32 < p.np; task += gridDim.x * p.t.warps) {
            const uint32_t x = task * 32 + lane;
            if (x >= p.np) break;
            uint64_t pos, end;
            piece_range(p, x, t0, pos, end);
            w.start();
            walk_blocks(w, pos, end, t0, t0 + p.len);
            p.res[x] = w.result();
        }
    }
    if (!fused) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        sh.last = atomicAdd(j.j.ticket + 1, 1) == gridDim.x - 1;
        if (sh.last) j.j.ticket[1] = 0;
    }
    __syncthreads();
    if (!sh.last) return;
    __threadfence();
    __syncthreads();
    stream_join(j, 0, 1, sh);
}

// --------------------------------------------------------------------------- host side
using StreamKernel = void (*)(StreamArgs);

template <int G, int E>
StreamKernel field_kernel(const HostStream &T) {
    return T.width == 1 ? rid_stream_kernel<kStreamField, G, E, 1> : rid_stream_kernel<kStreamField, G, E, 2>;
}

StreamKernel stream_kernel(const HostStream &T) {
    const bool b = T.entry == 1;
    switch (T.kind) {
        case kStreamField:
            return T.group == 4 ? (b ? field_kernel<4, 1>(T) : field_kernel<4, 2>(T))
                                : (b ? field_kernel<2, 1>(T) : field_kernel<2, 2>(T));
        case kStreamPair: return b ? rid_stream_kernel<kStreamPair, 2, 1, 0> : rid_stream_kernel<kStreamPair, 2, 2, 0>;
        default: return b ? rid_stream_kernel<kStreamSingle, 1, 1, 0> : rid_stream_kernel<kStreamSingle, 1, 2, 0>;
    }
}

// Chunks of more pieces are joined by groups of about the square root of their number (a launch more, 3
// us).  Merged pieces: a warp tests some 4,096 in 10 us.  Where runs stay apart every slot's run goes
// through the pieces one by one, 0.35 us each (1 MiB in 64 chunks of 256 pieces: 168 us without groups).
constexpr uint32_t kGroupFrom = 4096, kGroupApart = 32;
constexpr uint64_t kMinPiece = 64;             // bytes a piece has at least, where chunks are cut
// Pieces up to this length (and texts up to kWalkText) take one-byte steps throughout: a block then
// has only the walk table to set up, and pieces of 64 bytes are the shortest chains.  Measured with
// pieces of 64 / 96 to 192 bytes: 1 MiB in 64 chunks 30.4 / 32.6 us.  With the walk kernel / the table
// kernels: 256 KiB 29.0 / 33.3 us, 1 MiB of record lines 33.2 / 35.4, 8 MiB in 64 chunks 47.8 / 41.0.
constexpr uint64_t kWalkPiece = 96, kWalkText = 2u << 20;

}  // namespace

bool stream_takes(const HostAutomaton &H, uint64_t len, uint32_t c) {
    // (the kernels keep a warp's 32 pieces within 32-bit offsets and number pieces in 32 bits;
    // stream_shape cuts any text of up to 2^40 bytes into pieces far below that)
    return H.stream.kind != kStreamNone && c <= (1u << 26) && len <= (1ull << 40);
}

StreamShape stream_shape(const HostAutomaton &H, uint64_t len, uint32_t c, int sms) {
    StreamShape S;
    const uint64_t W = H.stream.warps;
    const double L = static_cast<double>(len) / c;
    // Pieces per chunk: the SM with the most warps of pieces decides.  A full round of W warps and a
    // rest of fewer than 14 take about as long as 14 warps do; a piece costs some 60 bytes beside
    // its own (ragged ends, graph walk).
    auto time = [&](uint64_t s) {
        const uint64_t warps = (static_cast<uint64_t>(c) * s + 31) / 32, m = (warps + sms - 1) / sms;
        const uint64_t rest = m % W;
        return static_cast<double>(m / W * W + (rest ? std::max<uint64_t>(rest, std::min<uint64_t>(14, W)) : 0)) *
               (L / static_cast<double>(s) + 60.0);
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
    if (len <= kWalkText && len / c / best > kWalkPiece / 2) {
        // a short text in pieces of some 64 bytes instead
        const uint64_t s = std::max<uint64_t>(1, len / c / kMinPiece);
        if (len / c / s <= kWalkPiece) best = s;
    }
    S.per_chunk = static_cast<uint32_t>(best);
    S.pieces = static_cast<uint64_t>(c) * best;
    S.walk_only = len <= kWalkText && len / S.pieces <= kWalkPiece;
    const uint64_t tasks = (S.pieces + 31) / 32;
    if (S.per_chunk > (H.merges ? kGroupFrom : kGroupApart)) {
        S.group = std::min<uint32_t>(256, std::max<uint32_t>(8, static_cast<uint32_t>(std::sqrt(static_cast<double>(S.per_chunk)))));
        S.groups = (S.per_chunk + S.group - 1) / S.group;
    }
    // a join block takes 256 chunks, one thread each; where chunks have many pieces, a warp each
    S.join_chunks = S.per_chunk <= 4 ? kBatch : std::min<uint32_t>(kBatch, std::max<uint32_t>(kJoinThreads / 32, (c + 1023) / 1024));
    if (S.walk_only) {
        // spread over the SMs first, then up to 8 warps a block, 4 blocks an SM
        S.block = kJoinThreads;
        S.warps = static_cast<uint32_t>(std::min<uint64_t>(kJoinThreads / 32, (tasks + sms - 1) / sms));
        S.grid = static_cast<uint32_t>(std::min<uint64_t>(static_cast<uint64_t>(sms) * 4, (tasks + S.warps - 1) / S.warps));
        S.smem = stream_walk_bytes(H);
        S.fused = !S.groups && static_cast<uint64_t>(c) * std::max<uint64_t>(1, S.per_chunk / 32) <= 64;
        if (S.fused) S.join_chunks = kBatch;
    } else {
        S.warps = static_cast<uint32_t>(std::min<uint64_t>(W, (tasks + sms - 1) / sms));
        S.block = std::max<uint32_t>(S.warps * 32, 512);       // the idle ones help to load the tables
        S.grid = static_cast<uint32_t>(std::min<uint64_t>(sms, (tasks + S.warps - 1) / S.warps));
        S.smem = stream_table_bytes(H) + (H.stream.kind == kStreamField ? 0 : S.warps * kStreamStaging);
    }
    S.join_blocks = static_cast<uint32_t>((static_cast<uint64_t>(c) + S.join_chunks - 1) / S.join_chunks);
    return S;
}

ridfa_kernel_report stream_report(const HostAutomaton &H, const StreamShape &S) {
    const HostStream &T = H.stream;
    if (S.walk_only) return {RIDFA_KERNEL_STREAM_WALK, 1, 1, 2, 1, S.per_chunk, S.block, S.grid};
    return {RIDFA_KERNEL_STREAM, T.group, T.kind == kStreamField ? 0u : 1u, T.entry, T.copies, S.per_chunk, S.block, S.grid};
}

cudaError_t stream_launch(const StreamCall &C, const StreamShape &S, cudaStream_t st) {
    const HostAutomaton &H = *C.H;
    const DeviceAutomaton &D = *C.D;
    const HostStream &T = H.stream;
    StreamArgs a{};
    a.t = stream_tables(H, D, S.walk_only, S.warps);
    a.text = C.text;
    a.len = C.len;
    a.q = C.len / C.c;
    // ceil(2^64 * (len mod c) / c): exact floors, as i * frac is off by less than i / 2^64 < 1 / c
    const uint64_t rem = C.len % C.c;
    a.frac = rem ? static_cast<uint64_t>((static_cast<unsigned __int128>(rem) << 64) / C.c) + 1 : 0;
    a.step = static_cast<uint64_t>((static_cast<unsigned __int128>(C.len) << 16) / C.c / S.per_chunk);
    a.np = static_cast<uint32_t>(S.pieces);
    a.per_chunk = S.per_chunk;
    a.res = C.res;
    const Automaton A{D.trans, D.classmap, D.final_bits, D.ifmask, D.slot_state,
                      H.n_states, H.n_classes, H.k, H.kw, H.q0_slot, H.merges};
    StreamJoinArgs j{};
    j.j = JoinArgs{A, C.c, C.maps, C.dinfo, C.work, C.partials, C.ticket, C.accept, 1, C.summary};
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
    j.status = C.status;
    j.h_accept = C.h_accept;
    j.h_status = C.h_status;
    cudaError_t e;
    if (S.walk_only) {
        // (its static and dynamic shared memory together may pass 48 KB)
        e = ensure_smem_cap(reinterpret_cast<const void *>(rid_stream_walk_kernel), 64 * 1024);
        if (e != cudaSuccess) return e;
        rid_stream_walk_kernel<<<S.grid, S.block, S.smem, st>>>(a, j, S.fused ? 1 : 0);
    } else {
        const StreamKernel kern = stream_kernel(T);
        e = ensure_smem_cap(reinterpret_cast<const void *>(kern), S.smem);
        if (e != cudaSuccess) return e;
        kern<<<S.grid, S.block, S.smem, st>>>(a);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (C.between) {
        e = cudaEventRecord(C.between, st);
        if (e != cudaSuccess) return e;
    }
    if (S.fused) return cudaSuccess;
    // the join's blocks may be set up while the last stream blocks run (they wait at their start)
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kJoinThreads);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = C.between ? 0 : 1;
    if (S.groups) {
        StreamGroupArgs g{};
        g.j = j;
        g.per_chunk = S.groups;
        g.size = S.group;
        g.groups = static_cast<uint64_t>(C.c) * S.groups;
        g.inner = H.merge.inner;
        g.n_images = static_cast<uint32_t>(H.merge.images.size());
        g.out = C.groups;
        g.tables = C.tables;
        cfg.gridDim = dim3(static_cast<unsigned>((g.groups + kJoinThreads / 32 - 1) / (kJoinThreads / 32)));
        e = cudaLaunchKernelEx(&cfg, rid_stream_group_kernel, g);
        if (e != cudaSuccess) return e;
        cfg.numAttrs = 1;
        j.res = C.groups;
        j.tables = C.tables;
        j.per_chunk = S.groups;
    }
    cfg.gridDim = dim3(S.join_blocks);
    return cudaLaunchKernelEx(&cfg, rid_stream_join_kernel, j);
}

}  // namespace ridfa

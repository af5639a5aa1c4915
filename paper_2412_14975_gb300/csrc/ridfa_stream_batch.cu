// Batched recognition by automata with a merge graph.
//
// A lane takes a piece of a text as in the single-text kernels.  The pieces of all programs of one
// table form are one list, cut into equal shares of estimated cost, one per block; a block loads a
// program's tables when its share comes to that program.  The launches of the forms run side by side,
// each on its share of the SMs.  (One kernel for all forms spilled 1.7 KB a thread; the general batch
// kernel hands out tasks of up to 16 MB by tickets, which left half of the SMs idle on batches of a GB
// over 16 programs.)  A text is accepted iff the join of its pieces' functions is: a block per text
// tests every boundary, as the single-text join does.
// Bound by the shared-memory pipe, the one-byte tables above all (2,000 texts of 0.8 GB against 16 REs:
// 789 us in the general kernels, 450 us with these and the set kernels).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "ridfa_stream.cuh"
#include "ridfa_stream_batch.h"

namespace ridfa {
namespace {

struct StreamBatchProg {
    uint32_t n;                  // states
    uint32_t kw, q0_slot, n_texts, np;
    uint32_t inner, n_images;    // nodes of the graph and their images
    const StreamBatchText *texts;
    const uint32_t *bases;
    uint32_t *res;
    const uint32_t *ifmask, *slot_alive, *final_bits, *node_img;
    const uint16_t *slot_state, *part, *node_part, *images;
};

// Instantiations, numbered: pair / single by entry size, field by bytes a lookup, entry size, width.
constexpr uint32_t kFormWalk = 255;
uint32_t form_of(const HostStream &T) {
    const uint32_t e = T.entry - 1;
    if (T.kind == kStreamPair) return e;
    if (T.kind == kStreamSingle) return 2 + e;
    return 4 + (T.group == 4 ? 4 : 0) + 2 * e + (T.width - 1);
}

// Piece x of the program: its text, found by bisection, and its range of addresses.
__device__ __forceinline__ void batch_piece(const StreamBatchProg &P, uint32_t x, uint64_t &pos, uint64_t &end, uint64_t &t0, uint64_t &t1) {
    uint32_t lo = 0, hi = P.n_texts - 1;          // last text with base <= x
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) / 2;
        if (__ldg(P.bases + mid) <= x) lo = mid;
        else hi = mid - 1;
    }
    const StreamBatchText td = P.texts[lo];
    const uint32_t t = x - td.base;
    t0 = reinterpret_cast<uint64_t>(td.text);
    t1 = t0 + td.len;
    pos = t ? (t0 + (t * td.step >> 16)) & ~static_cast<uint64_t>(31) : t0;
    end = t + 1 < td.pieces ? (t0 + ((t + 1) * td.step >> 16)) & ~static_cast<uint64_t>(31) : t1;
}

template <class S>
__device__ __forceinline__ void batch_part(const StreamBatchProg &P, const StreamTables &t, const StreamBatchPart &part, uint8_t *smem) {
    load_tables<S>(t, smem);
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp >= t.warps) return;
    const S T(t, smem_addr(smem));
    Walk w(t, smem_addr(smem));
    for (uint32_t task = part.task0 + warp; task < part.task1; task += t.warps) {
        const uint32_t x = task * 32 + lane;
        const bool have = x < P.np;
        uint64_t pos = 0, end = 0, t0 = 0, t1 = 0;
        if (have) batch_piece(P, x, pos, end, t0, t1);
        w.start();
        if constexpr (S::kStaged) {
            // the lanes whose texts lie within 2 GB of each other go together (nearly always all)
            for (uint32_t left = __ballot_sync(kFull, have); left;) {
                const bool mine = (left >> lane) & 1;
                const uint64_t key = mine ? pos : ~0ull;
                const uint32_t kh = __reduce_min_sync(kFull, static_cast<uint32_t>(key >> 32));
                const uint32_t kl = __reduce_min_sync(kFull, static_cast<uint32_t>(key >> 32) == kh ? static_cast<uint32_t>(key) : 0xFFFFFFFFu);
                const uint64_t base = (static_cast<uint64_t>(kh) << 32 | kl) & ~static_cast<uint64_t>(15);
                const bool go = mine && end - base < (1ull << 31);
                stream_staged(T, w, smem_addr(smem) + t.off_stage + warp * kWarpCoopBytes, base, go ? pos : end, end, t0, t1);
                left &= ~__ballot_sync(kFull, go);
            }
        } else {
            stream_direct(T, w, pos, end, t0, t1);
        }
        if (have) P.res[x] = w.result();
    }
}

__device__ __forceinline__ void batch_walk(const StreamBatchProg &P, const StreamTables &t, const StreamBatchPart &part, uint8_t *smem) {
    load_walk(t, smem);
    __syncthreads();
    Walk w(t, smem_addr(smem));
    for (uint32_t x = part.task0 * 32 + threadIdx.x; x < min(P.np, part.task1 * 32); x += blockDim.x) {
        uint64_t pos, end, t0, t1;
        batch_piece(P, x, pos, end, t0, t1);
        w.start();
        walk_blocks(w, pos, end, t0, t1);
        P.res[x] = w.result();
    }
}

// (the tables' arguments are kernel parameters: read again from the constant bank where they are
// needed, they take no registers through the main loops)
struct BatchTables {
    StreamTables t[kStreamBatchProgs];
};

constexpr int kBatchBlock = 768;      // (1,024 threads leave 64 registers, which spill here)

// S: the table form, or void for one-byte steps throughout.
template <class S>
__global__ void __launch_bounds__(kBatchBlock, 1) rid_stream_batch_kernel(const __grid_constant__ BatchTables tables, const StreamBatchProg *progs,
                                                                          const StreamBatchPart *parts, const uint32_t *first_part) {
    extern __shared__ __align__(128) uint8_t smem[];
    for (uint32_t i = first_part[blockIdx.x]; i < first_part[blockIdx.x + 1]; ++i) {
        const StreamBatchPart part = parts[i];
        const StreamBatchProg &P = progs[part.prog];
        const StreamTables &t = tables.t[part.prog];
        __syncthreads();                         // the last part's tables are done with
        if constexpr (std::is_void<S>::value) batch_walk(P, t, part, smem);
        else batch_part<S>(P, t, part, smem);
    }
}

// The state a piece's function takes x to (the dead state n: none).
__device__ __forceinline__ uint32_t piece_to(const StreamBatchProg &P, uint32_t f, uint32_t x) {
    const uint32_t n = P.n;
    if (x >= n) return n;
    if (f & kNodeResult) {
        const uint32_t u = f & ~kNodeResult;
        const uint16_t b = __ldg(P.part + static_cast<uint64_t>(__ldg(P.node_part + u)) * n + x);
        return b == kNoBlock ? n : __ldg(P.images + __ldg(P.node_img + u) + b);
    }
    return __ldg(P.part + static_cast<uint64_t>(f >> 16) * n + x) == kNoBlock ? n : f & 0xFFFF;
}

// Accept bits, a block per text, a piece per thread (a warp per text took 25 us on texts of up to 2,000
// pieces, one after another).  While every piece merged, piece i is entered iff if_min of piece i - 1's
// end state meets the slots alive in piece i.  With a piece that did not, the run from q0's start state
// is followed piece by piece instead: every warp takes a strip of the pieces from all states that the
// piece before the strip can end in (up to 32; repeats of one function on fixed points at once), and one
// warp strings the strips together.
// Threads a block; 1,024 where a text has very many pieces (two texts of 32 MB whose runs stay apart
// took 5.9 ms with one warp's chain).
constexpr uint32_t kBatchJoinBlock = 128, kBatchJoinMany = 4096;
__global__ void __launch_bounds__(1024) rid_stream_batch_join_kernel(const StreamBatchProg *progs, const StreamBatchText *texts,
                                                                               uint8_t *accept) {
    const uint32_t lane = threadIdx.x & 31;
    const StreamBatchText td = texts[blockIdx.x];
    const StreamBatchProg &P = progs[td.prog];
    const uint32_t n = P.n;
    const uint32_t start = __ldg(P.slot_state + P.q0_slot);
    auto final_state = [&](uint32_t s) { return s < n && ((__ldg(P.final_bits + (s >> 5)) >> (s & 31)) & 1); };
    if (td.pieces == 0) {                        // empty text: is the empty word in L?
        if (threadIdx.x == 0) accept[td.item] = final_state(start) ? 1 : 0;
        return;
    }
    const uint32_t *r = P.res + td.base;
    bool node = false, ok = true;
#pragma unroll 2
    for (uint32_t t = threadIdx.x; t < td.pieces; t += blockDim.x) {
        const uint32_t f = __ldg(r + t), y = t ? __ldg(r + t - 1) : 0;
        node = node || (f & kNodeResult);
        if (!((f | y) & kNodeResult)) {
            const uint32_t *alive = P.slot_alive + (f >> 16) * P.kw;
            uint32_t hit = 0;
            if (t == 0) hit = (__ldg(alive + (P.q0_slot >> 5)) >> (P.q0_slot & 31)) & 1;
            else if ((y & 0xFFFF) < n)
                for (uint32_t w = 0; w < P.kw; ++w) hit |= __ldg(P.ifmask + static_cast<uint64_t>(y & 0xFFFF) * P.kw + w) & __ldg(alive + w);
            ok = ok && hit && (f & 0xFFFF) < n;
        }
    }
    if (!__syncthreads_or(node)) {
        const int all = __syncthreads_and(ok);
        if (threadIdx.x == 0) accept[td.item] = all && final_state(__ldg(r + td.pieces - 1) & 0xFFFF) ? 1 : 0;
        return;
    }
    __shared__ uint32_t s_from[32][32], s_to[32][32];
    const uint32_t warp = threadIdx.x >> 5, strips = blockDim.x / 32, per = (td.pieces + strips - 1) / strips;
    // the functions r[b0, b1) on every lane's state x
    auto follow = [&](uint32_t b0, uint32_t b1, uint32_t x) {
        for (uint32_t b = b0; b < b1 && __any_sync(kFull, x < n); b += 32) {
            const uint32_t f = b + lane < b1 ? __ldg(r + b + lane) : 0;
            const uint32_t cnt = min(32u, b1 - b);
            for (uint32_t j = 0; j < cnt;) {
                const uint32_t fj = __shfl_sync(kFull, f, j);
                const uint32_t nx = piece_to(P, fj, x);
                ++j;
                if (__all_sync(kFull, nx == x)) {    // the same function again changes nothing
                    const uint32_t other = __ballot_sync(kFull, lane >= j && lane < cnt && f != fj);
                    j = other ? __ffs(other) - 1 : cnt;
                }
                x = nx;
            }
        }
        return x;
    };
    const uint32_t b0 = min(td.pieces, warp * per), b1 = min(td.pieces, b0 + per);
    const uint32_t before = warp && b0 < b1 ? __ldg(r + b0 - 1) : 0, u = before & ~kNodeResult;
    uint32_t x = n, wide = 0;
    if (warp == 0) {
        if (lane == 0) x = start;
    } else if (b0 < b1 && (before & kNodeResult)) {
        const uint32_t at = __ldg(P.node_img + u), d = (u + 1 < P.inner ? __ldg(P.node_img + u + 1) : P.n_images) - at;
        wide = d > 32;
        if (lane < d) x = __ldg(P.images + at + lane);
    } else if (b0 < b1 && lane == 0) {
        x = before & 0xFFFF;
    }
    wide = __syncthreads_or(wide);
    if (wide) {
        if (warp) return;
        x = follow(0, td.pieces, x);
        if (lane == 0) accept[td.item] = final_state(x) ? 1 : 0;
        return;
    }
    s_from[warp][lane] = x;
    s_to[warp][lane] = follow(b0, b1, x);
    __syncthreads();
    if (warp) return;
    x = s_to[0][0];
    for (uint32_t w = 1; w < strips && w * per < td.pieces && x < n; ++w) {
        const uint32_t hit = __ballot_sync(kFull, s_from[w][lane] == x);
        x = hit ? s_to[w][__ffs(hit) - 1] : n;
    }
    if (lane == 0) accept[td.item] = final_state(x) ? 1 : 0;
}

// Warps of a block that take pieces.
inline uint32_t batch_warps(const HostStream &T) { return std::min<uint32_t>(T.warps, kBatchBlock / 32); }

// Relative time per byte (per-SM rates measured on the batch of 2,000 texts against 16 REs: 12.6 bytes a
// clock for the two-byte table, 8.6 for the one-byte one, 10.7 for field codes, whose single-text
// kernel HBM holds back before an SM does).
inline double time_of(const HostStream &T) {
    return T.kind == kStreamPair ? 0.78 * T.cost : T.kind == kStreamField ? std::max(2.0f, T.cost) : T.entry == 2 ? 0.86 * T.cost : 1.2 * T.cost;
}

using BatchKernel = void (*)(BatchTables, const StreamBatchProg *, const StreamBatchPart *, const uint32_t *);
BatchKernel batch_kernel(uint32_t form) {
    switch (form) {
        case 0: return rid_stream_batch_kernel<Steps<kStreamPair, 2, 1>>;
        case 1: return rid_stream_batch_kernel<Steps<kStreamPair, 2, 2>>;
        case 2: return rid_stream_batch_kernel<Steps<kStreamSingle, 1, 1>>;
        case 3: return rid_stream_batch_kernel<Steps<kStreamSingle, 1, 2>>;
        case 4: return rid_stream_batch_kernel<Steps<kStreamField, 2, 1, 1>>;
        case 5: return rid_stream_batch_kernel<Steps<kStreamField, 2, 1, 2>>;
        case 6: return rid_stream_batch_kernel<Steps<kStreamField, 2, 2, 1>>;
        case 7: return rid_stream_batch_kernel<Steps<kStreamField, 2, 2, 2>>;
        case 8: return rid_stream_batch_kernel<Steps<kStreamField, 4, 1, 1>>;
        case 9: return rid_stream_batch_kernel<Steps<kStreamField, 4, 1, 2>>;
        case 10: return rid_stream_batch_kernel<Steps<kStreamField, 4, 2, 1>>;
        case 11: return rid_stream_batch_kernel<Steps<kStreamField, 4, 2, 2>>;
        default: return rid_stream_batch_kernel<void>;
    }
}

inline size_t al(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

}  // namespace

void plan_stream_batch(StreamBatchPlan &P, std::vector<StreamBatchSource> &src, uint32_t blocks) {
    P = StreamBatchPlan{};
    const uint32_t np = static_cast<uint32_t>(src.size());
    std::stable_sort(src.begin(), src.end(), [](const StreamBatchSource &a, const StreamBatchSource &b) {
        return form_of(a.H->stream) < form_of(b.H->stream);
    });
    std::vector<uint64_t> bytes(np, 0);
    double cost = 0, lanes = 0;
    for (uint32_t p = 0; p < np; ++p) {
        P.H.push_back(src[p].H);
        P.D.push_back(src[p].D);
        for (const auto &it : src[p].items) bytes[p] += it.len;
        P.bytes += bytes[p];
        cost += static_cast<double>(bytes[p]) * time_of(src[p].H->stream);
    }
    const auto &H = P.H;
    const auto &D = P.D;
    // One-byte steps alone where a block's share would not pay for setting up its tables (5 us a
    // program, about 150 KB through them); pieces of about 96 bytes then.  Otherwise two rounds of
    // pieces a lane, so that the shares even out.
    P.walk_only = P.bytes / blocks < 96 * 1024;
    uint64_t piece = kStreamBatchPiece;
    if (!P.walk_only) {
        for (uint32_t p = 0; p < np; ++p)
            if (cost > 0) lanes += batch_warps(H[p]->stream) * 32.0 * (static_cast<double>(bytes[p]) * time_of(H[p]->stream) / cost);
        piece = std::max<uint64_t>(1024, static_cast<uint64_t>(static_cast<double>(P.bytes) / (2.0 * blocks * std::max(lanes, 32.0))));
    }
    std::vector<double> weight(np, 0);               // cost of one task of each program
    for (uint32_t p = 0; p < np; ++p) {
        P.text0.push_back(static_cast<uint32_t>(P.texts.size()));
        P.res0.push_back(static_cast<uint32_t>(P.result_words));
        uint32_t base = 0;
        for (const auto &it : src[p].items) {
            StreamBatchText t{it.text, it.len, 0, base, 0, p, it.item};
            if (it.len) {
                t.pieces = static_cast<uint32_t>(std::max<uint64_t>(1, it.len / piece));
                t.step = static_cast<uint64_t>((static_cast<unsigned __int128>(it.len) << 16) / t.pieces);
            }
            base += t.pieces;
            P.texts.push_back(t);
            P.bases.push_back(t.base);
        }
        P.np.push_back(base);
        P.result_words += base;
        const uint32_t tasks = (base + 31) / 32;
        weight[p] = tasks ? std::max(1.0, static_cast<double>(bytes[p]) * (P.walk_only ? 1.0 : time_of(H[p]->stream)) / tasks) : 0;
    }
    // launches by table form, each on its share of the blocks
    std::vector<std::pair<uint32_t, std::vector<uint32_t>>> forms;
    for (uint32_t p = 0; p < np; ++p) {
        const uint32_t f = P.walk_only ? kFormWalk : form_of(H[p]->stream);
        if (forms.empty() || forms.back().first != f) forms.push_back({f, {}});
        forms.back().second.push_back(p);
    }
    // one block each, the others where a block's share is the largest
    std::vector<double> totals(forms.size(), 0.0);
    std::vector<uint32_t> given(forms.size(), 1);
    for (size_t fi = 0; fi < forms.size(); ++fi)
        for (uint32_t p : forms[fi].second) totals[fi] += weight[p] * ((P.np[p] + 31) / 32);
    for (size_t have = forms.size(); have < blocks && !forms.empty(); ++have) {
        size_t most = 0;
        for (size_t fi = 1; fi < forms.size(); ++fi)
            if (totals[fi] / given[fi] > totals[most] / given[most]) most = fi;
        ++given[most];
    }
    for (size_t fi = 0; fi < forms.size(); ++fi) {
        StreamBatchLaunch L;
        L.form = forms[fi].first;
        L.text0 = P.text0[forms[fi].second[0]];
        for (uint32_t p : forms[fi].second) {
            const HostAutomaton &A = *H[p];
            L.n_texts += static_cast<uint32_t>(src[p].items.size());
            for (uint32_t t = P.text0[p]; t < P.text0[p] + src[p].items.size(); ++t) L.most = std::max(L.most, P.texts[t].pieces);
            L.smem = std::max(L.smem, P.walk_only ? stream_walk_bytes(A)
                                                  : stream_table_bytes(A) + (A.stream.kind == kStreamField ? 0 : batch_warps(A.stream) * kStreamStaging));
        }
        if (!P.walk_only) L.smem = std::max(L.smem, kStreamBatchSmem);
        const double total = totals[fi];
        const uint32_t n = given[fi];
        // equal shares of the cost, block by block
        const double share = total / n;
        double left = share;
        L.first = static_cast<uint32_t>(P.first_part.size());
        L.grid = 1;
        L.block = kBatchBlock;
        P.first_part.push_back(static_cast<uint32_t>(P.parts.size()));
        for (uint32_t p : forms[fi].second) {
            const uint32_t tasks = (P.np[p] + 31) / 32;
            for (uint32_t t = 0; t < tasks;) {
                const bool last = L.grid == n;       // (rounding leaves the rest to the last)
                const uint32_t take = last ? tasks - t
                                           : static_cast<uint32_t>(std::min<double>(tasks - t, std::max(0.0, left / weight[p] + 0.5)));
                if (take) {
                    P.parts.push_back(StreamBatchPart{p, t, t + take, 0});
                    t += take;
                    left -= take * weight[p];
                }
                if (t < tasks && !last) {
                    P.first_part.push_back(static_cast<uint32_t>(P.parts.size()));
                    ++L.grid;
                    left += share;
                }
            }
        }
        P.first_part.push_back(static_cast<uint32_t>(P.parts.size()));
        P.launches.push_back(L);
    }
    // (kept by value: the plan may be enqueued long after)
    BatchTables bt{};
    for (uint32_t p = 0; p < np; ++p) bt.t[p] = stream_tables(*H[p], *D[p], P.walk_only, batch_warps(H[p]->stream));
    P.tables.resize(sizeof(bt));
    std::memcpy(P.tables.data(), &bt, sizeof(bt));
    size_t off = 0;
    P.o_progs = off;  off += al(np * sizeof(StreamBatchProg));
    P.o_texts = off;  off += al(P.texts.size() * sizeof(StreamBatchText));
    P.o_bases = off;  off += al(P.bases.size() * 4);
    P.o_parts = off;  off += al(P.parts.size() * sizeof(StreamBatchPart));
    P.o_first = off;  off += al(P.first_part.size() * 4);
    P.image_bytes = off;
}

void stream_batch_image(const StreamBatchPlan &P, uint8_t *dev, uint32_t *res, uint8_t *img) {
    StreamBatchProg *d = reinterpret_cast<StreamBatchProg *>(img + P.o_progs);
    for (size_t p = 0; p < P.H.size(); ++p) {
        const HostAutomaton &H = *P.H[p];
        const DeviceAutomaton &D = *P.D[p];
        StreamBatchProg b{};
        b.n = H.n_states;
        b.kw = H.kw;
        b.q0_slot = H.q0_slot;
        b.n_texts = (p + 1 < P.H.size() ? P.text0[p + 1] : static_cast<uint32_t>(P.texts.size())) - P.text0[p];
        b.np = P.np[p];
        b.inner = H.merge.inner;
        b.n_images = static_cast<uint32_t>(H.merge.images.size());
        b.texts = reinterpret_cast<const StreamBatchText *>(dev + P.o_texts) + P.text0[p];
        b.bases = reinterpret_cast<const uint32_t *>(dev + P.o_bases) + P.text0[p];
        b.res = res + P.res0[p];
        b.ifmask = D.ifmask;
        b.slot_alive = D.mg_slot_alive;
        b.final_bits = D.final_bits;
        b.node_img = D.mg_node_img;
        b.slot_state = D.slot_state;
        b.part = D.mg_part;
        b.node_part = D.mg_node_part;
        b.images = D.mg_images;
        d[p] = b;
    }
    std::memcpy(img + P.o_texts, P.texts.data(), P.texts.size() * sizeof(StreamBatchText));
    std::memcpy(img + P.o_bases, P.bases.data(), P.bases.size() * 4);
    if (!P.parts.empty()) std::memcpy(img + P.o_parts, P.parts.data(), P.parts.size() * sizeof(StreamBatchPart));
    std::memcpy(img + P.o_first, P.first_part.data(), P.first_part.size() * 4);
}

cudaError_t stream_batch_reach(const StreamBatchPlan &P, const StreamBatchLaunch &L, const uint8_t *dev, cudaStream_t st) {
    if (P.first_part[L.first] == P.first_part[L.first + L.grid]) return cudaSuccess;     // empty texts only
    const BatchKernel kern = batch_kernel(L.form);
    cudaError_t e = ensure_smem_cap(reinterpret_cast<const void *>(kern), L.smem);
    if (e != cudaSuccess) return e;
    BatchTables t;
    std::memcpy(&t, P.tables.data(), sizeof(t));
    kern<<<L.grid, L.block, L.smem, st>>>(t, reinterpret_cast<const StreamBatchProg *>(dev + P.o_progs),
                                          reinterpret_cast<const StreamBatchPart *>(dev + P.o_parts),
                                          reinterpret_cast<const uint32_t *>(dev + P.o_first) + L.first);
    return cudaGetLastError();
}

cudaError_t stream_batch_join(const StreamBatchPlan &P, const StreamBatchLaunch &L, const uint8_t *dev, uint8_t *d_accept, cudaStream_t st) {
    rid_stream_batch_join_kernel<<<L.n_texts, L.most > kBatchJoinMany ? 1024 : kBatchJoinBlock, 0, st>>>(reinterpret_cast<const StreamBatchProg *>(dev + P.o_progs),
                                                                       reinterpret_cast<const StreamBatchText *>(dev + P.o_texts) + L.text0,
                                                                       d_accept);
    return cudaGetLastError();
}

}  // namespace ridfa

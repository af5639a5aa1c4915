// Per-chunk join states: the full scan of the join (Sec. 3.2) instead of its reduction.
//
// For every chunk i the entry set E_i = if_min(PLAS_{i-1}) ∩ PIS_i (E_1 = {q0's slot} ∩ PIS_1),
// i.e. the interface slots through which chunk i is entered on the way to PLAS_i = λ_i(E_i), and
// the first chunk whose PLAS_i is empty (the text is rejected there).
//
// While every chunk has at most one end state (runs that merge), E_i does not depend on how the
// chunks before i - 1 went, only on whether PLAS_{i-1} is empty: one warp per row works out every
// E_i as if it were not, the first empty one is where the text is rejected, and the sets after it
// are cleared.  Otherwise PLAS_i = PLAS_{i-1} · M_i over the distinct end states D_i of each chunk
// (M_i as in the join kernel):
//   1. a warp per boundary forms M_i;
//   2. a warp per segment of kScanSeg boundaries multiplies them, a row of the product per lane;
//   3. one block: the incoming PLAS vector of every segment;
//   4. a warp per segment walks its boundaries from that vector;
//   5. a warp per chunk forms E_i from PLAS_{i-1}.
// Boundaries go through these launches kScanTile at a time, so that the matrices take 35 MB at most, however many
// chunks there are.
// When some chunk has more than 32 distinct end states, one block propagates the k-bit sets
// chunk by chunk instead (exact, sequential in c).
//
// Record lines, 65,537 chunks of 68 slots: a whole call 1,750 us with one thread walking 64 rows at a
// time (every row sorted entry by entry, twice), 39 us by the first form; the codon RE, 65,536
// chunks with several end states, 197 us by the second.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ridfa_internal.h"
#include "ridfa_kernels.cuh"

namespace ridfa {
namespace {

constexpr uint32_t kScanSeg = 32;          // boundaries per warp of launches 2 and 4
constexpr uint32_t kScanThreads = 256;
constexpr uint32_t kScanWarps = kScanThreads / 32;
constexpr uint32_t kScanRows = 8;          // consecutive rows per warp of rid_scan_rows
constexpr uint32_t kStatusSeveral = 8u;    // some chunk has two or more end states
constexpr uint32_t kScanTile = 1u << 18;   // boundaries that launches 1 to 5 take at a time (2^20 chunks of the
                                           // codon RE: 2,530 us in one, 2,546 in 4 tiles, 2,910 in 16)
constexpr int kScanRegs = RIDFA_MAX_SLOTS / 32;

struct ScanArgs {
    Automaton A;
    const uint16_t *maps;      // [c][k]
    uint32_t c;
    uint32_t first, end, nseg; // boundaries [first, end) of this tile, in nseg segments
    uint32_t *mats;            // [boundary - first][32]: row z of M_i, bits over D_i
    uint32_t *prods;           // [nseg][32]
    uint32_t *vin;             // [nseg]: PLAS before the segment's first boundary, over its D
    uint32_t *plas;            // [1 + kScanTile]: PLAS_i as bits over D_i, i from first - 1
    uint32_t *entry;           // [c][kw], or null
    unsigned long long *reject;
    uint32_t *status;
};

// Row i across the warp: lane l holds entries l, 32 + l, ...
__device__ __forceinline__ void load_row(const ScanArgs &p, uint64_t i, uint32_t lane, uint32_t (&v)[kScanRegs]) {
    const uint16_t *row = p.maps + i * p.A.k;
#pragma unroll
    for (int r = 0; r < kScanRegs; ++r) {
        const uint32_t a = r * 32 + lane;
        v[r] = a < p.A.k ? __ldg(row + a) : kUndef;
    }
}

// The distinct defined values of a row, ascending: lane g gets the g-th; returns their number
// (kMaxD + 1: more than kMaxD).
__device__ __forceinline__ uint32_t warp_distinct(const uint32_t (&v)[kScanRegs], uint32_t lane, uint32_t &mine) {
    uint32_t cnt = 0, cur = 0;
    mine = kUndef;
    for (;;) {
        uint32_t m = 0xFFFFFFFFu;
#pragma unroll
        for (int r = 0; r < kScanRegs; ++r)
            if (v[r] != kUndef && (cnt == 0 || v[r] > cur)) m = min(m, v[r]);
        m = __reduce_min_sync(kFull, m);
        if (m == 0xFFFFFFFFu) return cnt;
        if (cnt == static_cast<uint32_t>(kMaxD)) return kMaxD + 1;
        if (lane == cnt) mine = m;
        cur = m;
        ++cnt;
    }
}

// Word `lane` of the row's set of defined slots (lanes below kw).
__device__ __forceinline__ uint32_t alive_word(const uint32_t (&v)[kScanRegs], uint32_t lane) {
    uint32_t alive = 0;
#pragma unroll
    for (int r = 0; r < kScanRegs; ++r) {
        const uint32_t b = __ballot_sync(kFull, v[r] != kUndef);
        if (lane == static_cast<uint32_t>(r)) alive = b;
    }
    return alive;
}

// The case of at most one end state per chunk, a warp per kScanRows rows: E_i as if PLAS_{i-1} were
// not empty, and the first empty one.  Bound by the maps' bytes (L2 or HBM).
__global__ void __launch_bounds__(kScanThreads) rid_scan_rows(ScanArgs p) {
    const Automaton &A = p.A;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t i0 = (static_cast<uint64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5)) * kScanRows;
    if (i0 >= p.c) return;
    const uint64_t i1 = min(static_cast<uint64_t>(p.c), i0 + kScanRows);
    uint32_t v[kScanRegs], y = kUndef;       // y: the previous chunk's end state
    uint32_t bad = 0;
    auto only = [&]() -> uint32_t {          // the row's one defined value
        uint32_t lo = 0xFFFFFFFFu, hi = 0;
#pragma unroll
        for (int r = 0; r < kScanRegs; ++r)
            if (v[r] != kUndef) {
                lo = min(lo, v[r]);
                hi = max(hi, v[r]);
            }
        lo = __reduce_min_sync(kFull, lo);
        hi = __reduce_max_sync(kFull, hi);
        if (lo == 0xFFFFFFFFu) return kUndef;
        if (lo != hi) bad |= kStatusSeveral;
        if (hi >= A.n) bad |= kStatusBad;
        return min(lo, A.n);
    };
    if (i0) {
        load_row(p, i0 - 1, lane, v);
        y = only();
    }
    for (uint64_t i = i0; i < i1; ++i) {
        load_row(p, i, lane, v);
        uint32_t in = 0;                     // word `lane` of if_min of the previous end state
        if (lane < A.kw) {
            if (i == 0) in = (A.q0_slot >> 5) == lane ? 1u << (A.q0_slot & 31) : 0u;
            else if (y != kUndef) in = __ldg(A.ifmask + static_cast<uint64_t>(y) * A.kw + lane);
        }
        const uint32_t e = in & alive_word(v, lane);
        if (p.entry && lane < A.kw) p.entry[i * A.kw + lane] = e;
        if (!__any_sync(kFull, e != 0) && lane == 0) atomicMin(p.reject, static_cast<unsigned long long>(i));
        y = only();
    }
    if (bad && lane == 0) atomicOr(p.status, bad);
}

// ... and the sets after the first empty one.
__global__ void __launch_bounds__(kScanThreads) rid_scan_clear(ScanArgs p) {
    const unsigned long long f = *p.reject;
    if (f >= p.c) return;
    const uint64_t lo = (f + 1) * p.A.kw, hi = static_cast<uint64_t>(p.c) * p.A.kw;
    for (uint64_t e = lo + static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < hi; e += static_cast<uint64_t>(gridDim.x) * blockDim.x)
        p.entry[e] = 0;
}

// Launch 1: M_i, a warp per boundary.
__global__ void __launch_bounds__(kScanThreads) rid_scan_matrices(ScanArgs p) {
    __shared__ uint8_t s_idx[kScanWarps][RIDFA_MAX_SLOTS];
    const Automaton &A = p.A;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t i = p.first + static_cast<uint64_t>(blockIdx.x) * kScanWarps + warp;
    if (i >= p.end) return;
    uint32_t v[kScanRegs], prev, mine;
    load_row(p, i - 1, lane, v);
    const uint32_t mp = warp_distinct(v, lane, prev);
    load_row(p, i, lane, v);
    const uint32_t mc = warp_distinct(v, lane, mine);
    if (mp > static_cast<uint32_t>(kMaxD) || mc > static_cast<uint32_t>(kMaxD)) {
        if (lane == 0) atomicOr(p.status, kStatusWide);
        return;
    }
    // each slot's place in D_i
    uint32_t idx[kScanRegs];
#pragma unroll
    for (int r = 0; r < kScanRegs; ++r) idx[r] = 0xFF;
    for (uint32_t g = 0; g < mc; ++g) {
        const uint32_t d = __shfl_sync(kFull, mine, g);
#pragma unroll
        for (int r = 0; r < kScanRegs; ++r)
            if (v[r] == d) idx[r] = g;
    }
#pragma unroll
    for (int r = 0; r < kScanRegs; ++r) s_idx[warp][r * 32 + lane] = static_cast<uint8_t>(idx[r]);
    __syncwarp();
    uint32_t row = 0;
    if (lane < mp) {
        if (prev >= A.n) atomicOr(p.status, kStatusBad);
        else
            for (uint32_t w = 0; w < A.kw; ++w)
                for (uint32_t bits = __ldg(A.ifmask + static_cast<uint64_t>(prev) * A.kw + w); bits; bits &= bits - 1) {
                    const uint32_t g = s_idx[warp][w * 32 + __ffs(bits) - 1];
                    if (g != 0xFF) row |= 1u << g;
                }
    }
    p.mats[(i - p.first) * 32 + lane] = row;
}

// rows <- rows · M, a row per lane; m: the lane's row of M.
__device__ __forceinline__ uint32_t times(uint32_t row, uint32_t m) {
    uint32_t out = 0;
    for (uint32_t nz = __ballot_sync(kFull, m != 0); nz; nz &= nz - 1) {
        const uint32_t z = __ffs(nz) - 1, mz = __shfl_sync(kFull, m, z);
        if ((row >> z) & 1) out |= mz;
    }
    return out;
}

// v · M for a vector that every lane holds.
__device__ __forceinline__ uint32_t vec_times(uint32_t v, uint32_t m, uint32_t lane) {
    return __reduce_or_sync(kFull, (v >> lane) & 1 ? m : 0u);
}

// Launch 2: the product of each segment's matrices.
__global__ void __launch_bounds__(kScanThreads) rid_scan_products(ScanArgs p) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t sg = blockIdx.x * kScanWarps + (threadIdx.x >> 5);
    if (sg >= p.nseg) return;
    const uint32_t b0 = sg * kScanSeg, b1 = min(p.end - p.first, b0 + kScanSeg);
    uint32_t row = 1u << lane, m = p.mats[b0 * 32 + lane];
    for (uint32_t i = b0; i < b1; ++i) {
        const uint32_t next = i + 1 < b1 ? p.mats[(i + 1) * 32 + lane] : 0;
        row = times(row, m);
        m = next;
    }
    p.prods[static_cast<uint64_t>(sg) * 32 + lane] = row;
}

// Launch 3 (one block of 32 warps): the incoming PLAS vector of every segment; in the first tile, PLAS and
// entry set of chunk 0.
__global__ void __launch_bounds__(1024) rid_scan_prefix(ScanArgs p) {
    __shared__ uint32_t s_tot[32][32], s_in[32];
    const Automaton &A = p.A;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t per = (p.nseg + 31) / 32, s0 = min(p.nseg, warp * per), s1 = min(p.nseg, s0 + per);
    // (four products are loaded together: one after the other, the loads' latency was the time)
    auto load4 = [&](uint32_t sg, uint32_t (&m)[4]) {
#pragma unroll
        for (int u = 0; u < 4; ++u) m[u] = sg + u < s1 ? p.prods[static_cast<uint64_t>(sg + u) * 32 + lane] : 0;
    };
    uint32_t row = 1u << lane;
    for (uint32_t sg = s0; sg < s1; sg += 4) {
        uint32_t m[4];
        load4(sg, m);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (sg + u < s1) row = times(row, m[u]);
    }
    s_tot[warp][lane] = row;
    __syncthreads();
    if (warp == 0) {
        uint32_t x;
        if (p.first > 1) {
            x = p.plas[kScanTile];               // (the tile before was a whole one)
        } else {
            // PLAS_1 = {λ_1(q0)} over D_1 (chunk 0 here); E_1 = {q0's slot} if that move is defined
            uint32_t v[kScanRegs], mine;
            load_row(p, 0, lane, v);
            const uint32_t m0 = warp_distinct(v, lane, mine);
            const uint32_t v0 = p.maps[A.q0_slot];
            x = m0 <= static_cast<uint32_t>(kMaxD) ? __ballot_sync(kFull, v0 != kUndef && lane < m0 && mine == v0) : 0;
            if (p.entry && lane < A.kw) p.entry[lane] = (v0 != kUndef && (A.q0_slot >> 5) == lane) ? 1u << (A.q0_slot & 31) : 0u;
            if (lane == 0 && v0 == kUndef) atomicMin(p.reject, 0ull);
        }
        if (lane == 0) p.plas[0] = x;
        for (uint32_t t = 0; t < 32; ++t) {
            if (lane == 0) s_in[t] = x;
            x = vec_times(x, s_tot[t][lane], lane);
        }
    }
    __syncthreads();
    uint32_t v = s_in[warp];
    for (uint32_t sg = s0; sg < s1; sg += 4) {
        uint32_t m[4];
        load4(sg, m);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (sg + u < s1) {
                if (lane == 0) p.vin[sg + u] = v;
                v = vec_times(v, m[u], lane);
            }
    }
}

// Launch 4: PLAS after every boundary of a segment.
__global__ void __launch_bounds__(kScanThreads) rid_scan_walk(ScanArgs p) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t sg = blockIdx.x * kScanWarps + (threadIdx.x >> 5);
    if (sg >= p.nseg) return;
    const uint32_t b0 = sg * kScanSeg, b1 = min(p.end - p.first, b0 + kScanSeg);
    uint32_t v = p.vin[sg], keep = 0, m = p.mats[b0 * 32 + lane];
    for (uint32_t i = b0; i < b1; ++i) {
        const uint32_t next = i + 1 < b1 ? p.mats[(i + 1) * 32 + lane] : 0;
        const uint32_t nv = vec_times(v, m, lane);
        if (nv == 0 && v != 0 && lane == 0) atomicMin(p.reject, static_cast<unsigned long long>(p.first) + i);
        if (lane == i - b0) keep = nv;
        v = nv;
        m = next;
    }
    if (b0 + lane < b1) p.plas[b0 + lane + 1] = keep;
}

// Launch 5: E_i from PLAS_{i-1}, a warp per chunk.
__global__ void __launch_bounds__(kScanThreads) rid_scan_entries(ScanArgs p) {
    const Automaton &A = p.A;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t i = p.first + static_cast<uint64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5);
    if (i >= p.end) return;
    const uint32_t plas = p.plas[i - p.first];
    uint32_t e = 0;
    if (plas) {
        uint32_t v[kScanRegs], prev;
        load_row(p, i - 1, lane, v);
        warp_distinct(v, lane, prev);
        load_row(p, i, lane, v);
        const uint32_t alive = alive_word(v, lane);
        for (uint32_t w = 0; w < A.kw; ++w) {
            const uint32_t in = __reduce_or_sync(kFull, ((plas >> lane) & 1) && prev < A.n ? __ldg(A.ifmask + static_cast<uint64_t>(prev) * A.kw + w) : 0u);
            if (lane == w) e = in & alive;
        }
    }
    if (lane < A.kw) p.entry[i * A.kw + lane] = e;
}

// Some chunk has more than kMaxD end states: one block propagates the k-bit slot sets.
__global__ void __launch_bounds__(kScanThreads) rid_scan_wide(ScanArgs p) {
    __shared__ uint32_t s_vec[RIDFA_MAX_SLOTS / 32], s_nvec[RIDFA_MAX_SLOTS / 32];
    __shared__ uint32_t s_any;
    const Automaton &A = p.A;
    const uint32_t tid = threadIdx.x;
    for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_vec[w] = (A.q0_slot >> 5) == w ? 1u << (A.q0_slot & 31) : 0u;
    __syncthreads();
    for (uint64_t i = 0; i < p.c; ++i) {
        const uint16_t *row = p.maps + i * A.k;
        for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_nvec[w] = 0;
        if (tid == 0) s_any = 0;
        __syncthreads();
        // entry set E_i = s_vec ∩ PIS_i; next slots = if_min(λ_i(E_i))
        for (uint32_t a = tid; a < A.k; a += blockDim.x) {
            const bool in = (s_vec[a >> 5] >> (a & 31)) & 1;
            if (!in || row[a] == kUndef) continue;
            if (row[a] >= A.n) {
                atomicOr(p.status, kStatusBad);
                continue;
            }
            s_any = 1;
            for (uint32_t w = 0; w < A.kw; ++w) {
                const uint32_t m = A.ifmask[static_cast<uint64_t>(row[a]) * A.kw + w];
                if (m) atomicOr(&s_nvec[w], m);
            }
        }
        __syncthreads();
        if (p.entry)
            for (uint32_t w = tid; w < A.kw; w += blockDim.x) {
                uint32_t live = 0;
                for (uint32_t b = 0; b < 32; ++b) {
                    const uint32_t a = w * 32 + b;
                    if (a < A.k && ((s_vec[w] >> b) & 1) && row[a] != kUndef) live |= 1u << b;
                }
                p.entry[i * A.kw + w] = live;
            }
        if (tid == 0 && !s_any) atomicMin(p.reject, static_cast<unsigned long long>(i));
        __syncthreads();
        for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_vec[w] = s_nvec[w];
        __syncthreads();
    }
}

}  // namespace
}  // namespace ridfa

extern "C" int ridfa_join_scan(const ridfa_program *prog, const uint16_t *d_maps, uint32_t n_chunks,
                               uint32_t *d_entry, int64_t *h_reject, void *stream) {
    using namespace ridfa;
    if (!prog || !d_maps || !h_reject || n_chunks == 0) return RIDFA_E_ARG;
    const HostAutomaton &H = prog->rid;
    if (H.k > RIDFA_MAX_SLOTS) return RIDFA_E_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    ScanArgs a{};
    struct Space {                               // given back once nothing of the call is in flight
        const ridfa_program *prog;
        int dev;
        cudaStream_t st;
        ScanSpace sp;
        bool idle = true;
        ~Space() {
            if (!idle) cudaStreamSynchronize(st);
            std::lock_guard<std::mutex> lock(prog->mu);
            scan_give(prog, dev, sp);
        }
    } space{prog, dev, st, {}};
    int err = RIDFA_OK;
    {
        std::lock_guard<std::mutex> lock(prog->mu);
        const DeviceAutomaton *D = device_copy(prog, false, dev, &err);
        if (!D) return err;
        a.A = Automaton{D->trans, D->classmap, D->final_bits, D->ifmask, D->slot_state, H.n_states, H.n_classes,
                        H.k, H.kw, H.q0_slot};
        err = scan_take(prog, dev, &space.sp);
    }
    // the result words: {first rejecting chunk, status}, on the device and page-locked on the host
    if (err == RIDFA_OK) err = scan_grow(&space.sp, 0);
    if (err != RIDFA_OK) return err;
    const uint32_t c = n_chunks;
    uint64_t *words = nullptr;
    const uint64_t *h = space.sp.host;
    auto place = [&]() {
        words = static_cast<uint64_t *>(space.sp.base);
        a.reject = reinterpret_cast<unsigned long long *>(words);
        a.status = reinterpret_cast<uint32_t *>(words + 1);
    };
    place();
    a.maps = d_maps;
    a.c = c;
    a.entry = d_entry;
    auto blocks = [](uint64_t items, uint64_t per) { return static_cast<unsigned>((items + per - 1) / per); };
    auto fetch = [&]() {
        e = cudaMemcpyAsync(space.sp.host, words, 16, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        space.idle = e == cudaSuccess;
        return e;
    };
    auto clear = [&]() {
        space.idle = false;
        e = cudaMemsetAsync(words, 0xFF, 8, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(words + 1, 0, 8, st);
        return e;
    };
    if (clear() != cudaSuccess) return cuda_fail(e);
    rid_scan_rows<<<blocks(c, kScanWarps * kScanRows), kScanThreads, 0, st>>>(a);
    if (d_entry) rid_scan_clear<<<blocks(static_cast<uint64_t>(c) * H.kw, 4096) < 608 ? blocks(static_cast<uint64_t>(c) * H.kw, 4096) : 608, kScanThreads, 0, st>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) fetch();
    if (e != cudaSuccess) return cuda_fail(e);
    uint32_t status = static_cast<uint32_t>(h[1]);
    if (status & kStatusSeveral) {
        const size_t tile = std::min<size_t>(kScanTile, c - 1), segs = (tile + kScanSeg - 1) / kScanSeg;
        const size_t bytes = (tile * 32 + segs * 33 + kScanTile + 1) * 4;
        err = scan_grow(&space.sp, bytes);
        if (err != RIDFA_OK) return err;
        place();
        if (clear() != cudaSuccess) return cuda_fail(e);
        a.mats = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(space.sp.base) + 256);
        a.prods = a.mats + tile * 32;
        a.vin = a.prods + segs * 32;
        a.plas = a.vin + segs;
        uint64_t at = 1;
        do {                                     // (one tile without boundaries where there is one chunk)
            a.first = static_cast<uint32_t>(at);
            a.end = static_cast<uint32_t>(std::min<uint64_t>(c, at + kScanTile));
            const uint32_t n = a.end - a.first;
            a.nseg = (n + kScanSeg - 1) / kScanSeg;
            if (n) {
                rid_scan_matrices<<<blocks(n, kScanWarps), kScanThreads, 0, st>>>(a);
                rid_scan_products<<<blocks(a.nseg, kScanWarps), kScanThreads, 0, st>>>(a);
            }
            rid_scan_prefix<<<1, 1024, 0, st>>>(a);
            if (n) {
                rid_scan_walk<<<blocks(a.nseg, kScanWarps), kScanThreads, 0, st>>>(a);
                if (d_entry) rid_scan_entries<<<blocks(n, kScanWarps), kScanThreads, 0, st>>>(a);
            }
            e = cudaGetLastError();
            at = a.end;
        } while (e == cudaSuccess && at < c);
        if (e == cudaSuccess) fetch();
        if (e != cudaSuccess) return cuda_fail(e);
        status = static_cast<uint32_t>(h[1]);
        if (status & kStatusWide) {
            if (clear() != cudaSuccess) return cuda_fail(e);
            rid_scan_wide<<<1, kScanThreads, 0, st>>>(a);
            e = cudaGetLastError();
            if (e == cudaSuccess) fetch();
            if (e != cudaSuccess) return cuda_fail(e);
            status = static_cast<uint32_t>(h[1]);
        }
    }
    if (status & kStatusBad) return RIDFA_E_STATE;
    *h_reject = h[0] == ~0ull ? -1 : static_cast<int64_t>(h[0]);
    return RIDFA_OK;
}

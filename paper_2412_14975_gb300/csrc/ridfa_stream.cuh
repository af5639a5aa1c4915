// Device building blocks of the stream kernels, shared by the single-text kernels (ridfa_stream.cu)
// and the batched one (ridfa_stream_batch.cu): the walk through the merge graph, the table steps of
// merged runs, and the two ways of reading a lane's text.
#pragma once

#include "ridfa_kernels.cuh"

namespace ridfa {
namespace {

constexpr uint32_t kNodeResult = 0x80000000u;   // a piece that ended in an inner node
constexpr uint32_t kGlobal = 0xFFFFFFFFu;       // a ragged-end table left in global memory
constexpr int kStreamBlock = 1024;

// The tables of one automaton and where a block puts them (dynamic shared memory).
struct StreamTables {
    uint32_t warps;               // warps of a block that take pieces (all of them load the tables)
    const uint16_t *walk, *edge_pid;
    const uint8_t *classmap;
    const uint32_t *code, *words;
    uint32_t n, C, n_walk;        // n_walk: entries of the walk table
    uint32_t n_words, copies, row;                       // row: bytes per state
    // field codes: byte of code 0 (four times) and what each field bit and both add to it; where the
    // codes of bytes 0.. (and 2.. for two-byte lookups) gather; column -> byte offset
    // (second: mask of the field's second bit, 0 in a field of one)
    uint32_t shift, second, canon0, d1, d2, d12, mul, mul_h, take_bits, part_mask, col_mul, part_mul;
    uint32_t off_table, off_walk, off_cls, off_stage;
};


// A lane between bytes, and the one-byte steps that everything outside whole granules of a merged
// run takes: the graph walk, ragged starts and ends.  id: a state (id <= n, one run left), or a
// node of the graph (id - n - 1); edge: the last step taken from a node, which names the leaf.
struct Walk {
    const StreamTables &p;
    uint32_t cls, tab;           // shared addresses of the byte classes and of the walk table
    uint32_t id, edge;
    __device__ __forceinline__ Walk(const StreamTables &args, uint32_t base) : p(args), cls(base + args.off_cls), tab(base + args.off_walk) {}
    __device__ __forceinline__ void start() {
        id = p.n + 1;
        edge = 0;
    }
    __device__ __forceinline__ bool merged() const { return id <= p.n; }
    __device__ __forceinline__ bool dead() const { return id == p.n; }
    __device__ __forceinline__ uint32_t class_of(uint32_t b) const { return lds_u8(cls + b); }
    __device__ __forceinline__ void step_class(uint32_t c) {
        const uint32_t at = id * p.C + c;
        edge = id > p.n ? at : edge;
        id = p.off_walk != kGlobal ? lds_u16(tab + 2 * at) : __ldg(p.walk + at);
    }
    // bytes [lo, hi) of 4 * N bytes: the classes are looked up ahead of the dependent steps
    template <int N>
    __device__ __forceinline__ void take(const uint32_t (&w)[N], int lo, int hi) {
        uint32_t c[4 * N];
#pragma unroll
        for (int i = 0; i < 4 * N; ++i) c[i] = class_of((w[i >> 2] >> (8 * (i & 3))) & 0xFF);
        if (lo <= 0 && hi >= 4 * N) {
#pragma unroll
            for (int i = 0; i < 4 * N; ++i) step_class(c[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 4 * N; ++i)
                if (i >= lo && i < hi) step_class(c[i]);
        }
    }
    __device__ __forceinline__ uint32_t result() const {
        if (!merged()) return kNodeResult | (id - p.n - 1);
        return static_cast<uint32_t>(__ldg(p.edge_pid + (edge - (p.n + 1) * p.C))) << 16 | id;
    }
};

template <int E>
__device__ __forceinline__ uint32_t lds_entry(uint32_t a) {
    return E == 1 ? lds_u8(a) : lds_u16(a);
}

// Table steps of a merged run.  KIND, G (bytes a lookup) and W (field bits) as in HostStream, E: bytes
// per entry.
template <int KIND, int G, int E, int W = 0>
struct Steps {
    static constexpr bool kStaged = KIND != kStreamField;
    const StreamTables &p;         // (kernel parameters: constant operands, not registers)
    uint32_t lc, lt;             // this lane's class codes; its copy of the table
    __device__ __forceinline__ Steps(const StreamTables &args, uint32_t base) : p(args) {
        const uint32_t lane = threadIdx.x & 31;
        lc = base + lane * 4;
        lt = base + p.off_table + (lane & (p.copies - 1)) * 4;
    }
    // one lookup of G bytes whose codes a multiplication gathered in the top bits of g
    __device__ __forceinline__ uint32_t column_step(uint32_t s, uint32_t g) const {
        const uint32_t col = __umulhi(g, p.take_bits);           // (a shift on the multiplier's pipe)
        return lds_entry<E>(s * p.row + (col * p.col_mul + ((col & p.part_mask) * p.part_mul + lt)));
    }
    // address of the class codes of byte q: mask the byte where it is, then one multiply-add for the
    // shift and the base (the logic pipe is the busier one)
    __device__ __forceinline__ uint32_t code_at(const uint32_t *w, int q) const {
        const uint32_t x = w[q >> 2] & (0xFFu << (8 * (q & 3)));
        if ((q & 3) == 0) return x * 128 + lc;
        uint32_t a;
        asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(a) : "r"(x), "r"(1u << (39 - 8 * (q & 3))), "r"(lc));
        return a;
    }
    // N 32-bit words of text
    template <int N>
    __device__ __forceinline__ uint32_t take(uint32_t s, const uint32_t (&w)[N]) const {
        if constexpr (KIND == kStreamField) {
            // The field of all four bytes is masked out (m) and the codes of a lookup's bytes are
            // gathered by one multiplication (no two partial products share a bit).  Each byte is
            // rebuilt from its field bits by multiplications, which share the work with the logic
            // pipe; a byte that differs is outside the alphabet, and its run is dead after it.
            uint32_t bad = 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint32_t f = w[i] >> p.shift;
                const uint32_t m1 = f & 0x01010101u;
                uint32_t m = m1, whole = m1 * p.d1 + p.canon0;
                if (W == 2) {
                    const uint32_t m2 = (w[i] >> (p.shift + 1)) & 0x01010101u;
                    m = f & 0x03030303u;
                    whole += m2 * p.d2 + (m1 & m2) * p.d12;
                }
                bad |= whole ^ w[i];
                s = column_step(s, m * p.mul);
                if (G == 2) s = column_step(s, m * p.mul_h);
            }
            return bad ? p.n : s;
        } else if constexpr (KIND == kStreamPair) {
            uint32_t x[2 * N];
#pragma unroll
            for (int i = 0; i < 2 * N; ++i)
                x[i] = lds_u16(code_at(w, 2 * i)) + lds_u16(code_at(w, 2 * i + 1) + 2) + lt;
#pragma unroll
            for (int i = 0; i < 2 * N; ++i) s = lds_entry<E>(s * p.row + x[i]);
            return s;
        } else {
            uint32_t x[4 * N];
#pragma unroll
            for (int i = 0; i < 4 * N; ++i) x[i] = lds_u32(code_at(w, i)) + lt;
#pragma unroll
            for (int i = 0; i < 4 * N; ++i) s = lds_entry<E>(s * p.row + x[i]);
            return s;
        }
    }
};

// The one-byte tables in shared memory (a large walk table stays in global memory).
__device__ __forceinline__ void load_walk(const StreamTables &p, uint8_t *smem) {
    const uint32_t base = smem_addr(smem);
    for (uint32_t i = threadIdx.x; i < 64; i += blockDim.x)
        sts_u32(base + p.off_cls + 4 * i, __ldg(reinterpret_cast<const uint32_t *>(p.classmap) + i));
    if (p.off_walk != kGlobal)
        for (uint32_t i = threadIdx.x; i < p.n_walk / 2; i += blockDim.x)
            sts_u32(base + p.off_walk + 4 * i, __ldg(reinterpret_cast<const uint32_t *>(p.walk) + i));
}

// Shared-memory tables of a block: class codes (32 lane copies), the main table in its lane copies,
// and the one-byte tables of the ragged ends.
template <class S>
__device__ __forceinline__ void load_tables(const StreamTables &p, uint8_t *smem) {
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
    } else if (p.copies == 2) {
        for (uint32_t i = threadIdx.x; i < p.n_words; i += nt) {
            const uint32_t v = __ldg(p.words + i);
            sts_u32(base + p.off_table + i * 8, v);
            sts_u32(base + p.off_table + i * 8 + 4, v);
        }
    } else {
        // one copy, as it is: 16 bytes a thread (the upload is padded to whole ones)
#pragma unroll 4
        for (uint32_t i = threadIdx.x; i < (p.n_words + 3) / 4; i += nt) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p.words) + i);
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(base + p.off_table + i * 16), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
        }
    }
    load_walk(p, smem);
}

// Text through 32-byte loads of each lane's own piece: an L1 line per lane and load, so 1.2 LSU
// cycles per 32 text bytes; worth it where the lookups take less than one.
__device__ __forceinline__ void load32(const uint8_t *a, uint32_t (&w)[8]) {
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(a));
}

// One-byte steps over [pos, end) by 32-byte blocks of the text, one block ahead.
__device__ __forceinline__ void walk_blocks(Walk &w, uint64_t pos, uint64_t end, uint64_t t0, uint64_t t1) {
    uint32_t cur[8], nxt[8];
    uint64_t a = pos & ~static_cast<uint64_t>(31);
    auto inside = [&](uint64_t x) { return x >= t0 && x + 32 <= t1; };
    if (pos < end && inside(a)) load32(reinterpret_cast<const uint8_t *>(a), cur);
    while (pos < end && !w.dead()) {
        const uint64_t b = min(end, a + 32);
        if (b < end && inside(a + 32)) load32(reinterpret_cast<const uint8_t *>(a + 32), nxt);
        if (inside(a)) {
            int lo = static_cast<int>(pos - a), hi = static_cast<int>(b - a);
#pragma unroll 1
            for (int h = 0; h < 4; ++h, lo -= 8, hi -= 8) {       // (the block moves down 8 bytes a turn)
                const uint32_t v[2] = {cur[0], cur[1]};
                if (lo < 8 && hi > 0) w.take(v, lo, hi);
#pragma unroll
                for (int i = 0; i < 6; ++i) cur[i] = cur[i + 2];
            }
            pos = b;
        } else {
            while (pos < b) w.step_class(w.class_of(__ldg(reinterpret_cast<const uint8_t *>(pos++))));
        }
        a += 32;
#pragma unroll
        for (int i = 0; i < 8; ++i) cur[i] = nxt[i];
    }
}

// One-byte steps over [pos, end), until the end or -- with `to_block` -- until one run is left at a
// 32-byte boundary: the few ragged bytes at the ends of a long piece, by 8-byte words, with little held in registers beside the main loop's blocks.
__device__ __forceinline__ void walk_ends(Walk &w, uint64_t &pos, uint64_t end, uint64_t t0, uint64_t t1, bool to_block) {
#pragma unroll 1
    while (pos < end && !w.dead() && !(to_block && w.merged() && !(pos & 31))) {
        const uint64_t a = pos & ~static_cast<uint64_t>(7);
        if (a >= t0 && a + 8 <= t1) {
            const uint2 x = __ldg(reinterpret_cast<const uint2 *>(a));
            const uint32_t v[2] = {x.x, x.y};
            const int lo = static_cast<int>(pos & 7), hi = static_cast<int>(min(static_cast<uint64_t>(8), end - a));
            w.take(v, lo, hi);
            pos += hi - lo;
        } else {
            w.step_class(w.class_of(__ldg(reinterpret_cast<const uint8_t *>(pos++))));
        }
    }
}

template <class S>
__device__ __forceinline__ void stream_direct(const S &T, Walk &w, uint64_t pos, uint64_t end, uint64_t t0, uint64_t t1) {
    walk_ends(w, pos, end, t0, t1, true);
    uint32_t blocks = pos < end && !w.dead() ? static_cast<uint32_t>((end - pos) >> 5) : 0;
    if (blocks) {
        auto take_block = [&](const uint32_t (&x)[8]) {
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                const uint32_t v[4] = {x[h], x[h + 1], x[h + 2], x[h + 3]};
                w.id = T.template take<4>(w.id, v);
            }
        };
        // three blocks in flight or in hand, each loaded again as soon as it is done with
        uint32_t b[3][8];
        const uint8_t *t = reinterpret_cast<const uint8_t *>(pos);
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (blocks > static_cast<uint32_t>(i)) load32(t + 32 * i, b[i]);
        pos += static_cast<uint64_t>(blocks) * 32;
        for (;;) {
            take_block(b[0]);
            if (blocks > 3) load32(t + 96, b[0]);
            if (blocks == 1) break;
            take_block(b[1]);
            if (blocks > 4) load32(t + 128, b[1]);
            if (blocks == 2) break;
            take_block(b[2]);
            if (blocks > 5) load32(t + 160, b[2]);
            if (blocks == 3 || w.dead()) break;
            blocks -= 3;
            t += 96;
        }
        if (w.dead()) return;
    }
    walk_ends(w, pos, end, t0, t1, false);
}

// Text staged by the warp: rounds of one 64-byte window per lane, copied with cp.async (L2 to
// shared memory) so that four neighbouring lanes move one window; double-buffered, in the layout of
// coop_unit.  A lane's copies always serve the same four windows, whose places are worked out once
// (offsets from the warp's first window), not passed round by shuffles each time.
// `base` (16-byte aligned) lies at or below every lane's piece, within 2 GB; [t0, t1) is the lane's
// text.  Lanes without a piece pass pos = end.
template <class S>
__device__ __forceinline__ void stream_staged(const S &T, Walk &w, uint32_t stage, uint64_t base, uint64_t pos, uint64_t end, uint64_t t0, uint64_t t1) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t lo = (t0 + 15) & ~static_cast<uint64_t>(15), hi = t1 & ~static_cast<uint64_t>(15);
    while (pos < min(end, lo)) w.step_class(w.class_of(__ldg(reinterpret_cast<const uint8_t *>(pos++))));
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
        if (r < nwin && !w.dead()) {
            const uint32_t ws = wrel + kCoopWin * r;
            const uint32_t sb = stage + (r & 1) * kCoopBufBytes + 64 * lane;
            const uint32_t stop = min(srel, ws + kCoopWin);
            if (w.merged() && prel == ws && stop == ws + kCoopWin) {
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q) {
                    const uint4 x = lds_v4(sb + 16 * (q ^ sw));
                    const uint32_t v[4] = {x.x, x.y, x.z, x.w};
                    w.id = T.template take<4>(w.id, v);
                }
            } else {
#pragma unroll 1
                for (uint32_t q = 0; q < 4; ++q) {
                    const uint32_t g0 = ws + 16 * q, a = max(prel, g0), b = min(stop, g0 + 16);
                    if (a >= b) continue;
                    const uint4 x = lds_v4(sb + 16 * (q ^ sw));
                    const uint32_t v[4] = {x.x, x.y, x.z, x.w};
                    if (w.merged() && b - a == 16) w.id = T.template take<4>(w.id, v);
                    else w.take(v, static_cast<int>(a - g0), static_cast<int>(b - g0));
                }
            }
            prel = stop;
        }
        __syncwarp();
    }
    cp_async_wait0();
    __syncwarp();
    if (w.dead()) return;
    if (have) pos = base + prel;
    while (pos < end) w.step_class(w.class_of(__ldg(reinterpret_cast<const uint8_t *>(pos++))));
}

// Host: what a table says of itself, the field codes among it.
inline StreamTables stream_field_tables(const HostStream &T) {
    StreamTables a{};
    a.n_words = static_cast<uint32_t>(T.words.size());
    a.copies = T.copies;
    a.row = T.row_words * 4 * T.copies;
    if (T.kind == kStreamField) {
        const uint32_t w = T.width, bits = w * T.group, part = 4 / T.entry;
        auto byte = [&](uint32_t code) { return T.canon >> (8 * code) & 0xFF; };
        a.shift = T.shift;
        a.second = w == 2 ? 0x01010101u : 0u;
        a.canon0 = byte(0) * 0x01010101u;
        a.d1 = byte(1) - byte(0);
        a.d2 = byte(2) - byte(0);
        a.d12 = byte(3) - byte(2) - byte(1) + byte(0);
        // byte i's code to bit 32 - bits + w * i
        for (uint32_t i = 0; i < T.group; ++i) {
            a.mul |= 1u << (32 - bits + w * i - 8 * i);
            if (T.group == 2) a.mul_h |= 1u << (32 - bits + w * i - 8 * (i + 2));
        }
        a.take_bits = 1u << bits;
        // column c sits at word c / part, entry c % part
        a.part_mask = part - 1;
        a.col_mul = 4 * T.copies / part;
        a.part_mul = T.entry - a.col_mul;
    }
    return a;
}

// Host: the tables' part of a launch's arguments.  walk_only: no main table.
inline StreamTables stream_tables(const HostAutomaton &H, const DeviceAutomaton &D, bool walk_only, uint32_t warps) {
    const HostStream &T = H.stream;
    StreamTables a = stream_field_tables(T);
    a.warps = warps;
    a.walk = D.mg_walk;
    a.classmap = D.classmap;
    a.edge_pid = D.mg_edge_pid;
    a.code = D.st_code;
    a.words = D.st_words;
    a.n = H.n_states;
    a.C = H.n_classes;
    a.n_walk = static_cast<uint32_t>(H.merge.walk.size());
    uint32_t off = 0;
    if (!walk_only) {
        off = T.kind == kStreamField ? 0 : 256 * 128;
        a.off_table = off;
        off += a.n_words * 4 * T.copies;
        off = (off + 15) & ~15u;
    }
    const uint32_t wb = a.n_walk * 2;
    a.off_cls = off;
    off += 256;
    a.off_walk = wb <= kStreamWalkSmem ? off : kGlobal;
    off += wb <= kStreamWalkSmem ? (wb + 15) & ~15u : 0;
    a.off_stage = (off + 127) & ~127u;
    return a;
}

}  // namespace
}  // namespace ridfa

// The join's device building blocks (Sec. 3.2), shared by the join after the reach kernel
// (ridfa_device.cu) and the one after the stream kernels (ridfa_stream.cu): the distinct end states
// of a chunk, transfer matrices between chunks and their products, shard summaries.
#pragma once

#include "ridfa_kernels.cuh"

namespace ridfa {
namespace {

// ------------------------------------------------------------------------------- join
struct JoinArgs {
    Automaton A;
    uint32_t c;
    const uint16_t *maps;
    const uint32_t *dinfo;
    uint32_t *status;
    uint32_t *partials;       // [gridDim.x][2 + kMaxD]
    uint32_t *ticket;
    uint8_t *accept;
    uint32_t per_thread;      // boundaries per thread
    ridfa_shard_summary *summary;   // non-null: write the shard's relation instead of accept
};

// Distinct defined values of lambda_i, ascending (at most kMaxD; caller checked m <= kMaxD).
__device__ uint32_t distinct_of(const JoinArgs &p, uint32_t i, uint16_t *D) {
    const uint32_t info = p.dinfo[i];
    const uint32_t m = info >> 16;
    if (m <= 1) {
        D[0] = static_cast<uint16_t>(info & 0xFFFF);
        return m;
    }
    const uint16_t *row = p.maps + static_cast<uint64_t>(i) * p.A.k;
    uint32_t cnt = 0;
    for (uint32_t a = 0; a < p.A.k; ++a) {
        const uint16_t v = row[a];
        if (v == kUndef) continue;
        uint32_t j = 0;
        while (j < cnt && D[j] < v) ++j;
        if (j < cnt && D[j] == v) continue;
        if (cnt == kMaxD) return 0xFFFFFFFFu;
        for (uint32_t t = cnt; t > j; --t) D[t] = D[t - 1];
        D[j] = v;
        ++cnt;
    }
    return cnt;
}

__device__ __forceinline__ uint32_t index_of(const uint16_t *D, uint32_t m, uint16_t v) {
    for (uint32_t j = 0; j < m; ++j)
        if (D[j] == v) return j;
    return 0xFFFFFFFFu;
}

// Row x of M_i: bits y with lambda_i(a) = D_i[y] for some slot a in if_min({D_{i-1}[x]}).
__device__ uint32_t transfer_row(const JoinArgs &p, uint32_t i, uint16_t d_prev, const uint16_t *D,
                                 uint32_t m, bool *bad) {
    const uint32_t *mask = p.A.ifmask + static_cast<uint64_t>(d_prev) * p.A.kw;
    const uint16_t *row = p.maps + static_cast<uint64_t>(i) * p.A.k;
    uint32_t out = 0;
    for (uint32_t w = 0; w < p.A.kw; ++w) {
        uint32_t bits = mask[w];
        while (bits) {
            const uint32_t a = w * 32 + __ffs(bits) - 1;
            bits &= bits - 1;
            const uint16_t v = row[a];
            if (v == kUndef) continue;
            const uint32_t y = index_of(D, m, v);
            if (y == 0xFFFFFFFFu) *bad = true;
            else out |= 1u << y;
        }
    }
    return out;
}

// Product of a thread's run of boundaries: rows over D_{s-1}, columns over D_{e-1}.
struct Prod {
    uint32_t nrows;           // 0xFFFFFFFF = identity (no boundary)
    uint32_t rows[kMaxD];
};

__device__ void compose(Prod &a, const Prod &b) {   // a <- a x b
    if (b.nrows == 0xFFFFFFFFu) return;
    if (a.nrows == 0xFFFFFFFFu) {
        a = b;
        return;
    }
    for (uint32_t x = 0; x < a.nrows; ++x) {
        uint32_t bits = a.rows[x], out = 0;
        while (bits) {
            const uint32_t z = __ffs(bits) - 1;
            bits &= bits - 1;
            out |= b.rows[z];
        }
        a.rows[x] = out;
    }
}

__device__ bool is_final(const Automaton &A, uint32_t s) {
    return s < A.n && ((A.final_bits[s >> 5] >> (s & 31)) & 1);
}

// The accept bit when some chunk has more than kMaxD distinct end states (one block alone):
// if_min(PLAS_i) as a k-bit set, chunk by chunk.
__device__ void accept_wide(const JoinArgs &p, uint32_t *s_vec, uint32_t *s_nvec) {
    const Automaton &A = p.A;
    const uint32_t tid = threadIdx.x;
    const uint16_t *row0 = p.maps;
    const uint16_t v0 = row0[A.q0_slot];
    if (p.c == 1 || v0 == kUndef) {
        if (tid == 0) *p.accept = (v0 != kUndef && is_final(A, v0)) ? 1 : 0;
        return;
    }
    for (uint32_t w = tid; w < A.kw; w += blockDim.x)
        s_vec[w] = A.ifmask[static_cast<uint64_t>(v0) * A.kw + w];
    __syncthreads();
    for (uint32_t i = 1; i + 1 < p.c; ++i) {
        for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_nvec[w] = 0;
        __syncthreads();
        const uint16_t *row = p.maps + static_cast<uint64_t>(i) * A.k;
        for (uint32_t a = tid; a < A.k; a += blockDim.x) {
            if (!((s_vec[a >> 5] >> (a & 31)) & 1)) continue;
            const uint16_t v = row[a];
            if (v == kUndef) continue;
            for (uint32_t w = 0; w < A.kw; ++w) {
                const uint32_t m = A.ifmask[static_cast<uint64_t>(v) * A.kw + w];
                if (m) atomicOr(&s_nvec[w], m);
            }
        }
        __syncthreads();
        for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_vec[w] = s_nvec[w];
        __syncthreads();
    }
    __shared__ uint32_t s_acc;
    if (tid == 0) s_acc = 0;
    __syncthreads();
    const uint16_t *last = p.maps + static_cast<uint64_t>(p.c - 1) * A.k;
    for (uint32_t a = tid; a < A.k; a += blockDim.x)
        if (((s_vec[a >> 5] >> (a & 31)) & 1) && last[a] != kUndef && is_final(A, last[a]))
            s_acc = 1;
    __syncthreads();
    if (tid == 0) *p.accept = s_acc ? 1 : 0;
}

// Shard summary when some chunk has more than kMaxD distinct end states (block 0 alone):
// for every distinct state x the shard's first chunk ends in, propagate if_min({x}) chunk by
// chunk and record the end states reached, as bits over the last chunk's distinct end states.
__device__ void summary_wide(const JoinArgs &p, uint32_t *s_vec, uint32_t *s_nvec) {
    const Automaton &A = p.A;
    const uint32_t tid = threadIdx.x;
    ridfa_shard_summary *S = p.summary;
    __shared__ uint16_t s_out[RIDFA_MAX_SLOTS];
    __shared__ uint32_t s_nout, s_bits[RIDFA_MAX_SLOTS / 32];
    const uint16_t *row0 = p.maps;
    const uint16_t *last = p.maps + static_cast<uint64_t>(p.c - 1) * A.k;
    if (tid == 0) {
        // distinct defined end states of the last chunk, ascending
        uint32_t n = 0;
        for (uint32_t a = 0; a < A.k; ++a) {
            const uint16_t v = last[a];
            if (v == kUndef) continue;
            uint32_t j = 0;
            while (j < n && s_out[j] < v) ++j;
            if (j < n && s_out[j] == v) continue;
            for (uint32_t t = n; t > j; --t) s_out[t] = s_out[t - 1];
            s_out[j] = v;
            ++n;
        }
        s_nout = n;
        S->k = A.k;
        S->n_out = n;
    }
    __syncthreads();
    for (uint32_t a = tid; a < RIDFA_MAX_SLOTS; a += blockDim.x) {
        S->out_state[a] = a < s_nout ? s_out[a] : kUndef;
        S->entry[a] = a < A.k ? row0[a] : kUndef;
        for (uint32_t w = 0; w < RIDFA_MAX_SLOTS / 32; ++w) S->reach[a][w] = 0;
    }
    __syncthreads();
    for (uint32_t a0 = 0; a0 < A.k; ++a0) {
        const uint16_t x = row0[a0];
        if (x == kUndef) continue;
        bool seen = false;                    // handled with an earlier slot of the same state
        for (uint32_t b = 0; b < a0 && !seen; ++b) seen = row0[b] == x;
        if (seen) continue;
        if (tid < RIDFA_MAX_SLOTS / 32) s_bits[tid] = 0;
        __syncthreads();
        if (p.c == 1) {
            if (tid == 0)
                for (uint32_t y = 0; y < s_nout; ++y)
                    if (s_out[y] == x) s_bits[y >> 5] |= 1u << (y & 31);
        } else {
            for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_vec[w] = A.ifmask[static_cast<uint64_t>(x) * A.kw + w];
            __syncthreads();
            for (uint32_t i = 1; i + 1 < p.c; ++i) {
                for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_nvec[w] = 0;
                __syncthreads();
                const uint16_t *row = p.maps + static_cast<uint64_t>(i) * A.k;
                for (uint32_t a = tid; a < A.k; a += blockDim.x) {
                    if (!((s_vec[a >> 5] >> (a & 31)) & 1)) continue;
                    const uint16_t v = row[a];
                    if (v == kUndef) continue;
                    for (uint32_t w = 0; w < A.kw; ++w) {
                        const uint32_t m = A.ifmask[static_cast<uint64_t>(v) * A.kw + w];
                        if (m) atomicOr(&s_nvec[w], m);
                    }
                }
                __syncthreads();
                for (uint32_t w = tid; w < A.kw; w += blockDim.x) s_vec[w] = s_nvec[w];
                __syncthreads();
            }
            for (uint32_t a = tid; a < A.k; a += blockDim.x) {
                if (!((s_vec[a >> 5] >> (a & 31)) & 1) || last[a] == kUndef) continue;
                for (uint32_t y = 0; y < s_nout; ++y)
                    if (s_out[y] == last[a]) atomicOr(&s_bits[y >> 5], 1u << (y & 31));
            }
        }
        __syncthreads();
        for (uint32_t a = tid; a < A.k; a += blockDim.x)
            if (row0[a] == x)
                for (uint32_t w = 0; w < RIDFA_MAX_SLOTS / 32; ++w) S->reach[a][w] = s_bits[w];
        __syncthreads();
    }
}

// Shard summary from the chain product (thread 0 of the last block): tot maps the first chunk's
// distinct end states D_1 to the last chunk's D_c.
__device__ void summary_matrix(const JoinArgs &p, const Prod &tot) {
    const Automaton &A = p.A;
    ridfa_shard_summary *S = p.summary;
    uint16_t D0[kMaxD], Dl[kMaxD];
    const uint32_t m0 = distinct_of(p, 0, D0);
    const uint32_t ml = distinct_of(p, p.c - 1, Dl);
    if (m0 == 0xFFFFFFFFu || ml == 0xFFFFFFFFu || (p.c > 1 && tot.nrows == 0xFFFFFFFFu)) {
        atomicOr(p.status, kStatusBad);
        return;
    }
    S->k = A.k;
    S->n_out = ml;
    for (uint32_t y = 0; y < RIDFA_MAX_SLOTS; ++y) S->out_state[y] = y < ml ? Dl[y] : kUndef;
    for (uint32_t a = 0; a < RIDFA_MAX_SLOTS; ++a) {
        const uint16_t x = a < A.k ? p.maps[a] : kUndef;
        S->entry[a] = x;
        uint32_t bits = 0;
        if (x != kUndef) {
            const uint32_t xi = index_of(D0, m0, x);
            if (xi == 0xFFFFFFFFu) atomicOr(p.status, kStatusBad);
            else bits = p.c == 1 ? (1u << xi) : tot.rows[xi];
        }
        S->reach[a][0] = bits;
        for (uint32_t w = 1; w < RIDFA_MAX_SLOTS / 32; ++w) S->reach[a][w] = 0;
    }
}

}  // namespace
}  // namespace ridfa

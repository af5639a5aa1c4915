// Host construction of the merge graph and of the stream kernels' main-loop table
// (HostMerge, HostStream in ridfa_internal.h), from a compiled automaton.
//
// The graph holds the functions that byte-class sequences perform on the set of all states
// (Sec. 5's state convergence, precomputed: runs that meet in one state go on as one).  It is the
// part of the simultaneous automaton over the runs up to the point where one run is left, which
// stays small where the whole would not.
#include <algorithm>
#include <cstring>
#include <map>
#include <string>
#include <unordered_map>

#include "ridfa_internal.h"

namespace ridfa {
namespace {

// Limits of the graph: inner nodes (codon-like automata, whose runs stay apart, run into it),
// entries of the partition table, and the images stepped while building (compile time: 500,000 steps with
// their partitions take up to some 20 ms on one core, which a graph over the limits costs for nothing).
constexpr uint32_t kMaxInner = 6144;
constexpr uint32_t kMaxInnerApart = 1536;      // without the merge hint
constexpr uint64_t kMaxPartEntries = 1u << 20;
constexpr uint64_t kMaxSteps = 500000;

std::string key_of(uint32_t pid, const uint16_t *v, size_t n) {
    std::string k(4 + n * 2, '\0');
    std::memcpy(&k[0], &pid, 4);
    std::memcpy(&k[4], v, n * 2);
    return k;
}

bool build_graph(const HostAutomaton &H, HostMerge &G) {
    const uint32_t n = H.n_states, C = H.n_classes;
    if (n == 0 || n > 8192) return false;
    const uint32_t max_inner = H.merges ? kMaxInner : kMaxInnerApart;
    std::unordered_map<std::string, uint32_t> node_id, part_id, step_id;
    // partition 0: every run dead; partition 1: the identity
    G.part.assign(n, kNoBlock);
    for (uint32_t x = 0; x < n; ++x) G.part.push_back(static_cast<uint16_t>(x));
    part_id[key_of(0, &G.part[0], n)] = 0;
    part_id[key_of(0, &G.part[n], n)] = 1;
    uint32_t parts = 2;
    G.leaf.push_back(n);                                   // leaf 0: partition 0, the dead state
    std::unordered_map<uint32_t, uint32_t> leaf_id;
    std::vector<uint32_t> node_d;                          // blocks of each inner node
    auto add_node = [&](uint32_t pid, const std::vector<uint16_t> &img) -> uint32_t {
        const auto r = node_id.emplace(key_of(pid, img.data(), img.size()), static_cast<uint32_t>(node_d.size()));
        if (r.second) {
            G.node_part.push_back(static_cast<uint16_t>(pid));
            G.node_img.push_back(static_cast<uint32_t>(G.images.size()));
            G.images.insert(G.images.end(), img.begin(), img.end());
            node_d.push_back(static_cast<uint32_t>(img.size()));
        }
        return r.first->second;
    };
    auto add_leaf = [&](uint32_t pid, uint32_t state) -> uint32_t {
        const auto r = leaf_id.emplace(pid << 16 | state, static_cast<uint32_t>(G.leaf.size()));
        if (r.second) G.leaf.push_back(pid << 16 | state);
        return r.first->second;
    };
    std::vector<uint16_t> img(n), next_img, block(n), pv(n);
    for (uint32_t x = 0; x < n; ++x) img[x] = static_cast<uint16_t>(x);
    add_node(1, img);
    std::vector<uint32_t> where(n + 1, 0), stamp(n + 1, 0);
    uint32_t gen = 0;
    uint64_t steps = 0;
    for (uint32_t u = 0; u < node_d.size(); ++u) {
        const uint32_t d = node_d[u], pid = G.node_part[u], off = G.node_img[u];
        for (uint32_t c = 0; c < C; ++c) {
            // step the distinct images; block[b]: the new block of old block b.  Blocks are numbered
            // by their smallest state, an order that first appearance keeps.
            steps += d;
            ++gen;
            next_img.clear();
            for (uint32_t b = 0; b < d; ++b) {
                const uint32_t t = H.trans[static_cast<size_t>(G.images[off + b]) * C + c];
                if (t == n) {
                    block[b] = kNoBlock;
                } else {
                    if (stamp[t] != gen) {
                        stamp[t] = gen;
                        where[t] = static_cast<uint32_t>(next_img.size());
                        next_img.push_back(static_cast<uint16_t>(t));
                    }
                    block[b] = static_cast<uint16_t>(where[t]);
                }
            }
            uint32_t code;
            if (next_img.empty()) {
                code = kLeafBit;                           // leaf 0
            } else {
                uint32_t npid = pid;
                bool same = next_img.size() == d;
                for (uint32_t b = 0; b < d && same; ++b) same = block[b] == b;
                if (!same) {
                    const auto r = step_id.emplace(key_of(pid, block.data(), d), 0u);
                    if (r.second) {
                        for (uint32_t x = 0; x < n; ++x) {
                            const uint16_t o = G.part[static_cast<size_t>(pid) * n + x];
                            pv[x] = o == kNoBlock ? kNoBlock : block[o];
                        }
                        steps += n / 4;
                        const auto q = part_id.emplace(key_of(0, pv.data(), n), parts);
                        if (q.second) {
                            if (static_cast<uint64_t>(parts + 1) * n > kMaxPartEntries || parts >= 0x7FFF) return false;
                            G.part.insert(G.part.end(), pv.begin(), pv.end());
                            ++parts;
                        }
                        r.first->second = q.first->second;
                    }
                    npid = r.first->second;
                }
                code = next_img.size() == 1 ? kLeafBit | add_leaf(npid, next_img[0]) : add_node(npid, next_img);
            }
            if (!H.merges && node_d.size() > 256 && G.leaf.size() == 1) return false;    // nothing merges
            if (node_d.size() > max_inner || G.leaf.size() >= 0x8000 || steps > kMaxSteps) return false;
            G.next.push_back(static_cast<uint16_t>(code));
        }
    }
    G.inner = static_cast<uint32_t>(node_d.size());
    G.parts = parts;
    if (n + 1 + G.inner > 0xFFFF) return false;
    // one-byte steps of states and nodes in one table: states first, then the nodes
    G.walk = H.trans;
    for (uint16_t e : G.next) {
        const uint32_t l = e & kLeafBit ? G.leaf[e & 0x7FFF] : 0;
        G.walk.push_back(static_cast<uint16_t>(e & kLeafBit ? l & 0xFFFF : e + n + 1));
        G.edge_pid.push_back(static_cast<uint16_t>(l >> 16));
    }
    G.walk.resize(G.walk.size() + (G.walk.size() & 1), static_cast<uint16_t>(n));    // whole words
    G.slot_alive.assign(static_cast<size_t>(parts) * H.kw, 0);
    for (uint32_t p = 0; p < parts; ++p)
        for (uint32_t a = 0; a < H.k; ++a)
            if (G.part[static_cast<size_t>(p) * n + H.slot_state[a]] != kNoBlock)
                G.slot_alive[static_cast<size_t>(p) * H.kw + (a >> 5)] |= 1u << (a & 31);
    return true;
}

// Every index the kernels take from the graph unchecked.
bool graph_in_bounds(const HostAutomaton &H, const HostMerge &G) {
    const uint32_t n = H.n_states;
    if (G.next.size() != static_cast<size_t>(G.inner) * H.n_classes || G.part.size() != static_cast<size_t>(G.parts) * n ||
        G.node_part.size() != G.inner || G.node_img.size() != G.inner || G.leaf.empty())
        return false;
    if (G.walk.size() < static_cast<size_t>(n + 1 + G.inner) * H.n_classes || G.edge_pid.size() != G.next.size()) return false;
    for (uint16_t c : G.walk)
        if (c >= n + 1 + G.inner) return false;
    for (uint16_t q : G.edge_pid)
        if (q >= G.parts) return false;
    for (uint32_t l : G.leaf)
        if ((l >> 16) >= G.parts || (l & 0xFFFF) > n) return false;
    for (uint16_t s : G.images)
        if (s >= n) return false;
    for (uint32_t u = 0; u < G.inner; ++u) {
        if (G.node_part[u] >= G.parts) return false;
        for (uint32_t x = 0; x < n; ++x) {
            const uint16_t b = G.part[static_cast<size_t>(G.node_part[u]) * n + x];
            if (b != kNoBlock && static_cast<size_t>(G.node_img[u]) + b >= G.images.size()) return false;
        }
    }
    return true;
}

// Shared-memory wavefronts of one 32-lane gather into `copies` lane copies (rows at random): by
// counting for 32, at most 2 for 16, by simulation below that.
double wavefronts(uint32_t copies) {
    switch (copies) {
        case 32: return 1.0;
        case 16: return 1.9;
        case 8: return 2.7;
        case 4: return 3.2;
        default: return 3.4;
    }
}

size_t rest_bytes(const HostAutomaton &H, uint32_t kind) {
    // class codes; byte classes and the one-byte table of the ragged ends
    const size_t walk = H.merge.walk.size() * 2;
    return (kind == kStreamField ? 0 : 256 * 128) + 256 + (walk <= kStreamWalkSmem ? (walk + 15) / 16 * 16 : 0) + 256;
}

// Column offsets of a pair table: offset(c1, c2) = first[c1] + second[c2], where equal sums mean
// equal columns.  Every first class takes a place (word, part) so that its whole row of columns,
// the undefined ones included, meets only equal columns; second classes shift by whole words.
// Tries a few layouts of the second classes and returns the words of a row (0: none found).
uint32_t place_pairs(const std::vector<uint32_t> &col, uint32_t C, uint32_t per_word, uint32_t limit,
                     std::vector<uint32_t> &first, std::vector<uint32_t> &second, std::vector<int64_t> &slots) {
    uint32_t best = 0;
    std::vector<uint32_t> rows_live(C, 0), cols_live(C, 0), ord(C), rord(C);
    for (uint32_t a = 0; a < C; ++a)
        for (uint32_t b = 0; b < C; ++b)
            if (col[a * C + b]) {
                ++rows_live[a];
                ++cols_live[b];
            }
    for (uint32_t i = 0; i < C; ++i) ord[i] = rord[i] = i;
    std::stable_sort(rord.begin(), rord.end(), [&](uint32_t x, uint32_t y) { return rows_live[x] > rows_live[y]; });
    for (uint32_t gap = 1; gap <= 6; ++gap)
        for (uint32_t asc = 0; asc < 2; ++asc) {
            // the class most rows have a move on comes first, `gap` words before the others
            std::stable_sort(ord.begin(), ord.end(), [&](uint32_t x, uint32_t y) { return cols_live[x] > cols_live[y]; });
            if (asc) std::reverse(ord.begin() + 1, ord.end());
            std::vector<uint32_t> sec(C), fst(C);
            for (uint32_t i = 0; i < C; ++i) sec[ord[i]] = i == 0 ? 0 : gap + i - 1;
            std::vector<int64_t> occ(static_cast<size_t>(limit + 2 * C + 16) * per_word, -1);
            uint32_t words = 0;
            bool ok = true;
            for (uint32_t ri = 0; ri < C && ok; ++ri) {
                const uint32_t a = rord[ri];
                bool placed = false;
                for (uint32_t w = 0; w < limit && !placed; ++w)
                    for (uint32_t q = 0; q < per_word && !placed; ++q) {
                        bool fit = true;
                        for (uint32_t b = 0; b < C && fit; ++b) {
                            const int64_t o = occ[static_cast<size_t>(w + sec[b]) * per_word + q];
                            fit = o < 0 || o == static_cast<int64_t>(col[a * C + b]);
                        }
                        if (!fit) continue;
                        for (uint32_t b = 0; b < C; ++b) {
                            occ[static_cast<size_t>(w + sec[b]) * per_word + q] = col[a * C + b];
                            words = std::max(words, w + sec[b] + 1);
                        }
                        fst[a] = w * per_word + q;
                        placed = true;
                    }
                ok = placed && words <= limit;
            }
            if (ok && (best == 0 || words < best)) {
                best = words;
                first = fst;
                second.assign(C, 0);
                for (uint32_t b = 0; b < C; ++b) second[b] = sec[b] * per_word;
                occ.resize(static_cast<size_t>(words) * per_word);
                slots = occ;
            }
        }
    return best;
}

// Codes by a bit field of the byte: the field's place and the byte of each code, when the live bytes
// differ in at most two adjacent bits.
bool find_field(const HostAutomaton &H, HostStream &t) {
    const uint32_t n = H.n_states, C = H.n_classes;
    std::vector<uint8_t> class_live(C, 0);
    for (uint32_t c = 0; c < C; ++c)
        for (uint32_t s = 0; s < n && !class_live[c]; ++s) class_live[c] = H.trans[static_cast<size_t>(s) * C + c] != n;
    std::vector<uint32_t> live;
    for (uint32_t b = 0; b < 256; ++b)
        if (class_live[H.classmap[b]]) live.push_back(b);
    bool field = false;
    for (uint32_t w = 1; w <= 2 && !field && live.size() <= 4; ++w)
        for (uint32_t sh = 0; sh + w <= 8 && !field; ++sh) {
            uint32_t seen = 0, canon = 0, m = (1u << w) - 1;
            bool inj = live.size() <= m + 1;
            for (uint32_t b : live) {
                const uint32_t code = (b >> sh) & m;
                if (seen >> code & 1) inj = false;
                seen |= 1u << code;
                canon |= b << (8 * code);
            }
            // a code no live byte has: its canonical byte has another code, so no byte passes
            for (uint32_t code = 0; code <= 3; ++code)
                if (!(seen >> code & 1)) canon |= ((code ^ 1) & m) << sh << (8 * code);
            if (inj) {
                field = true;
                t.shift = sh;
                t.width = w;
                t.canon = canon;
            }
        }
    return field;
}

// Entries of a field table: column = the codes of `group` bytes, the first one lowest.
void fill_field(const HostAutomaton &H, HostStream &t) {
    const uint32_t n = H.n_states, per_word = 4 / t.entry, W = t.row_words, m = (1u << t.width) - 1;
    t.words.assign(static_cast<size_t>(n + 1) * W, 0);
    // columns of half a group, then of two halves
    const uint32_t half = t.width * t.group / 2, cols = 1u << half;
    std::vector<uint16_t> mid(static_cast<size_t>(n + 1) * cols);
    std::vector<uint32_t> cls(m + 1);
    for (uint32_t v = 0; v <= m; ++v) cls[v] = H.classmap[(t.canon >> (8 * v)) & 0xFF];
    for (uint32_t s = 0; s <= n; ++s)
        for (uint32_t c = 0; c < cols; ++c) {
            uint32_t x = s;
            for (uint32_t i = 0; i < t.group / 2; ++i) x = H.trans[static_cast<size_t>(x) * H.n_classes + cls[(c >> (t.width * i)) & m]];
            mid[static_cast<size_t>(s) * cols + c] = static_cast<uint16_t>(x);
        }
    for (uint32_t s = 0; s <= n; ++s)
        for (uint32_t c = 0; c < W * per_word; ++c) {
            const uint32_t y = mid[static_cast<size_t>(s) * cols + (c & (cols - 1))];
            const uint32_t x = c >> (2 * half) ? n : mid[static_cast<size_t>(y) * cols + (c >> half)];
            t.words[static_cast<size_t>(s) * W + c / per_word] |= x << (8 * t.entry * (c % per_word));
        }
}

void build_table(HostAutomaton &H) {
    const uint32_t n = H.n_states, C = H.n_classes;
    HostStream best;
    double best_cost = 1e9;
    const uint32_t entry = n + 1 <= 256 ? 1 : 2, per_word = 4 / entry;
    // the most copies that fit, with their cost in shared-memory cycles per 32 text bytes
    auto consider = [&](HostStream t, double fixed, double per_lookup) {
        const size_t rest = rest_bytes(H, t.kind);
        for (uint32_t f = 32; f >= 1; f /= 2) {
            const size_t table = static_cast<size_t>(n + 1) * t.row_words * 4 * f;
            uint32_t warps = 32;
            if (t.kind != kStreamField) {
                if (rest + table + 8 * kStreamStaging > kStreamSmem) continue;
                warps = static_cast<uint32_t>(std::min<size_t>(32, (kStreamSmem - rest - table) / kStreamStaging));
            } else if (rest + table > kStreamSmem) {
                continue;
            }
            // fewer warps hide less of the lookups' latency
            const double thin = warps >= 24 ? 1.0 : warps >= 16 ? 1.08 : warps >= 12 ? 1.2 : 1.45;
            const double cost = std::max(1.75, fixed + wavefronts(f) * per_lookup) * thin;
            if (cost < best_cost) {
                best_cost = cost;
                t.cost = static_cast<float>(cost);
                t.copies = f;
                t.warps = warps;
                best = t;
            }
        }
    };
    HostStream t;
    t.entry = entry;
    const bool field = find_field(H, t);
    if (field) {
        t.kind = kStreamField;
        for (uint32_t g : {4u, 2u}) {
            t.group = g;
            const uint32_t cols = 1u << (t.width * g);
            t.row_words = (cols + per_word - 1) / per_word;
            consider(t, 1.2, 1.0 / g);
        }
    }
    // two bytes a lookup through class codes
    std::vector<uint32_t> col(static_cast<size_t>(C) * C, 0), first, second, firsts, seconds;
    std::vector<uint32_t> reps(1, 0);                   // a class pair of each distinct column
    std::vector<int64_t> slots, best_slots;
    if (!field && C <= 24) {
        std::map<std::vector<uint16_t>, uint32_t> ids;
        std::vector<uint16_t> v(n);
        for (uint32_t a = 0; a < C; ++a)
            for (uint32_t b = 0; b < C; ++b) {
                bool any = false;
                for (uint32_t s = 0; s < n; ++s) {
                    v[s] = H.trans[static_cast<size_t>(H.trans[static_cast<size_t>(s) * C + a]) * C + b];
                    any |= v[s] != n;
                }
                if (!any) continue;
                const auto r = ids.emplace(v, static_cast<uint32_t>(ids.size() + 1));
                if (r.second) reps.push_back(a * C + b);
                col[a * C + b] = r.first->second;
            }
        const uint32_t limit = static_cast<uint32_t>(std::min<size_t>(256, kStreamSmem / 4 / (n + 1)));
        const uint32_t words = place_pairs(col, C, per_word, limit, first, second, slots);
        if (words) {
            t.kind = kStreamPair;
            t.group = 2;
            t.row_words = words;
            consider(t, 1.64, 0.5);
        }
    }
    if (!field) {
        t.kind = kStreamSingle;
        t.group = 1;
        t.row_words = (C + per_word - 1) / per_word;
        consider(t, 1.64, 1.0);
    }
    if (best_cost >= 1e9) return;
    // entries, then the codes in byte offsets of the chosen number of copies
    const uint32_t W = best.row_words;
    best.words.assign(static_cast<size_t>(n + 1) * W, 0);
    auto put = [&](uint32_t s, uint32_t c, uint32_t v) {
        const uint32_t bits = 8 * entry;
        best.words[static_cast<size_t>(s) * W + c / per_word] |= v << (bits * (c % per_word));
    };
    auto step = [&](uint32_t s, uint32_t c) -> uint32_t { return H.trans[static_cast<size_t>(s) * C + c]; };
    auto offset = [&](uint32_t c) { return c / per_word * 4 * best.copies + c % per_word * entry; };
    if (best.kind == kStreamField) {
        fill_field(H, best);
    } else {
        best.byte_code.assign(256, 0);
        if (best.kind == kStreamPair) {
            for (uint32_t s = 0; s <= n; ++s)
                for (uint32_t c = 0; c < W * per_word; ++c) {
                    const int64_t id = c < slots.size() ? slots[c] : -1;
                    put(s, c, id > 0 ? step(step(s, reps[id] / C), reps[id] % C) : n);
                }
            for (uint32_t b = 0; b < 256; ++b)
                best.byte_code[b] = offset(first[H.classmap[b]]) | offset(second[H.classmap[b]]) << 16;
        } else {
            for (uint32_t s = 0; s <= n; ++s)
                for (uint32_t c = 0; c < W * per_word; ++c) put(s, c, c < C ? step(s, c) : n);
            for (uint32_t b = 0; b < 256; ++b) best.byte_code[b] = offset(H.classmap[b]);
        }
        for (uint32_t v : best.byte_code)
            if ((v & 0xFFFF) + (v >> 16) > 0xFFFF) return;
    }
    H.stream = best;
}

// The sets that strings of up to `back_depth` bytes lead the set of all states to, each followed until
// fewer than kSetRuns states are left: what a piece in the middle of a chunk can be entered with.  Sets
// are bit rows; left out when they are too many, or when some string of kMaxDepth bytes leaves more states.
void build_back(const HostAutomaton &H, HostSet &Z) {
    constexpr uint32_t kMaxNodes = 4096, kMaxDepth = 24, kHash = 4 * kMaxNodes;
    const uint32_t n = H.n_states, C = H.n_classes, words = (n + 63) / 64;
    if (n < kSetRuns) return;
    std::vector<uint64_t> sets(words, 0), row(words);     // bit row of every set met; 0: all states
    std::vector<uint32_t> depth{0}, code{0}, hash(kHash, UINT32_MAX), order{0};
    for (uint32_t x = 0; x < n; ++x) sets[x >> 6] |= 1ull << (x & 63);
    std::vector<uint16_t> images(kSetRuns, static_cast<uint16_t>(n)), next;   // leaf 0: all dead
    uint64_t steps = 0;
    std::vector<bool> dead_class(C, true);
    for (uint32_t x = 0; x < n; ++x)
        for (uint32_t c = 0; c < C; ++c)
            if (H.trans[static_cast<size_t>(x) * C + c] < n) dead_class[c] = false;
    uint32_t inner = 1, leaves = 1;                       // code: the inner node's index, or kLeafBit | leaf
    for (uint32_t u = 0; u < order.size(); ++u) {
        const uint32_t from = order[u];
        if (depth[from] >= kMaxDepth) return;
        for (uint32_t c = 0; c < C; ++c) {
            if (dead_class[c]) {
                next.push_back(kLeafBit);
                continue;
            }
            std::fill(row.begin(), row.end(), 0);
            for (uint32_t w = 0; w < words; ++w)
                for (uint64_t b = sets[static_cast<size_t>(from) * words + w]; b; b &= b - 1) {
                    const uint32_t t = H.trans[static_cast<size_t>(w * 64 + __builtin_ctzll(b)) * C + c];
                    if (t < n) row[t >> 6] |= 1ull << (t & 63);
                }
            uint32_t count = 0;
            uint64_t h = 0;
            for (uint64_t v : row) {
                count += static_cast<uint32_t>(__builtin_popcountll(v));
                h = (h ^ v) * 0x9E3779B97F4A7C15ull;
                h ^= h >> 29;
            }
            if ((steps += count) > kMaxSteps) return;
            if (!count) {
                next.push_back(kLeafBit);
                continue;
            }
            uint32_t at = static_cast<uint32_t>(h >> 32) % kHash;
            while (hash[at] != UINT32_MAX && !std::equal(row.begin(), row.end(), sets.begin() + static_cast<size_t>(hash[at]) * words))
                at = (at + 1) % kHash;
            if (hash[at] == UINT32_MAX) {
                const uint32_t id = static_cast<uint32_t>(depth.size());
                if (id >= 2 * kMaxNodes) return;
                hash[at] = id;
                sets.insert(sets.end(), row.begin(), row.end());
                depth.push_back(depth[from] + 1);
                if (count < kSetRuns) {
                    code.push_back(kLeafBit | leaves++);
                    for (uint32_t w = 0; w < words; ++w)
                        for (uint64_t b = row[w]; b; b &= b - 1) images.push_back(static_cast<uint16_t>(w * 64 + __builtin_ctzll(b)));
                    images.resize(static_cast<size_t>(leaves) * kSetRuns, static_cast<uint16_t>(n));
                } else {
                    if (inner >= kMaxNodes) return;
                    code.push_back(inner++);
                    order.push_back(id);
                }
            }
            next.push_back(static_cast<uint16_t>(code[hash[at]]));
        }
    }
    // every index the kernels take unchecked
    if (next.size() != static_cast<size_t>(inner) * C || images.size() != static_cast<size_t>(leaves) * kSetRuns) return;
    for (uint16_t e : next)
        if ((e & kLeafBit) ? (e & 0x7FFFu) >= leaves : e >= inner) return;
    // A string's way to a leaf may be longer than the shortest one to it, and a set that leads back to itself
    // has ways without end: the kernels walk as many bytes as the longest way has, if there is one.
    std::vector<uint32_t> ways(inner, 0), longest(inner, 0), ready{0};
    for (uint16_t e : next)
        if (!(e & kLeafBit)) ++ways[e];
    uint32_t done = 0, deepest = 0;
    if (ways[0]) return;
    while (!ready.empty()) {
        const uint32_t u = ready.back();
        ready.pop_back();
        ++done;
        deepest = std::max(deepest, longest[u] + 1);
        for (uint32_t c = 0; c < C; ++c) {
            const uint16_t e = next[static_cast<size_t>(u) * C + c];
            if (e & kLeafBit) continue;
            longest[e] = std::max(longest[e], longest[u] + 1);
            if (--ways[e] == 0) ready.push_back(e);
        }
    }
    if (done != inner || deepest > kMaxDepth) return;
    Z.back_next = std::move(next);
    Z.back_images = std::move(images);
    Z.back_depth = deepest;
}

// The functions of the first bytes on the slots, level by level, down to the first level on which all
// have fewer than kSetRuns distinct values.
bool build_set(const HostAutomaton &H, HostSet &Z) {
    constexpr uint32_t kMaxNodes = 4096;
    const uint32_t n = H.n_states, C = H.n_classes, k = H.k;
    if (n == 0 || n > 8192 || k > RIDFA_MAX_SLOTS) return false;
    HostStream t;
    t.entry = 2;
    if (!find_field(H, t)) return false;
    t.kind = kStreamField;
    // four bytes a lookup in one copy, else two bytes in the most copies that fit
    const size_t rest = set_rest_bytes(H);
    for (uint32_t g : {4u, 2u}) {
        t.group = g;
        t.row_words = ((1u << (t.width * g)) + 1) / 2;
        t.copies = 0;
        for (uint32_t f = 32; f >= 1 && !t.copies; f /= 2)
            if (rest + static_cast<size_t>(n + 1) * t.row_words * 4 * f <= kStreamSmem) t.copies = f;
        if (t.copies) break;
    }
    if (!t.copies) return false;
    fill_field(H, t);
    Z.table = t;
    using Fn = std::vector<uint16_t>;                     // state of each slot, n: dead
    std::map<Fn, uint32_t> ids, part_ids;
    std::vector<Fn> level, next_level;
    Z.leaf = {0, 0};
    Z.images.assign(kSetRuns, static_cast<uint16_t>(n));
    auto add_leaf = [&](const Fn &f) -> uint32_t {
        Fn img;
        Fn block(k, 0xFF);
        for (uint32_t a = 0; a < k; ++a) {
            if (f[a] == n) continue;
            const uint32_t b = static_cast<uint32_t>(std::find(img.begin(), img.end(), f[a]) - img.begin());
            if (b == img.size()) img.push_back(f[a]);
            block[a] = static_cast<uint16_t>(b);
        }
        img.resize(kSetRuns, static_cast<uint16_t>(n));
        const auto r = part_ids.emplace(block, Z.parts);
        if (r.second) {
            ++Z.parts;
            for (uint16_t b : block) Z.part.push_back(static_cast<uint8_t>(b));
        }
        Z.leaf.push_back(r.first->second);
        Z.leaf.push_back(static_cast<uint32_t>(Z.images.size()));
        Z.images.insert(Z.images.end(), img.begin(), img.end());
        return static_cast<uint32_t>(Z.leaf.size() / 2 - 1);
    };
    part_ids.emplace(Fn(k, 0xFF), 0u);                     // partition 0: all dead
    Z.parts = 1;
    Z.part.assign(k, 0xFF);
    level.push_back(Fn(H.slot_state.begin(), H.slot_state.end()));
    for (uint32_t d = 1; d <= 32; ++d) {
        ids.clear();
        next_level.clear();
        std::vector<uint16_t> edges;
        size_t most = 0;
        for (const Fn &f : level)
            for (uint32_t c = 0; c < C; ++c) {
                Fn g(k);
                bool any = false;
                for (uint32_t a = 0; a < k; ++a) {
                    g[a] = f[a] == n ? static_cast<uint16_t>(n) : H.trans[static_cast<size_t>(f[a]) * C + c];
                    any |= g[a] != n;
                }
                if (!any) {
                    edges.push_back(kLeafBit);
                    continue;
                }
                const auto r = ids.emplace(g, static_cast<uint32_t>(next_level.size()));
                if (r.second) {
                    next_level.push_back(g);
                    std::sort(g.begin(), g.end());
                    size_t v = std::unique(g.begin(), g.end()) - g.begin();
                    if (std::binary_search(g.begin(), g.begin() + v, static_cast<uint16_t>(n))) --v;
                    most = std::max(most, v);
                }
                edges.push_back(static_cast<uint16_t>(r.first->second));
            }
        if (Z.inner + level.size() + next_level.size() > kMaxNodes) return false;
        const bool last = most < kSetRuns;
        std::vector<uint32_t> leaf_of;
        if (last)
            for (const Fn &f : next_level) leaf_of.push_back(add_leaf(f));
        const uint32_t base = Z.inner + static_cast<uint32_t>(level.size());       // first node of the next level
        for (uint16_t e : edges)
            Z.next.push_back(e & kLeafBit ? kLeafBit : static_cast<uint16_t>(last ? kLeafBit | leaf_of[e] : base + e));
        Z.inner = base;
        if (last) {
            Z.depth = d;
            break;
        }
        level.swap(next_level);
        if (level.empty()) return false;
    }
    if (!Z.depth) return false;
    Z.block_mask.assign(static_cast<size_t>(Z.parts) * kSetRuns * H.kw, 0);
    for (uint32_t p = 0; p < Z.parts; ++p)
        for (uint32_t a = 0; a < k; ++a) {
            const uint8_t b = Z.part[static_cast<size_t>(p) * k + a];
            if (b != 0xFF) Z.block_mask[(static_cast<size_t>(p) * H.kw + (a >> 5)) * kSetRuns + b] |= 1u << (a & 31);
        }
    build_back(H, Z);
    // every index the kernels take unchecked
    if (Z.next.size() != static_cast<size_t>(Z.inner) * C || Z.parts > 0xFFFF) return false;
    for (uint16_t e : Z.next)
        if ((e & kLeafBit) ? 2u * (e & 0x7FFFu) + 1 >= Z.leaf.size() : e >= Z.inner) return false;
    for (size_t l = 0; l < Z.leaf.size(); l += 2)
        if (Z.leaf[l] >= Z.parts || Z.leaf[l + 1] + kSetRuns > Z.images.size()) return false;
    for (uint16_t s : Z.images)
        if (s > n) return false;
    return true;
}

}  // namespace

size_t set_rest_bytes(const HostAutomaton &H) { return 256 + (H.trans.size() * 2 + 15) / 16 * 16 + 256; }

size_t stream_table_bytes(const HostAutomaton &H) {
    return rest_bytes(H, H.stream.kind) + static_cast<size_t>(H.n_states + 1) * H.stream.row_words * 4 * H.stream.copies;
}

size_t stream_walk_bytes(const HostAutomaton &H) { return rest_bytes(H, kStreamField); }

void build_stream(HostAutomaton &H) {
    HostMerge G;
    if (H.k > RIDFA_MAX_SLOTS) return;
    if (!build_graph(H, G) || !graph_in_bounds(H, G)) {
        HostSet Z;
        if (build_set(H, Z)) {
            Z.ok = true;
            H.set = std::move(Z);
        }
        return;
    }
    G.ok = true;
    H.merge = std::move(G);
    build_table(H);
}

}  // namespace ridfa

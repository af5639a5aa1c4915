// The tables that ridfa_compile builds for the stream and set kernels, by name, for the host tests.
#include <cstring>

#include "ridfa_internal.h"

namespace {
const ridfa::HostAutomaton &automaton(const ridfa_program *p, int dfa) { return dfa ? p->dfa : p->rid; }
}  // namespace

// A table's address; its size in bytes to *bytes.  Null: no table of that name.
extern "C" const void *ht_table(const ridfa_program *prog, int dfa, const char *name, uint64_t *bytes) {
    const ridfa::HostAutomaton &H = automaton(prog, dfa);
    const void *at = nullptr;
    auto take = [&](const char *n, const auto &v) {
        if (std::strcmp(n, name)) return;
        at = v.data();
        *bytes = v.size() * sizeof(v[0]);
    };
    take("trans", H.trans);
    take("classmap", H.classmap);
    take("final_bits", H.final_bits);
    take("ifmask", H.ifmask);
    take("slot_state", H.slot_state);
    take("merge.walk", H.merge.walk);
    take("merge.edge_pid", H.merge.edge_pid);
    take("merge.node_part", H.merge.node_part);
    take("merge.node_img", H.merge.node_img);
    take("merge.images", H.merge.images);
    take("merge.part", H.merge.part);
    take("merge.slot_alive", H.merge.slot_alive);
    take("stream.byte_code", H.stream.byte_code);
    take("stream.words", H.stream.words);
    take("set.next", H.set.next);
    take("set.leaf", H.set.leaf);
    take("set.images", H.set.images);
    take("set.part", H.set.part);
    take("set.block_mask", H.set.block_mask);
    take("set.words", H.set.table.words);
    take("set.back_next", H.set.back_next);
    take("set.back_images", H.set.back_images);
    return at;
}

// A number of the automaton or its tables; -1: none of that name.
extern "C" int64_t ht_number(const ridfa_program *prog, int dfa, const char *name) {
    const ridfa::HostAutomaton &H = automaton(prog, dfa);
    const struct {
        const char *name;
        int64_t value;
    } all[] = {
        {"n_states", H.n_states},        {"n_classes", H.n_classes},       {"k", H.k},
        {"merge.ok", H.merge.ok},        {"stream.kind", H.stream.kind},   {"stream.entry", H.stream.entry},
        {"stream.copies", H.stream.copies}, {"stream.group", H.stream.group}, {"stream.width", H.stream.width},
        {"set.ok", H.set.ok},            {"set.depth", H.set.depth},       {"set.back_depth", H.set.back_depth},
        {"set.group", H.set.table.group},
    };
    for (const auto &x : all)
        if (!std::strcmp(x.name, name)) return x.value;
    return -1;
}

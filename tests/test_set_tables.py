"""The set kernels' graphs against stepping the RI-DFA's table, on the host (no GPU): every string of the
graph's depth has to come to a leaf, because the kernels take what they come to for one, and the leaf's states
are those that the bytes leave."""
import numpy as np
import pytest

from tests import host_tables as ht
from tests.set_res import generated

lib = pytest.importorskip("paper_2412_14975_gb300")

FIXED = [("([ab]{5,6}|bb)*", b"ab"), ("((bab|aa[ab]|[ab]{5}))*[ab]*", b"ab"), ("(([ab]{4})*ba([ab]{4}){1,1}ba)*([ab]{4})*", b"ab"),
         ("(([ACGT]{3})*ATG([ACGT]{3}){2,4}(TAA|TAG|TGA))*[ACGT]*", b"ACGT"), ("(([ab]{12})*ab)*", b"ab"),
         ("(([ab]{3})*abab([ab]{3}){1,1}bab)*([ab]{3})*", b"ab")]


def walks_end(edges, depth):
    """Whether every walk of `depth` edges from node 0 has met a leaf; every index it meets is in bounds."""
    level = {0}
    for _ in range(depth):
        to = np.unique(edges[sorted(level)])
        level = {int(e) for e in to if not e & ht.KEEP}
        assert all(e < edges.shape[0] for e in level)
        if not level:
            return True
    return False


def set_programs(seed, count):
    for src, alphabet in FIXED + generated(seed, count):
        try:
            prog = lib.ridfa_compile(src, build_dfa=False, max_states=4000)
        except lib.RidfaError:                   # (too many states)
            continue
        if ht.number(prog, "set.ok"):
            yield src, alphabet, prog


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_set_graphs(seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    programs = backs = 0
    for src, alphabet, prog in set_programs(seed, 150):
        programs += 1
        trans, cmap, _ = lib.ridfa_export_tables(prog)
        n, classes = trans.shape[0] - 1, trans.shape[1]
        starts = np.array(list(lib.ridfa_slots(prog)), dtype=np.int64)
        nxt = ht.table(prog, "set.next", np.uint16).reshape(-1, classes)
        leaf = ht.table(prog, "set.leaf", np.uint32).reshape(-1, 2)
        images, part = ht.table(prog, "set.images", np.uint16), ht.table(prog, "set.part", np.uint8).reshape(-1, starts.size)
        depth, back = ht.number(prog, "set.depth"), ht.number(prog, "set.back_depth")
        assert depth <= 32 and walks_end(nxt, depth), src
        back_next = ht.table(prog, "set.back_next", np.uint16).reshape(-1, classes)
        back_images = ht.table(prog, "set.back_images", np.uint16).reshape(-1, ht.RUNS)
        if back:
            backs += 1
            assert back <= 32 and walks_end(back_next, back), src
        for _ in range(60):
            x = cmap[np.frombuffer(alphabet, dtype=np.uint8)[rng.integers(0, len(alphabet), 32)]]
            node, s, t = 0, starts.copy(), 0
            while not node & ht.KEEP:            # the slots' functions
                node = int(nxt[node, int(x[t])])
                s = trans[s, x[t]].astype(np.int64)
                t += 1
            pid, at = (int(v) for v in leaf[node & 0x7FFF])
            got = [n if b == 0xFF else int(images[at + b]) for b in part[pid].tolist()]
            assert got == s.tolist(), src
            if not back:
                continue
            node, s, t = 0, np.arange(n), 32 - back
            while not node & ht.KEEP:            # the sets that the last bytes leave of all states
                node = int(back_next[node, int(x[t])])
                s = trans[s, x[t]].astype(np.int64)
                t += 1
            want = np.unique(s[s < n])
            assert want.size < ht.RUNS, src
            row = back_images[node & 0x7FFF]
            assert np.array_equal(row[:want.size], want) and (row[want.size:] == n).all(), src
    assert programs > 30 and backs > 15

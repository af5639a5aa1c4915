"""GPU join scan at the edges of its launches: chunk counts around a warp's rows, a segment and a
block; one, several, exactly 32 and more end states per chunk; rejection in the first, a middle and
the last chunk.  Entry sets and the rejecting chunk against the recurrence written out on the host
over the same chunk maps (E_i = if_min(PLAS_{i-1}) ∩ PIS_i, Sec. 3.2), tolerance 0."""
import numpy as np
import pytest

import textgen
from tests.gpu_util import to_device

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

XS, YS = "ABCDEFGHIJKLMNOPQRSTUVWXYZ0123456789!#%&", "bcdefghijklmnopqrstuvwxyz<>=;:@$'\"^_`~,/"


def branches(nb):
    return "(" + "|".join(f"{XS[i]}a*{YS[i]}" for i in range(nb)) + ")*"


def recurrence(prog, maps):
    slot = lib.ridfa_delegates(prog)
    cache = {}

    def interface(p):
        if p not in cache:
            cache[p] = {int(slot[q]) for q in lib.ridfa_state_set(prog, p)}
        return cache[p]

    enter, entries, reject = {int(slot[0])}, [], -1
    for i, row in enumerate(maps):
        e = {a for a in enter if row[a] != 0xFFFF}
        entries.append(e)
        if not e and reject < 0:
            reject = i
        enter = set().union(*(interface(int(row[a])) for a in e)) if e else set()
    return entries, reject


def check(prog, maps):
    c, k = maps.shape
    kw = (k + 31) // 32
    d = torch.from_numpy(maps.view(np.int16).copy()).to("cuda:0")
    ent = torch.full((c, kw), -1, dtype=torch.int32, device="cuda:0")
    rej = lib.ridfa_join_scan(prog, d, c, ent)
    entries, want = recurrence(prog, maps)
    assert rej == want
    bits = np.unpackbits(ent.cpu().numpy().view(np.uint8), axis=1, bitorder="little")
    for i in range(c):
        assert set(np.nonzero(bits[i])[0].tolist()) == entries[i], i


def maps_of(prog, x, c):
    m = torch.empty((c, prog.info["k"]), dtype=torch.int16, device="cuda:0")
    lib.ridfa_recognize(prog, to_device(x), x.size, c, d_chunk_maps=m)
    return m.cpu().numpy().view(np.uint16)


@pytest.mark.parametrize("c", [1, 2, 7, 8, 9, 31, 32, 33, 34, 63, 65, 255, 257, 1023, 1057])
def test_scan_chunk_counts(c):
    for re_src, x in ((textgen.C3_RE, textgen.c3_text(30_000, seed=c)),
                      (textgen.C2_RE.replace("{20,60}", "{2,4}"), textgen.c2_text(30_000, seed=c)),
                      (textgen.regexp_family_re(3), textgen.regexp_family_text(30_000, seed=c))):
        prog = lib.ridfa_compile(re_src, build_dfa=False)
        good = maps_of(prog, x, c)
        check(prog, good)
        for at in sorted({0, c // 2, c - 1}):          # every run of one chunk dies
            bad = good.copy()
            bad[at] = 0xFFFF
            check(prog, bad)


@pytest.mark.parametrize("nb", [2, 31, 32, 33, 40])
def test_scan_end_states(nb):
    rng = np.random.Generator(np.random.PCG64(nb))
    prog = lib.ridfa_compile(branches(nb), build_dfa=False)
    text = "".join(XS[i] + "a" * int(rng.integers(0, 200)) + YS[i] for i in rng.integers(nb, size=120))
    x = np.frombuffer(text.encode(), dtype=np.uint8)
    for c in (33, 257, 1000):
        check(prog, maps_of(prog, x, c))
    y = x.copy()
    y[x.size // 2] = ord(YS[0])
    check(prog, maps_of(prog, y, 257))

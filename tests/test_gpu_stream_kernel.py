"""GPU stream kernels, every table form: chunk maps, accept bits, shard summaries and scans of the path that a
call takes by itself against the general kernels' (a fixed piece length), and of some chunks against stepping
the automaton's own table on the host.  Texts from one byte to ones of several pieces a lane, aligned and not,
chunks of one byte and up (whose functions do not merge), bytes outside the alphabet.  Tolerance 0."""
import numpy as np
import pytest

import textgen

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

RES = {
    "field4x1": ("(a|b)*a(a|b){3}", b"ab"),
    "field4x1_two_bits": ("[ACGT]*AC[ACGT]{2}T[ACGT]*", b"ACGT"),
    "field2x2": ("(a|b)*a(a|b){8}", b"ab"),
    "field4x2": ("(a|b)*a(a|b){9}", b"ab"),
    "field_apart": ("([ab]{5})*", b"ab"),                        # runs that never merge: every result a node
    "pair1": ("([a-p]{1,9}:[0-9a-f]{2,5};)*([q-z]{1,30}[!-/])*", b"abcmop:09af;"),
    "pair2": (textgen.C3_RE_ANYFIELD, None),
    "single1": ("(([a-h][i-p]){0,20}[0-9]{1,3};|[A-Z]{200}x)*", b"aibj09;"),
}
PROGS = {}


def program(name):
    if name not in PROGS:
        PROGS[name] = lib.ridfa_compile(RES[name][0])
    return PROGS[name]


def text(name, n, rng):
    re_src, alphabet = RES[name]
    if alphabet is None:
        return np.frombuffer(bytes(textgen.c3_text(n, rng)[:n]), dtype=np.uint8).copy()
    return np.frombuffer(alphabet, dtype=np.uint8)[rng.integers(0, len(alphabet), n)]


def on_device(x, offset):
    d = torch.zeros(x.size + 48, dtype=torch.uint8, device="cuda:0")
    d[offset:offset + x.size] = torch.from_numpy(x)
    return d[offset:]


def step(trans, cmap, starts, chunk):
    dead = trans.shape[0] - 1
    s = starts.copy()
    for b in cmap[chunk]:
        s = trans[s, b].astype(np.int64)
    return np.where(s == dead, 0xFFFF, s).astype(np.uint16)


@pytest.mark.parametrize("name", list(RES))
@pytest.mark.parametrize("n,counts", [(1, [1]), (5, [1, 2, 5]), (4093, [1, 4, 33, 700, 4093]), (70_001, [1, 64, 1_000, 30_000]),
                                      (1_200_003, [1, 7, 4_865, 400_001]), (30_000_001, [3, 155_649])])
def test_stream_forms(name, n, counts):
    prog = program(name)
    rng = np.random.Generator(np.random.PCG64(n))
    trans, cmap, _ = lib.ridfa_export_tables(prog)
    starts = np.array(list(lib.ridfa_slots(prog)), dtype=np.int64)
    x = text(name, n, rng)
    for variant in range(3):
        if variant:
            x = x.copy()
            x[rng.integers(0, n, 1 if variant == 1 else 1 + n // 5_000)] = ord("~")
        offset = (0, 5, 16)[variant]
        d = on_device(x, offset)
        want = lib.ridfa_cpu_recognize(prog, x, 1)
        for c in counts:
            maps = torch.full((c, prog.info["k"]), -7, dtype=torch.int16, device="cuda:0")
            ref = torch.full_like(maps, -9)
            got = lib.ridfa_recognize(prog, d, n, c, d_chunk_maps=maps)
            gen = lib.ridfa_recognize(prog, d, n, c, tuning=dict(piece_len=1 << 20), d_chunk_maps=ref)
            assert got == gen == want, (c, variant)
            assert torch.equal(maps, ref), (c, variant)
            assert lib.ridfa_recognize(prog, d, n, c) == want                       # (no maps asked for)
            dacc = torch.full((1,), 9, dtype=torch.uint8, device="cuda:0")
            lib.ridfa_recognize_async(prog, d, n, c, dacc)
            assert bool(dacc.item()) == want
            rows = maps.cpu().numpy().view(np.uint16)
            for i in {0, c // 3, c - 1}:
                lo, hi = i * n // c, (i + 1) * n // c
                if hi - lo <= 3_000:
                    assert np.array_equal(rows[i], step(trans, cmap, starts, x[lo:hi])), (c, i)
            if n < 2_000_000:
                assert lib.ridfa_join_scan(prog, maps, c) == lib.ridfa_join_scan(prog, ref, c)
                if n > 1:
                    h = n // 2
                    summaries = [lib.ridfa_recognize_shard(prog, d, h, min(c, h)),
                                 lib.ridfa_recognize_shard(prog, d[h:], n - h, min(c, n - h))]
                    assert lib.ridfa_join_shards(prog, summaries) == want


@pytest.mark.parametrize("name", ["field4x1", "pair1", "pair2", "single1"])
@pytest.mark.parametrize("n,c", [(4093, 4), (500_003, 1_000), (5_000_001, 77_825)])
def test_stream_dfa(name, n, c):
    prog = program(name)
    rng = np.random.Generator(np.random.PCG64(n + 1))
    x = text(name, n, rng)
    d = on_device(x, 3)
    q = lib.ridfa_export_tables(prog, 1)[0].shape[0] - 1
    maps = torch.full((c, q), -7, dtype=torch.int16, device="cuda:0")
    ref = torch.full_like(maps, -9)
    got = lib.ridfa_recognize_dfa(prog, d, n, c, d_chunk_maps=maps)
    gen = lib.ridfa_recognize_dfa(prog, d, n, c, tuning=dict(piece_len=1 << 20), d_chunk_maps=ref)
    assert got == gen == lib.ridfa_cpu_recognize(prog, x, 1)
    assert torch.equal(maps, ref)

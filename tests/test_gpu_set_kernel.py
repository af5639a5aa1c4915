"""GPU set kernels: automata over at most four bytes whose runs stay apart (the codon RE), a chunk or a
piece of one per lane.  Chunk maps against stepping the RI-DFA's own table on the host, the accept bit
against the serial host recognizer, with many and few chunks, short and ragged ones, aligned and unaligned
texts, bytes outside the alphabet, chunk counts around a warp's, a block's and a join block's; and the same
answers as the general kernel.  Tolerance 0."""
import numpy as np
import pytest

import textgen

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CODON = textgen.C2_RE.replace("{20,60}", "{2,4}")
FRAMES = "(([ACGT]{3})*A([ACGT]{3}){1,3}T)*[ACGT]*"          # 2,103 states: two bytes a lookup
BINARY = "(([ab]{2})*ab([ab]{2}){1,2}ba)*[ab]*"                # two bytes


def step_rows(prog, x, c, rows):
    trans, cmap, _ = lib.ridfa_export_tables(prog)
    dead = trans.shape[0] - 1
    start = np.array([s for s in lib.ridfa_slots(prog)], dtype=np.int64)
    cls = cmap[x]
    out = {}
    for i in rows:
        s = start.copy()
        for b in cls[i * x.size // c:(i + 1) * x.size // c]:
            s = trans[s, b].astype(np.int64)
        out[i] = np.where(s == dead, 0xFFFF, s).astype(np.uint16)
    return out


def check(re_src, x, c, offset=0):
    prog = lib.ridfa_compile(re_src, build_dfa=False)
    base = torch.from_numpy(np.concatenate([np.zeros(32, np.uint8), x])).to("cuda:0")
    d = torch.empty(x.size + 32, dtype=torch.uint8, device="cuda:0")
    d[offset:offset + x.size] = base[32:]
    maps = torch.full((c, prog.info["k"]), -7, dtype=torch.int16, device="cuda:0")
    acc = lib.ridfa_recognize(prog, d[offset:], x.size, c, d_chunk_maps=maps)
    got = maps.cpu().numpy().view(np.uint16)
    rng = np.random.Generator(np.random.PCG64(c))
    rows = sorted({i for i in (0, 1, 31, 32, c // 2, c - 33, c - 2, c - 1) if 0 <= i < c} | set(rng.integers(0, c, 40).tolist()))
    rows = rows[:400_000 // (x.size // c)]                   # (long chunks: against the general kernel alone)
    for i, want in step_rows(prog, x, c, rows).items():
        assert np.array_equal(got[i], want), (c, i)
    assert acc == lib.ridfa_cpu_recognize(prog, x, 1)
    ref = torch.empty_like(maps)
    racc = lib.ridfa_recognize(prog, d[offset:], x.size, c, tuning=dict(piece_len=1), d_chunk_maps=ref)
    assert racc == acc and torch.equal(ref, maps)
    dacc = torch.full((1,), 9, dtype=torch.uint8, device="cuda:0")
    lib.ridfa_recognize_async(prog, d[offset:], x.size, c, dacc)
    torch.cuda.synchronize()
    assert bool(dacc.item()) == acc


@pytest.mark.parametrize("c", [38913, 38944, 40001, 65536, 131073])
def test_set_chunk_counts(c):
    x = textgen.c2_text(c * 131 + 17, seed=c)
    check(CODON, x, c)
    check(CODON, x, c, offset=5)


@pytest.mark.parametrize("per", [31, 32, 33, 64, 95, 127, 128, 129, 159, 160, 161, 300, 1000])
def test_set_chunk_lengths(per):
    c = 39000
    x = textgen.c2_text(c * per + 1, seed=per)
    check(CODON, x, c, offset=per % 32)
    y, _ = textgen.mutate(x, seed=per, n_subs=40, alphabet=b"ACGTNacgt\\n")
    check(CODON, y, c)


@pytest.mark.parametrize("re_src,alphabet", [(FRAMES, b"ACGT"), (BINARY, b"ab"), ("(([ACGT]{3})*ATG([ACGT]{3}){1,2}TAA)*[ACGT]*", b"ACGT")])
def test_set_other_res(re_src, alphabet):
    rng = np.random.Generator(np.random.PCG64(7))
    x = np.frombuffer(alphabet, dtype=np.uint8)[rng.integers(0, len(alphabet), 40_000 * 150)]
    check(re_src, x, 40_000, offset=3)
    y = x.copy()
    y[y.size // 3] = ord("Z")
    check(re_src, y, 40_000)


@pytest.mark.parametrize("c,per", [(1, 20_000_003), (2, 9_000_001), (67, 300_017), (1024, 19_001), (1030, 40_507), (4096, 5_003), (30_000, 701),
                                   (1, 32), (1, 128), (1, 511), (1, 512), (3, 1_400), (33, 1_000), (80, 64), (5045, 64)])
@pytest.mark.parametrize("re_src,alphabet", [(CODON, None), (BINARY, b"ab")])
def test_set_pieces(re_src, alphabet, c, per):
    """Few chunks, cut into pieces: one level of composition and several, ragged groups of pieces."""
    n = c * per + c // 3
    if alphabet is None:
        x = textgen.c2_text(n, seed=c)
    else:
        x = np.frombuffer(alphabet, dtype=np.uint8)[np.random.Generator(np.random.PCG64(c)).integers(0, len(alphabet), n)]
    check(re_src, x, c, offset=c % 32)
    y = x.copy()
    y[n // 2] = ord("Z")
    check(re_src, y, c)

"""GPU set kernels where many runs stay alive: automata that keep nine to fifteen runs, in warps whose lanes
have different numbers of blocks (chunks of some two to five blocks with ragged ends; a batch's texts of
different lengths), so that a lane ends its blocks with more runs than the lanes that go on.  Every entry of
the chunk maps against the general kernels' and, by rows, against stepping the RI-DFA's table; a batch's accept
bits against the serial host recognizer.  Tolerance 0."""
import numpy as np
import pytest

from tests.test_gpu_set_kernel import check

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

RES = [("(([ab]{4})*ba([ab]{4}){1,1}ba)*([ab]{4})*", b"ab"), ("(([ab]{3})*abab([ab]{3}){1,1}bab)*([ab]{3})*", b"ab"),
       ("(([ab]{12})*ab)*", b"ab"), ("(([ACGT]{4})*AAT([ACGT]{4}){1,2}TAA)*([ACGT]{3})*", b"ACGT"),
       ("(([ACGT]{5})*ACG([ACGT]{5}){1,2}TAA)*[ACGT]*", b"ACGT")]


@pytest.mark.parametrize("re_src,alphabet", RES)
@pytest.mark.parametrize("per", [70, 128, 130, 150, 160, 200, 280, 300, 320])
def test_set_many_runs(re_src, alphabet, per):
    c = 40_000
    rng = np.random.Generator(np.random.PCG64(per))
    x = np.frombuffer(alphabet, dtype=np.uint8)[rng.integers(0, len(alphabet), c * per + 7)]
    check(re_src, x, c, offset=per % 32)
    y = x.copy()
    y[rng.integers(0, y.size, c // 4)] = ord("Z")            # (lanes whose runs all die beside the others)
    check(re_src, y, c)


@pytest.mark.parametrize("n_texts", [500, 530])
def test_set_batch_mixed_lengths(n_texts):
    """Texts of two pieces that keep their thirteen runs beside longer pieces that soon have one.  The second
    program's text is so long that the set texts get one SM, and pieces of 2 KB."""
    rng = np.random.Generator(np.random.PCG64(n_texts))
    ab = np.frombuffer(b"ab", dtype=np.uint8)
    progs = [lib.ridfa_compile("(([ab]{12})*(aababba|c))*", build_dfa=False), lib.ridfa_compile("(a|b)*a(a|b){3}", build_dfa=False)]
    texts = []
    for i in range(n_texts):
        short = i % 4 == 0                       # its pieces are the shorter ones
        n = int(rng.integers(2300, 2800)) if short else int(rng.integers(1600, 1950))
        x = b""
        while len(x) < n - 19:
            m = n // 12 if short else int(rng.integers(0, 7))
            x += ab[rng.integers(0, 2, 12 * min(m, (n - 7 - len(x)) // 12))].tobytes()
            x += b"aababba" if rng.integers(0, 2 if short else 8) == 0 else b"c"
        texts.append(np.frombuffer(x if i % 3 else x[:-1], dtype=np.uint8).copy())
    want = [lib.ridfa_cpu_recognize(progs[0], x, 1) for x in texts]
    assert 50 < sum(want) < n_texts
    at = np.cumsum([0] + [x.size + i % 19 for i, x in enumerate(texts)])
    buf = np.zeros(int(at[-1]), dtype=np.uint8)
    for x, o in zip(texts, at):
        buf[o:o + x.size] = x
    d = torch.from_numpy(buf).to("cuda:0")
    long = torch.full((600_000_000,), ord("a"), dtype=torch.uint8, device="cuda:0")
    acc = torch.full((n_texts + 1,), 7, dtype=torch.uint8, device="cuda:0")
    b = lib.ridfa_batch_create(progs, [(d[int(o):], x.size, 0, 0) for x, o in zip(texts, at)] + [(long, long.numel(), 1, 0)], acc, chunk_len=8192)
    lib.ridfa_batch_run(b)
    torch.cuda.synchronize()
    got = acc.cpu().numpy()
    lib.ridfa_batch_free(b)
    assert got[-1] == 1
    assert [bool(v) for v in got[:-1]] == [bool(w) for w in want]

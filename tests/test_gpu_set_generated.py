"""GPU set kernels on generated REs of two to four letters (tests/set_res.py) whose set tables are built: every
entry of the chunk maps, with chunks cut into pieces (pieces entered with the sets that the bytes before leave of
all states, and REs without such sets), short uneven chunks, and batches of mixed lengths.  Against the general
kernels, by rows against stepping the RI-DFA's table, accept bits against the serial host recognizer.  Tolerance
0."""
import numpy as np
import pytest

from tests import host_tables as ht
from tests.set_res import generated
from tests.test_gpu_set_kernel import check

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def set_res(seed, count):
    out = []
    for src, alphabet in [("([ab]{5,6}|bb)*", b"ab"), ("((bab|aa[ab]|[ab]{5}))*[ab]*", b"ab")] + generated(seed, 400):
        try:
            prog = lib.ridfa_compile(src, build_dfa=False, max_states=4000)
        except lib.RidfaError:                   # (too many states)
            continue
        if ht.number(prog, "set.ok"):
            out.append((src, alphabet, ht.number(prog, "set.back_depth")))
    backs, others = [r for r in out if r[2]], [r for r in out if not r[2]]
    return backs[:count] + others[:count // 3]


def text(alphabet, n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return np.frombuffer(alphabet, dtype=np.uint8)[rng.integers(0, len(alphabet), n)]


@pytest.mark.parametrize("seed", [11, 12])
@pytest.mark.parametrize("c,per", [(1, 600_011), (3, 40_007), (67, 9_001), (700, 1_537), (3_000, 513), (40_000, 131)])
def test_set_generated(seed, c, per):
    res = set_res(seed, 24)
    assert len(res) >= 24
    for i, (src, alphabet, _) in enumerate(res):
        x = text(alphabet, c * per + c // 3, seed * 1000 + i)
        check(src, x, c, offset=(i * 7) % 32)
        if i % 4 == 0:
            y = x.copy()
            y[y.size // 2] = ord("Z")
            check(src, y, c)


@pytest.mark.parametrize("seed", [21, 22])
def test_set_generated_batches(seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    res = set_res(seed, 18)
    progs = [lib.ridfa_compile(r[0], build_dfa=False) for r in res]
    items, want, keep = [], [], []
    for p, (src, alphabet, _) in enumerate(res):
        for i in range(60):
            n = int(rng.integers(32, 601)) if i % 4 else int(rng.integers(600, 9_000))
            x = text(alphabet, n, seed * 100_000 + p * 100 + i).copy()
            if i % 7 == 3:
                x[rng.integers(0, n)] = ord("#")
            d = torch.from_numpy(np.concatenate([np.zeros(i % 23, np.uint8), x])).to("cuda:0")
            keep.append(d)
            items.append((d[i % 23:], n, p, 0))
            want.append(bool(lib.ridfa_cpu_recognize(progs[p], x, 1)))
    assert 0 < sum(want) < len(want)
    acc = torch.full((len(items),), 7, dtype=torch.uint8, device="cuda:0")
    b = lib.ridfa_batch_create(progs, items, acc, chunk_len=8192)
    lib.ridfa_batch_run(b)
    torch.cuda.synchronize()
    got = [bool(v) for v in acc.cpu().numpy()]
    lib.ridfa_batch_free(b)
    assert got == want

"""Batches over programs of every table form, with and without the large ones' launches: empty texts, texts
around a piece's and a block's sizes, unaligned texts, texts whose pieces do not merge, more programs than
one launch takes.  Accept bits against the serial host recognizer.  Tolerance 0."""
import numpy as np
import pytest

import textgen

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CODON = textgen.C2_RE.replace("{20,60}", "{2,4}")
RES = [
    (CODON, b"ACGT"),                                            # set kernels, four bytes a lookup
    ("(([ACGT]{3})*A([ACGT]{3}){1,3}T)*[ACGT]*", b"ACGT"),       # set kernels, two bytes a lookup
    ("(a|b)*a(a|b){3}", b"ab"),                                  # field codes, one-byte entries
    ("(a|b)*a(a|b){8}", b"ab"),                                  # field codes, two-byte entries
    ("([a-f]+[0-4]{1,3};)*", b"abcdef01234;"),                   # two bytes a lookup
    ("([a-p]{1,9}:[0-9a-f]{2,5};)*([q-z]{1,30}[!-/])*", b"abcdefghijklmnopqrstuvwxyz0123456789:;"),
    ("([ab]{5})*", b"ab"),                                       # every run stays apart
]
LENS = [0, 1, 2, 31, 33, 127, 128, 129, 1023, 1024, 1025, 1500, 4097, 65_537, 300_001]


def good_text(re_src, alphabet, n, rng):
    """A text of n bytes, of the language where that is easy."""
    if b";" in alphabet:
        unit = b"abc012;" if alphabet[:1] == b"a" and len(alphabet) == 12 else b"kmo:9af;"
        return np.frombuffer((unit * (n // len(unit) + 1))[:n], dtype=np.uint8).copy()
    return np.frombuffer(alphabet, dtype=np.uint8)[rng.integers(0, len(alphabet), n)]


@pytest.mark.parametrize("lens,large", [(LENS, 0), (LENS, 2_500_003), (LENS[:6], 0), ([4096] * 3, 40_000_000)])
@pytest.mark.parametrize("copies", [1, 11])
def test_batch_forms(lens, large, copies):
    rng = np.random.Generator(np.random.PCG64(len(lens) + large))
    progs, items, want, keep = [], [], [], []
    for c in range(copies):
        for re_src, alphabet in RES:
            prog = lib.ridfa_compile(re_src, build_dfa=False)
            progs.append(prog)
            if c >= 2 and c < copies - 1:
                continue                                         # (programs without texts between others)
            for i, n in enumerate(lens + ([large] if large and c == 0 else [])):
                x = good_text(re_src, alphabet, n, rng)
                if n > 4 and i % 3 == 1:
                    x[rng.integers(0, n)] = ord("#")
                off = int(rng.integers(0, 17)) if i % 2 else 0
                d = torch.zeros(n + 64, dtype=torch.uint8, device="cuda:0")
                d[off:off + n] = torch.from_numpy(x)
                keep.append(d)
                items.append((d[off:], n, len(progs) - 1, 0))
                want.append(lib.ridfa_cpu_recognize(prog, x, 1) if n else None)
    acc = torch.full((len(items),), 7, dtype=torch.uint8, device="cuda:0")
    b = lib.ridfa_batch_create(progs, items, acc)
    for _ in range(2):
        acc.fill_(7)
        lib.ridfa_batch_run(b)
        torch.cuda.synchronize()
        got = acc.cpu().numpy()
        for i, w in enumerate(want):
            if w is None:
                w = lib.ridfa_recognize(progs[items[i][2]], items[i][0], 0, 0)
            assert got[i] == int(w), (i, items[i][1], RES[items[i][2] % len(RES)][0])
    lib.ridfa_batch_free(b)

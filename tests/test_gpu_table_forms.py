"""GPU stream kernels on the table forms, each asserted to be the one that runs: fields of one and two bits by two
and four bytes a lookup, pairs and single bytes, entries of one and two bytes, few and many lane copies.  Chunk
maps against the general kernels' and accept bits against the serial host recognizer, single texts and batches.
Tolerance 0."""
import numpy as np
import pytest

from tests import host_tables as ht

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

# RE, letters, (kind, bytes a lookup, bytes an entry, field bits, lane copies)
FORMS = [
    ("((A|C)*G(T|A)+C)*", b"ACGT", (ht.FIELD, 4, 1, 2, 32)),
    ("[ACGT]*(AC|GT)[ACGT]{4}", b"ACGT", (ht.FIELD, 4, 1, 2, 16)),
    ("[ACGT]*A[ACGT]{5}", b"ACGT", (ht.FIELD, 2, 1, 2, 32)),
    ("[ACGT]*A[ACGT]{7}", b"ACGT", (ht.FIELD, 4, 2, 2, 1)),
    ("(a|b)*a(a|b){10}", b"ab", (ht.FIELD, 4, 2, 1, 2)),
    ("[a-e]*a[a-e]{7}", b"abcde", (ht.PAIR, 2, 2, 0, 16)),
    ("[a-e]*a[a-e]{9}", b"abcde", (ht.PAIR, 2, 2, 0, 4)),
    ("([a-p]{1,9}:[0-9a-f]{2,5};)*([q-z]{1,30}[!-/])*", b"kmo:9af;", (ht.PAIR, 2, 1, 0, 32)),
    ("([a-h][0-9]){0,9}[a-h]*a[a-h]{7}", b"abcdefgh", (ht.SINGLE, 1, 2, 0, 32)),
    ("(([a-h][i-p]){0,20}[0-9]{1,3};|[A-Z]{200}x)*", b"aibj09;", (ht.SINGLE, 1, 1, 0, 32)),
]


def compiled(re_src, form):
    prog = lib.ridfa_compile(re_src, build_dfa=False)
    assert tuple(ht.number(prog, "stream." + n) for n in ("kind", "group", "entry", "width", "copies")) == form
    return prog


def letters(alphabet, n, seed):
    return np.frombuffer(alphabet, dtype=np.uint8)[np.random.Generator(np.random.PCG64(seed)).integers(0, len(alphabet), n)].copy()


@pytest.mark.parametrize("re_src,alphabet,form", FORMS)
@pytest.mark.parametrize("n,counts", [(70_001, [1, 64, 30_000]), (3_000_017, [1, 7, 4_865, 1_000_003]), (20_000_003, [155_649])])
def test_form_texts(re_src, alphabet, form, n, counts):
    prog = compiled(re_src, form)
    x = letters(alphabet, n, n)
    for variant in range(2):
        if variant:
            x[np.random.Generator(np.random.PCG64(1)).integers(0, n, 1 + n // 5_000)] = ord("~")
        off = 5 * variant
        d = torch.zeros(n + 48, dtype=torch.uint8, device="cuda:0")
        d[off:off + n] = torch.from_numpy(x)
        want = lib.ridfa_cpu_recognize(prog, x, 1)
        for c in counts:
            maps = torch.full((c, prog.info["k"]), -7, dtype=torch.int16, device="cuda:0")
            ref = torch.full_like(maps, -9)
            got = lib.ridfa_recognize(prog, d[off:], n, c, d_chunk_maps=maps)
            ran = lib.ridfa_last_kernel(prog)
            if ran["kernel"] == "stream":
                assert (ran["lookup_bytes"], ran["entry_bytes"], ran["lane_copies"]) == (form[1], form[2], form[4])
            else:
                assert ran["kernel"] == "stream_walk" and n <= 2 << 20
            assert n < 3_000_000 or ran["kernel"] == "stream"
            gen = lib.ridfa_recognize(prog, d[off:], n, c, tuning=dict(piece_len=1 << 20), d_chunk_maps=ref)
            assert lib.ridfa_last_kernel(prog)["kernel"] == "general"
            assert got == gen == want, (c, variant)
            assert torch.equal(maps, ref), (c, variant)


@pytest.mark.parametrize("large", [0, 20_000_003])
def test_form_batches(large):
    progs = [compiled(r, f) for r, _, f in FORMS]
    items, want, keep = [], [], []
    for p, (_, alphabet, _) in enumerate(FORMS):
        for i, n in enumerate([1, 33, 4_097, 65_537, 300_001] + ([large] if large else [])):
            x = letters(alphabet, n, 10 * p + i)
            if i == 3:
                x[n // 2] = ord("#")
            d = torch.from_numpy(np.concatenate([np.zeros(i * 3, np.uint8), x])).to("cuda:0")
            keep.append(d)
            items.append((d[i * 3:], n, p, 0))
            want.append(bool(lib.ridfa_cpu_recognize(progs[p], x, 1)))
    acc = torch.full((len(items),), 7, dtype=torch.uint8, device="cuda:0")
    b = lib.ridfa_batch_create(progs, items, acc, chunk_len=8192)
    lib.ridfa_batch_run(b)
    torch.cuda.synchronize()
    got = [bool(v) for v in acc.cpu().numpy()]
    lib.ridfa_batch_free(b)
    assert got == want

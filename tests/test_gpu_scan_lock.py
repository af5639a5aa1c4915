"""GPU join scan beside other calls of its program: while a scan waits for its stream the program is not locked,
and scans of several threads on one stream get their own results."""
import threading

import numpy as np
import pytest

import textgen
from tests.gpu_util import to_device
from tests.test_gpu_scan_edges import maps_of

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CODON = textgen.C2_RE.replace("{20,60}", "{2,4}")


def test_scan_does_not_lock_the_program():
    prog = lib.ridfa_compile(textgen.C3_RE, build_dfa=False)
    maps = to_device(maps_of(prog, textgen.c3_text(30_000, seed=1), 300).view(np.uint8))
    torch.cuda.synchronize()
    torch.cuda._sleep(3_000_000_000)                         # 1.5 s of the stream that the scan goes to
    out = []
    t = threading.Thread(target=lambda: out.append(lib.ridfa_join_scan(prog, maps, 300)))
    t.start()
    t.join(0.3)
    assert t.is_alive()
    lib.ridfa_last_plan(prog)                                # takes the program's lock
    assert t.is_alive()
    t.join()
    assert out == [-1]


@pytest.mark.parametrize("re_src,make", [(textgen.C3_RE, textgen.c3_text), (CODON, textgen.c2_text)])
def test_scans_of_several_threads(re_src, make):
    prog = lib.ridfa_compile(re_src, build_dfa=False)
    c = 3_000
    good = maps_of(prog, make(c * 40, seed=2), c)
    ats = [None, 0, 1_500, c - 1]
    rows = []
    for at in ats:
        m = good.copy()
        if at is not None:
            m[at] = 0xFFFF
        rows.append(to_device(m.view(np.uint8)))
    got = [[] for _ in ats]

    def scans(i):
        torch.cuda.set_device(0)
        for _ in range(40):
            got[i].append(lib.ridfa_join_scan(prog, rows[i], c))

    threads = [threading.Thread(target=scans, args=(i,)) for i in range(len(ats))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for at, g in zip(ats, got):
        assert g == [-1 if at is None else at] * 40

"""GPU join scan of chunks with several end states over more boundaries than its launches take at a time: chunk
counts around one and two such tiles, rejections at their edges; entry sets and the rejecting chunk against the
recurrence on the host.  The device memory that a scan leaves taken.  Tolerance 0."""
import numpy as np
import pytest

import textgen
from tests.test_gpu_scan_edges import check, maps_of

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CODON = textgen.C2_RE.replace("{20,60}", "{2,4}")
TILE = 1 << 18


@pytest.mark.parametrize("c", [TILE, TILE + 1, TILE + 2, 2 * TILE + 2])
def test_scan_tiles(c):
    prog = lib.ridfa_compile(CODON, build_dfa=False)
    good = maps_of(prog, textgen.c2_text(c * 33 + 5, seed=c), c)
    check(prog, good)
    for at in sorted({TILE, TILE + 1, c - 1}):
        if at < c:
            bad = good.copy()
            bad[at] = 0xFFFF
            check(prog, bad)


def test_scan_keeps_little_memory():
    """A scan's working space does not grow with the chunks: 2**20 of them would take 138 MB at once."""
    c = 1 << 20
    maps = torch.from_numpy(maps_of(lib.ridfa_compile(CODON, build_dfa=False), textgen.c2_text(c * 32, seed=5), c).view(np.int16).copy()).to("cuda:0")
    prog = lib.ridfa_compile(CODON, build_dfa=False)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    assert lib.ridfa_join_scan(prog, maps, c) == -1
    assert before - torch.cuda.mem_get_info()[0] <= 56 << 20     # (tables, 2 MB; working space, 35 MB; whole pages)

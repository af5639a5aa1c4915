"""What ridfa_last_kernel says of stream, set and general calls, beside ridfa_last_plan's plan of the general one."""
import numpy as np
import pytest

import textgen

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def test_last_kernel():
    codon = lib.ridfa_compile(textgen.C2_RE.replace("{20,60}", "{2,4}"), build_dfa=False)
    x = torch.from_numpy(np.array(textgen.c2_text(1 << 20, seed=1))).to("cuda:0")
    with pytest.raises(lib.RidfaError):
        lib.ridfa_last_kernel(codon)                         # no call yet
    lib.ridfa_recognize(codon, x, 1 << 20, 1000)
    ran = lib.ridfa_last_kernel(codon)
    assert (ran["kernel"], ran["lookup_bytes"], ran["pieces_per_chunk"]) == ("set", 4, 4)
    assert lib.ridfa_last_plan(codon)["text_path"] == 5      # (the general kernels' plan for it)
    assert lib.ridfa_last_kernel(codon)["kernel"] == "set"
    lib.ridfa_recognize(codon, x, 1 << 20, 1000, tuning=dict(table_mode=9))
    ran = lib.ridfa_last_kernel(codon)
    assert ran["kernel"] == "general" and ran["block_threads"] == lib.ridfa_last_plan(codon)["block_threads"]
    records = lib.ridfa_compile(textgen.C3_RE, build_dfa=False)
    y = torch.from_numpy(np.array(textgen.c3_text(4096, seed=2))).to("cuda:0")
    lib.ridfa_recognize(records, y, 4096, 4)
    assert lib.ridfa_last_kernel(records)["kernel"] == "stream_walk"

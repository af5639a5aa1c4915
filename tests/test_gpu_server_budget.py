"""What a server's device budget counts, against the device memory that the same tables and batches take."""
import numpy as np
import pytest

import textgen

pytestmark = pytest.mark.gpu

lib = pytest.importorskip("paper_2412_14975_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("re_src,alphabet", [("(a|b)*a(a|b){3}", b"ab"), ("(([ab]{2})*ab([ab]{2}){1,2}ba)*[ab]*", b"ab"),
                                             (textgen.C2_RE.replace("{20,60}", "{2,4}"), b"ACGT"), (textgen.C3_RE, b"2024-01,")])
@pytest.mark.parametrize("n", [40_000, 1_000_003, 8_000_000])
def test_request_charge_covers_its_scratch(re_src, alphabet, n):
    prog = lib.ridfa_compile(re_src, build_dfa=False)
    x = np.frombuffer(alphabet, dtype=np.uint8)[np.random.Generator(np.random.PCG64(n)).integers(0, len(alphabet), n)]
    d = torch.from_numpy(x).to("cuda:0")
    with lib.Server(n_streams=1, arena_bytes=1 << 20, device_budget=1 << 30) as srv:
        slot = srv.add_program(prog)
        assert srv.stats()["table_bytes"] == prog.info["table_bytes"]
        srv.submit(slot, d.data_ptr(), length=n, device=True)
        srv.drain()
        st = srv.stats()
        charge = st["budget_peak"] - st["table_bytes"]
        assert st["budget_used"] == st["table_bytes"]
    acc = torch.zeros(1, dtype=torch.uint8, device="cuda:0")

    def device_bytes(m):
        b = lib.ridfa_batch_create([prog], [(d, m, 0, 0)], acc, chunk_len=1024)
        out = lib.ridfa_batch_get_stats(b)["device_bytes"]
        lib.ridfa_batch_free(b)
        return out

    # (8 KB: the launches' descriptors of a batch on all SMs, which the budget leaves out)
    assert device_bytes(n) - device_bytes(4096) <= charge + 8192

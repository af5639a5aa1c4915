"""ridfa_info's table bytes (what a server's device budget is charged) against the tables that go to the device,
counted one by one: every table of every kernel the automaton may take, each on a 256-byte boundary."""
import numpy as np
import pytest

import textgen
from tests import host_tables as ht

lib = pytest.importorskip("paper_2412_14975_gb300")

ALL = ["trans", "classmap", "final_bits", "ifmask", "slot_state"]
STREAM = ["merge.walk", "merge.edge_pid", "merge.node_part", "merge.node_img", "merge.images", "merge.part", "merge.slot_alive",
          "stream.byte_code", "stream.words"]
SET = ["set.next", "set.leaf", "set.images", "set.part", "set.block_mask", "set.words", "set.back_next", "set.back_images"]


@pytest.mark.parametrize("re_src", ["(a|b)*a(a|b){3}", textgen.C3_RE, textgen.C3_RE_ANYFIELD, textgen.C2_RE.replace("{20,60}", "{2,4}"),
                                    "(([ab]{12})*ab)*", "([0-9]+,[a-z]+\n)*"])
def test_table_bytes_count_every_table(re_src):
    prog = lib.ridfa_compile(re_src)
    for dfa, got in ((False, prog.info["table_bytes"]), (True, prog.info["dfa_table_bytes"])):
        names = ALL + (STREAM if ht.number(prog, "stream.kind", dfa) else []) + (SET if ht.number(prog, "set.ok", dfa) else [])
        sizes = [ht.table(prog, n, np.uint8, dfa).size for n in names] + [2 * ht.number(prog, "n_states", dfa)]
        assert got == sum((s + 255) // 256 * 256 for s in sizes), dfa

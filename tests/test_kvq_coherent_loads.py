"""The KVQuant decode may start while the quantize launch before it still writes the cache, so no load of the cache goes
through the read-only path: every __ldg of its source is of a table that no kernel of a step writes."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_07966_gb300", "csrc",
                   "decode_kvq.cu")


def test_read_only_loads_are_of_tables():
    code = re.sub(r"//.*", "", open(SRC).read())
    loads = re.findall(r"__ldg\s*\(\s*([\w.]+)", code)
    assert loads and set(loads) <= {"a.rope", "a.k_dq", "a.v_tbl"}
    assert "ld.global.nc" not in code

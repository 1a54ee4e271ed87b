"""CPU: in the tensor-core kernels no path leaves a loop or a function between a
tcgen05.ld and the wait for it (the loads would run into registers that are
reused and into the release of TMEM)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_23169_gb300", "csrc")


def exits_with_loads_in_flight(src):
    """(line, text) of every break / return / continue in the source order between a load and its wait."""
    src = re.sub(r"//[^\n]*", "", src)
    found, in_flight = [], False
    for n, line in enumerate(src.split("\n"), 1):
        # calls only (a definition names a parameter list), left to right
        for m in re.finditer(r"tmem_(ld\w*|wait_ld)\s*\((?!\s*uint32_t)|\b(break|return|continue)\b", line):
            if m.group(2):
                if in_flight:
                    found.append((n, line.strip()))
            else:
                in_flight = m.group(1) not in ("wait_ld", "ld64")  # tmem_ld64 waits itself
    return found


@pytest.mark.parametrize("name", ["attn_fwd_tc.cu", "attn_bwd_tc.cu"])
def test_no_exit_between_a_tmem_load_and_its_wait(name):
    src = open(os.path.join(CSRC, name)).read()
    assert "tmem_ld" in src
    assert exits_with_loads_in_flight(src) == []


def test_the_scan_sees_an_exit():
    assert exits_with_loads_in_flight("tmem_ld32(a, r);\nif (!ok) break;\ntmem_wait_ld();\n") == [(2, "if (!ok) break;")]
    assert exits_with_loads_in_flight("tmem_ld32(a, r);\ntmem_wait_ld();\nif (!ok) break;\n") == []

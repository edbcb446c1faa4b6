"""Every wait for tensor-memory loads names the registers that the loads fill:
without them nothing orders the uses of the values behind the wait."""
import os
import re

import paper_2507_01439_gb300 as trg

CSRC = os.path.join(os.path.dirname(trg.__file__), "csrc")


def test_every_load_wait_is_tied_to_its_registers():
    waits = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"tcgen05\.wait::ld\.sync\.aligned;\"(.*?)\);", text, re.S):
            waits += 1
            assert '"+r"(v[0])' in m.group(1), (name, m.group(0))
    assert waits >= 2

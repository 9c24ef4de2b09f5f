"""A CTA of the tensor-core network ends only when what it started in its shared and
tensor memory is over, also after a wait that gave up: the warp that copies waits
for its last bulk copy, the warp that issues the MMAs for its last commit."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_05783_gb300", "csrc",
                   "k_net_tc.cu")


def _roles():
    code = re.sub(r"//[^\n]*", "", open(SRC).read())
    copy = code[code.index("if (warp == 5)"):code.index("} else if (warp == 4) {")]
    mma = code[code.index("} else if (warp == 4) {"):]
    return copy, mma[:mma.index("} else {\n    int it = 0;")]


def test_the_last_copy_is_waited_for():
    copy, _ = _roles()
    assert "mbar_wait(full" in copy[copy.rindex("bulk_g2s("):]


def test_the_last_mmas_are_waited_for():
    _, mma = _roles()
    assert "mbar_wait(done" in mma[mma.rindex("mma_commit("):]

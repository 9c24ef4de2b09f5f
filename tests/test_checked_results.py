"""No source file drops the answer of a function of the engine that says whether
it worked (cudaError_t or bool in cams_internal.h): not as a statement of its own."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_05783_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_no_result_is_dropped():
    names = re.findall(r"^(?:\[\[nodiscard\]\] )?(?:cudaError_t|bool) (\w+)\(", _code(os.path.join(CSRC, "cams_internal.h")), re.M)
    assert {"ilu_set_smem", "ilu_sweep_smem", "launch_residual", "raise_smem_limit"} <= set(names)
    dropped = [(os.path.basename(p), m.group(1)) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
               for m in re.finditer(r"[;{}]\s*(" + "|".join(sorted(set(names))) + r")\s*\(", _code(p))]
    assert dropped == []

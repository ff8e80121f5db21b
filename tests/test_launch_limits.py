"""A kernel's limit of dynamic shared memory (cudaFuncSetAttribute) belongs to the
function in the whole context, not to a launch: a call that sets it to what its
own sizes need can fail another host thread's larger launch.  Read from the
source: every such limit is made of constants and template arguments only."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1008_1371_gb300", "csrc")
# template arguments, constants derived from them, and functions of these
FIXED = {"size_t", "sizeof", "double", "int", "NN", "NNX", "C", "P", "R", "RX", "SMEM", "B", "update_smem", "TrainSmem",
         "persist_smem"}


def _fixed(expr):
    return all(w in FIXED or re.match(r"k[A-Z]\w*$", w) for w in re.findall(r"[A-Za-z_]\w*", expr))


def test_limits_do_not_depend_on_the_call():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            src = f.read()
        for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize,\s*(?:\(int\))?((?:[^()]|\([^()]*\))*)\)", src):
            seen += 1
            expr = m.group(1)
            if re.match(r"(?!k[A-Z])[a-z]\w*$", expr):  # a local: its definition just before
                d = re.findall(r"const size_t %s = ([^;]*);" % expr, src[:m.start()])
                assert d, (path, expr)
                expr = d[-1]
            assert _fixed(expr), (os.path.basename(path), expr)
    assert seen >= 12

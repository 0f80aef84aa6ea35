"""Kernels launched as programmatic dependents: what they read of earlier kernels' results through
const __restrict__ parameters is tied to the wait (LAUNDER), as such loads count as constant otherwise."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_17081_gb300", "csrc")
# parameters that hold tables of set-up, written before the first kernel of a chain
SETUP = {"tasks", "ss", "inv", "recs", "sh", "sunits", "items", "tshape", "tlist", "tcoff", "A", "rexp", "S", "Dinv"}
# read by bulk copies (asm with a memory clobber, behind the copy warp's own wait), not by loads
COPIED = {("k_dense_mma", "B")}


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s[^{;]*?\b(k_\w+)\(", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params = src[m.end():i - 1]
            j = src.index("{", i)
            depth, k = 1, j + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[k], 0)
                k += 1
            yield m.group(1), params, src[j:k]


CHAINED = [k for k in _kernels() if "CHAIN_ENTER" in k[2] or "griddepcontrol.wait" in k[2]]


def test_chained_kernels_are_found():
    assert {"k_zt", "k_arnoldi_step", "k_dense_mma", "k_dense_finish", "k_odots2_df", "k_dst_pass"} <= {k[0] for k in CHAINED}


@pytest.mark.parametrize("name,params,body", CHAINED, ids=[k[0] for k in CHAINED])
def test_results_of_earlier_kernels_are_tied_to_the_wait(name, params, body):
    const = set(re.findall(r"const\s[^,]*?\*__restrict__\s+(\w+)", params))
    tied = set(re.findall(r"LAUNDER\((\w+)\)", body))
    loose = {p for p in const - tied - SETUP if (name, p) not in COPIED}
    assert not loose, loose

"""The dynamic shared-memory limit of a kernel belongs to the process, not to a context: it is set in
one place, to the same value whatever the problem, so that a context in another host thread cannot
lower it between the setting and the launch."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_17081_gb300", "csrc")


def test_one_place_sets_the_limit_and_to_one_value():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        found += [(os.path.basename(path), m) for m in re.findall(r"cudaFuncSetAttribute\((.*?)\);", src, re.S)]
    assert [f for f, _ in found] == ["hdd_common.cuh"], found
    assert re.search(r"const int most = 227 \* 1024 - \(int\)a\.sharedSizeBytes;", open(os.path.join(CSRC, "hdd_common.cuh")).read())
    assert found[0][1].endswith(", most"), found

"""The status word names the wait that gave up: no two kernels use the same wait-site code (read from the sources; no GPU needed)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_13612_b200", "csrc")


def test_codes_of_different_kernels_are_different():
    seen = {}
    for path in glob.glob(os.path.join(CSRC, "*_kernel*.cuh")):
        with open(path) as f:
            codes = {int(c) for c in re.findall(r"mbar_wait\w*(?:<[^>]*>)?\(.*?abort_flag,\s*(\d+)\)", f.read())}
        for c in codes:
            assert c not in seen, (c, seen[c], os.path.basename(path))
            seen[c] = os.path.basename(path)
    assert len(seen) >= 60 and max(seen) < 0x7e   # (0x7e, 0x7f: the self-test's)

"""The form of the bounded waits in the matmul kernels, read from the source: it takes a barrier that never completes to
see the difference on a GPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_04985_b200", "csrc")

# the last argument of a wait: who waits.  1 TMA producer, 2 and 3 the thread that issues the tensor-core instructions,
# 11 the thread that issues a tile's TMA store; all other roles are whole warps
SINGLE_THREADS = {1, 2, 3, 11}


def test_whole_warps_leave_a_wait_as_one():
    """A warp whose lanes give up one by one never meets again in front of the warp-wide instructions that follow."""
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "gemm_*.cu"))):
        for line, text in enumerate(open(path), 1):
            for form, role in re.findall(r"\b(mbar_wait\w*)\([^!]*?, (\d+)\)", text):
                seen += 1
                where = f"{os.path.basename(path)}:{line}: {text.strip()}"
                assert (form == "mbar_wait_warp") == (int(role) not in SINGLE_THREADS), where
    assert seen >= 20

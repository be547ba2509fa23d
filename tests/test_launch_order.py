"""Programmatic dependent launch and tensor memory, from the sources: a kernel that allocates TMEM lets its successor start behind the
allocation only.  tcgen05.alloc blocks until columns are free; a successor's CTAs that held them while they wait for this kernel
would never give them back."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21759_b200", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for body in text.split("__global__")[1:]:
            yield os.path.basename(path), re.search(r"(\w+_kernel)\s*\(", body).group(1), body


def test_successors_start_behind_a_kernels_tmem_allocation():
    seen = {}
    for source, name, body in _kernels():
        at = body.find("tcgen05.alloc")
        if at >= 0 and "pdl_launch_dependents()" in body:
            seen[name] = body.find("pdl_launch_dependents()") > at
    assert set(seen) == {"gemm_kernel", "gemm_rows_kernel", "attention_tc_kernel"}
    assert all(seen.values()), seen

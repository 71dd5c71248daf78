"""Kernels that may start before the one ahead has ended (programmatic dependent launches) read the solver's state
by volatile loads: through a const __restrict__ pointer the compiler may take the path of read-only data."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_0330_gb300", "csrc")
FIELDS = "done|iter|alpha|beta|pq|rr|rz|tol2"


def kernels():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(f).read())
        for body in re.split(r"(?=__global__ )", code)[1:]:
            yield os.path.basename(f), re.search(r"\b(k_\w+)\s*\(", body).group(1), body


def test_chained_kernels_read_the_state_by_volatile_loads():
    chained = 0
    for name, kernel, body in kernels():
        head = body[:body.index("{")]
        if not re.search(r"\b(griddep_wait|chain_wait)\s*\(", body) or not re.search(r"const SolverState\*", head):
            continue
        chained += 1
        plain = re.sub(r"const_cast<const volatile \w+\*>\(&st\[s\]\.\w+\)", "", body)
        assert not re.search(r"\bst(\[[^\]]*\]\.|\s*->)\s*(%s)\b" % FIELDS, plain), (name, kernel)
    assert chained >= 8

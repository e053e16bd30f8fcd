"""Host-side check of the kernels that are launched as programmatic dependents."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1702_01335_gb300", "csrc")

# written by the host alone, before any launch that reads it
CONSTANT = {"insts", "tiles", "is_w"}


def dependents():
    """(kernel name, parameter list) of every kernel that waits for its predecessor itself."""
    out = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"//[^\n]*", "", open(f).read())
        for part in re.split(r"\b__global__\b", src)[1:]:
            m = re.match(r"\s*void\s*(?:__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^)]*)\)\s*\{", part)
            if m and re.search(r"\bwait_predecessor\s*\(\s*\)\s*;", part[:part.find("\n}\n")]):
                out.append((m.group(1), [p.strip() for p in m.group(2).split(",")]))
    return out


def test_dependents_read_what_kernels_write_by_ordinary_loads():
    """Such a kernel starts while the one before it still writes.  A `const __restrict__` parameter
    promises memory that nobody writes while the kernel runs: its loads may go through the
    read-only path and move above the wait.  Only tables that no kernel writes may be one."""
    found = dependents()
    assert {"stage_kernel", "finalize_cells", "forward_gemm", "backward_gemm", "adam"} <= {k for k, _ in found}
    bad = [(k, p) for k, ps in found for p in ps
           if "__restrict__" in p and re.match(r"const\b", p) and p.split()[-1].strip("*") not in CONSTANT]
    assert not bad, bad

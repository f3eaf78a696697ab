"""Kernels that start before the kernel ahead of them has ended (programmatic
dependents, griddep_wait) read its results with ordinary loads.  A const
__restrict__ parameter of a kernel takes the read-only path, which is for
data that nothing writes while the kernel runs: such a kernel may have only
parameters of that kind that are fixed before the chain begins.  Checked on
the sources (no run can show a stale read to be absent)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# factors, scales, patterns and A itself: written before the chain of launches
FIXED = {"Rcm", "Rrm", "Xcm", "Xrm", "dinv", "scale", "rp", "col", "val", "Ahi", "Alo", "items",
         # a panel's reflectors: complete before the update behind the next panel starts
         "vhead", "Tp", "Y"}


def _kernels():
    """(file, name, parameters, body) of every kernel that calls griddep_wait."""
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2406_03468_gb300", "csrc", "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        src = re.sub(r"__launch_bounds__\([^\n]*\)", "", src)
        for m in re.finditer(r"(?:__global__|__device__)[^;{}()]*?(\w+)\(([^{};]*)\)\s*\{", src):
            depth, i = 1, m.end()
            while depth and i < len(src):
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            if "griddep_wait()" in src[m.end():i]:
                yield os.path.basename(path), m.group(1), m.group(2), src[m.end():i]


def test_no_read_only_loads_of_dependent_data():
    seen = set()
    for path, name, params, body in _kernels():
        seen.add(name)
        ro = set(re.findall(r"const\s+\w+\s*\*__restrict__\s+(\w+)", params))
        assert ro <= FIXED, (path, name, ro - FIXED)
        for arg in re.findall(r"__ldg\(\s*(\w+)", body):
            assert arg in FIXED, (path, name, arg)
    assert {"reduce_kernel", "csr_pass_kernel", "df_pass_body", "inner_w_body"} <= seen

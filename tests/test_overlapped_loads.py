"""Kernels launched over their predecessor (launch_over) start before its
results are written.  Read-only loads (const __restrict__ parameters, __ldg) are
for data that no one writes during a kernel's whole life: in the sources of
those kernels only the mesh's tables, constants and the copy into element order
use them, and the switched load of a result is the read-only one only where the
launch does not overlap."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1006_0720_gb300", "csrc")
TABLES = {"tri", "dN", "nse_off", "nse", "xy", "geo", "nsw_line"}  # written once, with the mesh
LOADS = {"p", "p + 1", "p + 2", "reinterpret_cast<const int4*>(p + 3)", "reinterpret_cast<const int4*>(p + 4)",  # load_geo
         "src", "src + 1", "src + 2", "src + 3", "reinterpret_cast<const int*>(src + 3)",                       # F.geo + e
         "reinterpret_cast<const int2*>(src + 4)", "reinterpret_cast<const int*>(F.geo + e) + 18",
         "&kRecip.v[c]", "R.src8[k] + j", "R.src4[k] + j"}


def _text(name):
    s = open(os.path.join(SRC, name)).read()
    return re.sub(r"//[^\n]*", "", s)


def _balanced(s, i):
    """The text between the bracket at s[i] and its partner."""
    depth = 0
    for j in range(i, len(s)):
        depth += s[j] == "("
        depth -= s[j] == ")"
        if depth == 0:
            return s[i + 1:j]
    raise AssertionError("unbalanced")


def test_read_only_loads_in_overlapped_kernels():
    seen = set()
    for name in ("step.cu", "stats.cu"):
        s = _text(name)
        kernels = {m.group(2) for m in re.finditer(r"launch_over\(([^;]*?),\s*(k_\w+)", s)}
        for k in kernels:
            m = re.search(r"__global__ void (?:__launch_bounds__\([^)]*\)\s*)?%s\s*\(" % k, s)
            assert m, k
            params = _balanced(s, m.end() - 1)
            const = set(re.findall(r"const [\w:]+\s*\*\s*__restrict__\s+(\w+)", params))
            assert const <= TABLES, (k, const - TABLES)
            seen.add(k)
        for m in re.finditer(r"__ldg\(", s):
            arg = _balanced(s, m.end() - 1)
            assert arg in LOADS, (name, arg)
        # the load that is read-only in ordinary launches goes with its launch
        for over, kernel, args in re.findall(r"launch_over\(([^,;]*), (k_\w+)(<[^>]*>)", s):
            if kernel in ("k_step", "k_step_fx", "k_step_f32", "k_elem_stats_grp"):
                assert args.strip("<>").split(",")[-1].strip() == over, (kernel, over, args)
    assert {"k_step", "k_step_fx", "k_step_f32", "k_elem_stats_grp", "k_elem_rows", "k_reorder", "k_radix_scatter"} <= seen

"""Kernels that wait for a grid dependency read what the preceding kernel of the stream writes by ordinary
loads.  A programmatically launched grid is resident while its predecessor still writes; griddepcontrol.wait
orders the ordinary loads behind it, but a `const ... __restrict__` parameter lets the compiler take the
read-only path, which is defined only for memory that nobody writes during the whole grid.  CPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2006_08303_gb300", "csrc")


def closing(s, i, pair):
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == pair[0]) - (s[j] == pair[1])
        if depth == 0:
            return j
    raise ValueError("unbalanced")


def kernels():
    """(file, name, parameter list, body) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", src):
            k = re.compile(r"(\w+_kernel|shrink_dual_\w+)\s*\(").search(src, m.end())
            end = closing(src, k.end() - 1, "()")
            body = src.index("{", end)
            yield os.path.basename(path), k.group(1), src[k.end():end], src[body:closing(src, body, "{}") + 1]


def test_no_read_only_pointers_behind_a_grid_dependency():
    waiting, bad = [], []
    for file, name, params, body in kernels():
        if "grid_dep_wait()" not in body:
            continue
        waiting.append(name)
        for p in params.split(","):
            # tw: the twiddle tables, written once when the plan is created
            if "const" in p and "*" in p and "__restrict__" in p and p.split()[-1] != "tw":
                bad.append((file, name, p.strip()))
    assert {"dwt2_fwd_kernel", "dwt2_inv_fused_kernel", "wdct_shrink_kernel", "solve_split_kernel", "passA_kernel",
            "row_kernel", "colpass_fused_kernel", "coldirect_kernel", "cd_fused_kernel", "dl_spec_kernel"} <= set(waiting)
    assert not bad, bad

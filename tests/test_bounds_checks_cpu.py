"""Every source whose kernels gather through the sorted order or a neighbour list
checks those indices in the bounds-checked build."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_gathers_are_checked():
    seen = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2010_01559_gb300", "csrc", "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        if not re.search(r"\b(perm|iperm|nbr)\[", src):
            continue
        seen.append(os.path.basename(path))
        assert "RBE_IN_BOUNDS" in src, path
    assert {"rbe_small.cu", "rbe_real64.cu"} <= set(seen)

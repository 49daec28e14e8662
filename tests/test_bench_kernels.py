"""The kernel names that the benchmark prints for each class are kernels of the
library, and no kernel is missing (no GPU)."""
import glob
import os
import re

import bench
from paper_2008_12820_gb300 import build as B

# kernels outside the classes: the allocation-free preconditioner's tables
NO_CLASS = {"k_twiddles"}


def test_class_names_are_the_librarys_kernels():
    src = "".join(open(f).read() for f in glob.glob(os.path.join(B.SRC, "*.cu*")))
    src = re.sub(r"//[^\n]*", "", src)
    defined = set(re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(k[rg]?_\w+)", src))
    named = set(re.findall(r"\bk[rg]?_\w+", " ".join(bench.KNAMES.values())))
    assert len(defined) > 40
    assert named - defined == set()
    assert defined - named - NO_CLASS == set()

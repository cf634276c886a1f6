"""The hash that ties a committed profile to the kernel sources covers every file of
this repository that the compiler reads for the split update."""
import os
import re
import subprocess

import bench
from paper_1901_06798_gb300 import build

CSRC = os.path.join(bench.ROOT, "paper_1901_06798_gb300", "csrc")


def test_hash_covers_what_the_update_is_compiled_from():
    read = set()
    for unit in ("step_f64.cu", "step_f32p.cu"):
        r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-M", os.path.join(CSRC, unit)], capture_output=True,
                           text=True, check=True)
        files = [os.path.realpath(f) for f in re.findall(r"[^\s\\]+\.(?:cu|cuh|h)\b", r.stdout)]
        read |= {os.path.basename(f) for f in files if os.path.dirname(f) == os.path.realpath(CSRC)}
    assert {"step_tail.cuh", "chain.cuh"} <= read
    assert read == set(bench.kernel_sources())

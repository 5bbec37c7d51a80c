"""The server's HBM footprint of a job counts every record that a plan keeps per primitive pair."""

import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2407_09700_gb300.serve import footprint_bytes
from workloads import custom_molecule

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_09700_gb300", "csrc")


def test_primitive_pair_records_are_counted(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src = tmp_path / "sizes.cpp"
    src.write_text('#include "eri_internal.h"\n#include <cstdio>\n'
                   'int main() { printf("%zu\\n", sizeof(PrimPair) + sizeof(PrimPairF) + sizeof(PrimFx)); }\n')
    exe = str(tmp_path / "sizes")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    record = int(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)

    def job(depth):         # one s shell: depth (depth + 1) / 2 primitive pairs by the estimate, depth^2 at most
        m = custom_molecule(np.zeros((1, 3)), [(0, 0, 0.5 + np.arange(depth), np.ones(depth))])
        return footprint_bytes(m, "jk")

    # depth^2 primitive pairs of the one shell pair (every product is kept on one centre)
    assert job(40) - job(1) >= record * (40 ** 2 - 1)

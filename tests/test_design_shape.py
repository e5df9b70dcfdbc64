"""The domain of the design's stratum permutation (host logic, no GPU): the smallest power
of four that holds the N strata, and cycle walking wherever it holds more than N -- a value
past N that is not walked on is a stratum that does not exist (an index past the score
table of the correlation-reducing permutation, which takes one column of up to 2^31 - 1
samples)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_03847_gb300", "csrc")


def test_every_domain_above_N_is_walked(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    sizes = [1, 2, 3, 4, 5, 15, 16, 17, 65536, 65537, 2**30 - 1, 2**30, 2**30 + 1, 2**31 - 1]
    src = tmp_path / "shape.cu"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "lhs_feistel.cuh"\n'
                   "int main(int c, char** v) {\n"
                   "    for (int i = 1; i < c; ++i) {\n"
                   "        const fmc::FeistelShape f = fmc::feistel_shape(atoll(v[i]));\n"
                   '        printf("%d %u %d\\n", f.h, f.mask, (int)f.walk);\n'
                   "    }\n}\n")
    exe = tmp_path / "shape"
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)] + [str(n) for n in sizes], check=True, capture_output=True, text=True).stdout
    for n, line in zip(sizes, out.splitlines(), strict=True):
        h, mask, walk = (int(x) for x in line.split())
        assert 4**h >= n and (h == 1 or 4 ** (h - 1) < n)
        assert mask == 2**h - 1
        assert bool(walk) == (4**h > n), n

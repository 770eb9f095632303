"""Which eigensolver a list of small matrices takes (csrc/blockops.h), compiled
for the host: the cluster per matrix for few wide ones, the block per matrix
for many, by the measured side of each (milliseconds, block / cluster)."""
import os
import shutil
import subprocess

import pytest

from paper_0902_3185_gb300 import build

# (size, count, measured with one block, with one cluster per matrix)
MEASURED = [(33, 24, 1.60, 1.70), (33, 150, 2.16, 4.93), (33, 600, 5.31, 15.4), (40, 1, 1.86, 1.59),
            (40, 150, 2.70, 5.71), (48, 1, 2.71, 2.01), (48, 24, 2.90, 2.36), (48, 150, 3.54, 7.24),
            (64, 1, 5.19, 2.67), (64, 24, 5.48, 3.22), (64, 60, 5.62, 4.20),
            (64, 80, 5.70, 7.00), (64, 150, 6.03, 10.5), (64, 600, 19.6, 33.9),
            (65, 1, 5.53, 2.97), (65, 24, 5.97, 4.61), (65, 40, 6.11, 7.28), (65, 150, 6.60, 20.5), (65, 600, 25.0, 75.7),
            (80, 1, 9.33, 3.75), (80, 24, 10.1, 5.95), (80, 60, 10.2, 11.4), (80, 150, 10.6, 26.9), (80, 600, 35.7, 101.3),
            (110, 1, 23.6, 5.86), (110, 24, 24.2, 10.1), (110, 150, 24.8, 45.5)]

# (size, count, measured with clusters of 16 blocks, of 8)
CLUSTERS = [(111, 10, 7.33, 7.62), (111, 50, 27.3, 12.3), (111, 100, 33.0, 23.3), (130, 1, 8.74, 11.7),
            (130, 10, 11.2, 11.9), (130, 24, 16.9, 15.2), (130, 50, 28.3, 21.2), (130, 100, 51.0, 40.4),
            (160, 10, 14.9, 16.2), (160, 24, 21.8, 21.5), (160, 50, 38.6, 30.1), (160, 150, 102.6, 89.1),
            (200, 1, 19.6, 28.9), (200, 10, 25.8, 29.5), (200, 24, 52.3, 42.1), (200, 50, 88.4, 83.3),
            (200, 100, 159.6, 125.1), (250, 1, 28.6, 45.6), (250, 24, 75.1, 91.0), (250, 50, 148.4, 179.8),
            (300, 24, 128.4, 151.1)]


def test_the_faster_side_is_taken(tmp_path):
    cxx = shutil.which("g++")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    if not cxx or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    lists = ["{%d, %d}" % m[:2] for m in MEASURED]
    (tmp_path / "route.cpp").write_text(
        '#include "blockops.h"\n#include <cstdio>\n'
        "int main() {\n"
        "  const int c[][2] = {" + ", ".join(lists) + "};\n"
        '  for (auto& x : c) printf("%d ", (int)dmrg::eig_clusters_pay(std::vector<int>(x[1], x[0])));\n'
        "  std::vector<int> v(400, 9);  // many small ones beside a wide one\n"
        '  v.push_back(36); printf("%d ", (int)dmrg::eig_clusters_pay(v));\n'
        '  printf("%d ", (int)dmrg::eig_clusters_pay({}));\n'
        "  const int w[][2] = {" + ", ".join("{%d, %d}" % m[:2] for m in CLUSTERS) + "};\n"
        '  for (auto& x : w) printf("%d ", dmrg::eig_cluster_blocks(std::vector<int>(x[1], x[0])));\n'
        "}\n")
    exe = str(tmp_path / "route")
    subprocess.run([cxx, "-std=c++17", "-I" + build.CSRC, "-I" + include, str(tmp_path / "route.cpp"), "-o", exe],
                   check=True)
    got = subprocess.run([exe], capture_output=True, text=True, timeout=60).stdout.split()
    assert got[:len(MEASURED) + 2] == [str(int(c < b)) for _, _, b, c in MEASURED] + ["0", "0"]
    assert got[len(MEASURED) + 2:] == ["8" if e < s else "16" for _, _, s, e in CLUSTERS]

"""Clusters that the device cannot place are not launched: the size comes down by halves until one fits."""
import os
import subprocess

import pytest

import paper_2510_25600_b200

CSRC = os.path.join(os.path.dirname(paper_2510_25600_b200.__file__), "csrc")
MAIN = """
#include <cstdio>
#include <cstdlib>
#include "cluster.cuh"
int main(int, char** v) {  // wanted size, largest size that fits
  const int most = atoi(v[2]);
  printf("%d", purekv::cluster_that_fits(atoi(v[1]), [&](int c) { return c <= most ? 16 / c : 0; }));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("fit")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    return str(d / "main")


@pytest.mark.parametrize("want,most,got", [(16, 16, 16), (16, 15, 8), (16, 8, 8), (16, 5, 4), (8, 16, 8), (4, 2, 2), (16, 1, 1), (16, 0, 1), (1, 0, 1)])
def test_largest_size_that_fits(program, want, most, got):
    assert int(subprocess.check_output([program, str(want), str(most)])) == got


@pytest.mark.parametrize("source,launches", [("decode.cu", 1), ("score.cu", 2)])
def test_every_cluster_launch_asks_first(source, launches):
    text = open(os.path.join(CSRC, source)).read()
    assert text.count("cudaLaunchAttributeClusterDimension;") == 1 and text.count("clusters_at_once(") == launches

"""The rules that choose launch shapes, compiled for the host from the library's
header and evaluated over the sizes they are stated for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "ct_internal.cuh"
int main(int argc, char **argv)
{
    long long v[6] = {};
    while (std::scanf("%lld %lld %lld %lld %lld", v, v + 1, v + 2, v + 3, v + 4) == 5)
        std::printf("%d\n", ctgb::adj_cluster_size((int)v[0], v[1], (int)v[2], (int)v[3], (int)v[4]));
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    inc = "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("rules")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-w", "-I", inc, "-I", os.path.join(ROOT, "paper_2605_06336_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", str(d / "main")], check=True)

    def run(rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        out = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout
        return [int(x) for x in out.split()]
    return run


@pytest.mark.parametrize("fixed", [8, 3])
def test_a_tile_gets_the_ctas_asked_for(rules, fixed):
    """Asking for more CTAs never gives fewer; at least as many as asked for where each keeps 8 views, else 2."""
    views = list(range(1, 70)) + [180, 1200]
    for tiles in (1, 9, 64, 169, 4096):
        got = {s: rules([(v, tiles, 152, s, fixed) for v in views]) for s in (1, 2, 4)}
        for i, v in enumerate(views):
            assert got[1][i] <= got[2][i] <= got[4][i] <= 8, (v, tiles)
            assert got[2][i] >= 2 and got[4][i] >= (4 if v >= 32 else 2), (v, tiles)


def test_sizes_whose_cluster_is_known(rules):
    """The cluster sizes that the operator tests of the tiled transpose are meant to reach (FP32)."""
    tiles = lambda N, groups: groups * ((N + 31) // 32) ** 2
    rows = [(130, tiles(65, 1), 152, 1, 8), (40, tiles(65, 1), 152, 1, 8), (60, tiles(65, 1), 152, 1, 8),
            (1100, tiles(65, 1), 152, 1, 8)]
    assert rules(rows) == [8, 4, 6, 8]

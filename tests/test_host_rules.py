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
    long long r, v[6] = {};
    while (std::scanf("%lld %lld %lld %lld %lld %lld %lld", &r, v, v + 1, v + 2, v + 3, v + 4, v + 5) == 7)
        std::printf("%llu\n", r == 0   ? (unsigned long long)ctgb::adj_cluster_size((int)v[0], v[1], (int)v[2], (int)v[3], (int)v[4], (int)v[5])
                              : r == 1 ? (unsigned long long)ctgb::adj_group_width((int)v[0], (int)v[1], v[2], (int)v[3], (int)v[4])
                                       : ctgb::order_key((int)v[0], (int)v[1], v[2], (int)v[3]));
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

    def run(rows, rule=0):
        text = "\n".join(" ".join(map(str, (rule, *r, *[0] * (6 - len(r))))) for r in rows)
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


def test_few_views_take_one_cta_and_narrow_groups(rules):
    """Few views: no cluster unless one is asked for, and groups that leave a CTA for every SM; never wider than kb."""
    assert rules([(8, 16, 152, 1, 8, 20), (8, 16, 152, 2, 8, 20), (8, 16, 152, 4, 8, 20), (22, 16, 152, 1, 8, 20)]) == [1, 2, 2, 2]
    tiles = lambda N: ((N + 31) // 32) ** 2
    rows = [(8, 8, tiles(96), 8, 152), (8, 8, tiles(256), 8, 152), (4, 5, tiles(256), 22, 152), (8, 8, tiles(256), 45, 152),
            (8, 8, tiles(256), 180, 152), (2, 2, tiles(2048), 120, 152)]
    assert rules(rows, rule=1) == [1, 4, 1, 4, 8, 2]
    rows = [(kb, K, t, v, 152) for kb, K in ((1, 1), (2, 3), (4, 7), (8, 9)) for t in (9, 64, 4096) for v in (1, 30, 1200)]
    assert all(1 <= w <= r[0] for w, r in zip(rules(rows, rule=1), rows))


def test_view_keys_sort_by_frame_axis_slope_and_index(rules):
    """Slopes up to and including the diagonals', whose fixed-point value is 2^47 itself."""
    h = 1 << 47
    rows = [(f, mode, q, i) for f in (0, 1, 4095) for mode in (0, 1)
            for q, i in ((-h, 5), (-h, 9), (-h + 512, 2), (-1, 4095), (0, 7), (h - 1024, 3), (h, 0), (h, 4))]
    keys = rules(rows, rule=2)
    assert keys == sorted(keys) and len(set(keys)) == len(keys)
    for (f, mode, _, i), k in zip(rows, keys):
        assert (k >> 52, k >> 51 & 1, k & 0xfff) == (f, mode, i)

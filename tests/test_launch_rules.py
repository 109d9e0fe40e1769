"""The rules that choose launch shapes are arithmetic on sizes and on what the device holds: compiled by themselves here,
so that devices are asked about that no test could bring up (one that cannot place a cluster of sixteen CTAs)."""
import ctypes
import os
import subprocess

import pytest

from paper_2410_12876_b200 import build

SHIM = """#include "launch_rules.cuh"
extern "C" int decode_ctas(int D, int slabs, int query_slabs, int G, int cap, int at_once, int apart) {
  return ag::decode_ctas(D, slabs, query_slabs, G, cap, at_once, apart);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, str(d / "shim.cpp"), "-o", str(d / "rules.so")], check=True)
    return ctypes.CDLL(os.fspath(d / "rules.so"))


SLABS = [(D, s, G) for D in (64, 128) for G in (1, 4, 8, 16) for s in (1, 2, 4, 7, 8, 9, 15, 16, 17, 64)]


@pytest.mark.parametrize("D,slabs,G", SLABS)
def test_clusters_of_sixteen_only_where_the_device_places_them(rules, D, slabs, G):
    for cap in (100, 600, 1100, 2100, 4200, 8192, 8300, 20000):
        for at_once, apart in ((0, 0), (1, 0), (4, 4), (14, 7), (21, 7), (31, 7)):
            ctas = rules.decode_ctas(D, slabs, slabs * G, G, cap, at_once, apart)
            assert ctas in (0, 1, 2, 4, 8, 16)
            assert ctas != 16 or slabs <= at_once
            # whether the split form is taken does not depend on it: a step's append is routed before the device is asked
            assert (ctas == 0) == (rules.decode_ctas(D, slabs, slabs * G, G, cap, 0, 0) == 0)


@pytest.mark.parametrize("D,slabs,G,cap,at_once,want", [
    # clusters that share SMs lost 80 - 100 % (16 heads, two CTAs per SM: 14 at once) and 20 - 35 % (8 heads)
    (128, 16, 16, 2200, 14, False), (128, 16, 16, 16000, 14, False), (128, 14, 16, 2200, 14, False), (64, 16, 16, 2200, 21, False),
    (128, 8, 8, 2200, 21, False), (128, 8, 8, 16000, 21, False), (64, 9, 8, 4400, 31, False),
    # few heads: 10 - 20 % lost in short caches, which a capacity of a few thousand rows does not outweigh
    (128, 8, 4, 2200, 21, False), (128, 16, 1, 4400, 21, False), (128, 8, 4, 8300, 21, True), (64, 16, 1, 8300, 31, True),
    # one cluster per GPC: never more than 3 % behind, up to 30 % ahead
    (128, 7, 8, 2200, 21, True), (128, 4, 16, 600, 14, True), (64, 2, 1, 2200, 31, True), (128, 2, 4, 2000, 21, False),
])
def test_clusters_of_sixteen_by_room_and_rows(rules, D, slabs, G, cap, at_once, want):
    # (query_slabs: few enough that the split form is not asked for)
    assert (rules.decode_ctas(D, slabs, 64, G, cap, at_once, 7) == 16) == want

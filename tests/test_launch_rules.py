"""The rules that choose launch shapes are arithmetic on sizes and on what the device holds: compiled by themselves here,
so that devices are asked about that no test could bring up (one that cannot place a cluster of sixteen CTAs)."""
import ctypes
import os
import subprocess

import pytest

from paper_2410_12876_b200 import build

SHIM = """#include "launch_rules.cuh"
extern "C" int decode_ctas(int D, int slabs, int query_slabs, int G, int cap, int wide, int apart, int ten) {
  return ag::decode_ctas(D, slabs, query_slabs, G, cap, ag::DecodePlaces{wide, apart, ten});
}
extern "C" int gate_linear_split(int tiles, int kb, int heads, int c1, int c2, int c4, int c8) {
  return ag::gate_linear_split(tiles, kb, heads, ag::GateLinearPlaces{{c1, c2, c4, c8}});
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
def test_larger_clusters_only_where_the_device_places_them(rules, D, slabs, G):
    for cap in (100, 600, 1100, 2100, 4200, 8192, 8300, 20000):
        for wide, apart, ten in ((0, 0, 0), (0, 0, 2), (1, 0, 0), (4, 4, 6), (14, 7, 0), (21, 7, 9), (31, 7, 9)):
            ctas = rules.decode_ctas(D, slabs, slabs * G, G, cap, wide, apart, ten)
            assert ctas in (0, 1, 2, 4, 8, 10, 16)
            assert ctas != 16 or slabs <= wide
            assert ctas != 10 or slabs <= ten and G <= 4
            # whether the split form is taken does not depend on it: a step's append is routed before the device is asked
            assert (ctas == 0) == (rules.decode_ctas(D, slabs, slabs * G, G, cap, 0, 0, 0) == 0)


@pytest.mark.parametrize("D,slabs,G,cap,wide,want", [
    # clusters that share SMs lost 80 - 100 % (16 heads, two CTAs per SM: 14 at once) and 20 - 35 % (8 heads)
    (128, 16, 16, 2200, 14, 8), (128, 16, 16, 16000, 14, 8), (128, 14, 16, 2200, 14, 8), (64, 16, 16, 2200, 21, 8),
    (128, 8, 8, 2200, 21, 8), (128, 8, 8, 16000, 21, 8), (64, 9, 8, 4400, 31, 8), (64, 9, 4, 4400, 31, 10), (128, 8, 16, 4400, 14, 8), (128, 10, 4, 4400, 21, 8),
    # few heads: 10 - 20 % lost in short caches, which a capacity of a few thousand rows does not outweigh
    (128, 8, 4, 2200, 21, 10), (128, 16, 1, 4400, 21, 8), (128, 8, 4, 8300, 21, 16), (64, 16, 1, 8300, 31, 16), (128, 8, 4, 2000, 21, 8),
    # an SM to each CTA: never more than 3 % behind, up to 30 % ahead
    (128, 7, 8, 2200, 21, 16), (128, 4, 16, 600, 14, 16), (64, 2, 1, 2200, 31, 16), (128, 2, 4, 2000, 21, 8),
])
def test_larger_clusters_by_room_and_rows(rules, D, slabs, G, cap, wide, want):
    # (query_slabs: few enough that the split form is not asked for)
    assert rules.decode_ctas(D, slabs, 64, G, cap, wide, 7, 9) == want


B200 = (444, 222, 104, 48)


@pytest.mark.parametrize("tiles,kb,heads,want", [
    (1, 64, 32, 8), (48, 64, 32, 8), (49, 64, 32, 4), (55, 64, 32, 4), (104, 64, 32, 4), (105, 64, 32, 2), (111, 64, 32, 2), (222, 64, 32, 2),
    (250, 64, 32, 1), (480, 64, 32, 2),                  # a second wave of single CTAs is longer than a third of pairs
    (250, 64, 8, (4, 8)), (400, 8, 8, 2),                # 8 heads: not one CTA to a tile
    (5, 1, 8, 1), (5, 2, 8, 2),                          # no more CTAs than k-blocks
])
def test_ctas_of_a_local_gate_tile(rules, tiles, kb, heads, want):
    got = rules.gate_linear_split(tiles, kb, heads, *B200)
    assert got in (want if isinstance(want, tuple) else (want,))


def test_local_gate_clusters_only_where_the_device_places_them(rules):
    for tiles in (1, 7, 50, 1000, 65535):
        for kb in (1, 3, 33, 64, 4096):
            assert rules.gate_linear_split(tiles, kb, 32, *B200) <= kb
            assert rules.gate_linear_split(tiles, kb, 32, 12, 5, 0, 0) <= 2
            assert rules.gate_linear_split(tiles, kb, 8, 0, 0, 0, 0) == 1

"""The rules that choose launch shapes are arithmetic on sizes and on what the device holds: compiled by themselves here,
so that devices are asked about that no test could bring up (one that cannot place a cluster of sixteen CTAs)."""
import ctypes
import os
import subprocess

import pytest

from paper_2410_12876_b200 import build

SHIM = """#include "launch_rules.cuh"
extern "C" int decode_ctas(int D, int slabs, int query_slabs, int G, int cap, int at_once) {
  return ag::decode_ctas(D, slabs, query_slabs, G, cap, at_once);
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
        for at_once in (0, 1, 7, 14, 21):
            ctas = rules.decode_ctas(D, slabs, slabs * G, G, cap, at_once)
            assert ctas in (0, 1, 2, 4, 8, 16)
            assert ctas != 16 or slabs <= at_once
            # whether the split form is taken does not depend on it: a step's append is routed before the device is asked
            assert (ctas == 0) == (rules.decode_ctas(D, slabs, slabs * G, G, cap, 0) == 0)

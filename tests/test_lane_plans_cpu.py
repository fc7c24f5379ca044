"""The register transforms' lane plans and the launch rules that go by them, compiled for the CPU."""
import ctypes
import os
import subprocess

import pytest

from helpers import ROOT

SRC = os.path.join(ROOT, "tests", "emu", "lane_driver.cpp")
LIB = os.path.join(ROOT, "tests", "emu", "_build", "libpme_lanes.so")


@pytest.fixture(scope="module")
def lanes():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    tmp = LIB + f".{os.getpid()}.tmp"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-pthread",
                           "-I/usr/local/cuda/include", "-x", "c++", SRC, "-o", tmp])
    os.replace(tmp, LIB)
    return ctypes.CDLL(LIB)


@pytest.fixture(scope="module")
def edges(lanes):
    out = (ctypes.c_int * 64)()
    return out[:lanes.lane_edges(out)]


def test_slab_threads_of_groups(lanes, edges):
    """A group with more slabs than SMs runs slabs of up to 10000 points on 512 threads, so that several CTAs share an
    SM; larger ones, fewer slabs, and every slab of a single system run on as many whole warps as both passes can use in
    one round (512 to 1024)."""
    for K2 in edges:
        for K3 in edges:
            one = lanes.lane_slab_threads(K2, K3, 0)
            assert 512 <= one <= 1024 and one % 32 == 0
            assert lanes.lane_slab_threads(K2, K3, 153) == (512 if K2 * K3 <= 10000 else one), (K2, K3)
            assert lanes.lane_slab_threads(K2, K3, 152) == one
    assert lanes.lane_slab_threads(80, 80, 0) > 512 and lanes.lane_slab_threads(108, 108, 1000) > 512

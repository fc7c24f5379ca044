"""The register transforms' lane plans and the launch rules of the stages, compiled for the CPU."""
import ctypes
import math
import os
import subprocess

import numpy as np
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


def test_lane_transforms(lanes):
    """Every plan's transforms, by a warp of 32 threads that exchange values as shuffles do: forward and inverse
    (unnormalised) against a 64-bit FFT, and the adjoint of the forward transform gives N times the input. Each output
    is a sum of N terms by log2 N levels of a few FP32 roundings: a relative error of 1e-6 in the 2-norm."""
    for c in range(lanes.lane_plans()):
        le = (ctypes.c_int * 2)()
        lanes.lane_plan(c, le)
        L, E = le
        N, T = L * E, 32 // L
        rng = np.random.default_rng(c)
        x = (rng.normal(size=(T, N)) + 1j * rng.normal(size=(T, N))).astype(np.complex64)
        out = [np.full((T, N), np.nan, np.complex64) for _ in range(3)]
        ptr = [a.ctypes.data_as(ctypes.POINTER(ctypes.c_float)) for a in (x, *out)]
        lanes.lane_run(c, *ptr)
        x64 = x.astype(np.complex128)
        for got, ref in zip(out, (np.fft.fft(x64), np.fft.ifft(x64) * N, x64 * N)):
            assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref), (L, E)


def test_stage_shared_memory(lanes, edges):
    """The slab buffers with their padded rows and the twiddles behind them, and the influence stage's sums, fit the
    shared memory that the stages are launched with, for every mesh."""
    used, given = (ctypes.c_longlong * 3)(), (ctypes.c_longlong * 3)()
    for K2 in edges:
        for K3 in edges:
            for K1 in edges if K2 == K3 == 8 else (8,):
                lanes.lane_smem(K1, K2, K3, used, given)
                assert all(u <= g for u, g in zip(used, given)), (K1, K2, K3, list(used), list(given))


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


@pytest.mark.parametrize("K", [(80, 80, 96), (90, 96, 100), (96, 96, 96), (72, 80, 100), (128, 128, 128), (64, 64, 64)],
                         ids=lambda K: "x".join(map(str, K)))
def test_default_tiles_hold_their_atoms(lanes, K):
    """Atoms beyond a tile's bucket take a path many times slower. At every density and order, buckets of the default
    16^3 tiles hold at least what the eight 8^3 tiles in each would, and eight times twice the mean over 8^3 tiles
    (ragged ones among them)."""
    Kc = (ctypes.c_int * 3)(*K)
    N = K[0] * K[1] * K[2]
    for p in (4, 5, 6, 8):
        edges = set()
        for density in (0.01, 0.03, 0.06, 0.1, 0.15, 0.2, 0.25, 0.3, 0.4, 0.6, 0.85, 0.95):
            n = int(density * N)
            edge = lanes.lane_tile_edge(ctypes.c_longlong(n), Kc, p)
            cap = lanes.lane_bucket_capacity(ctypes.c_longlong(n), Kc, edge)
            edges.add(edge)
            if edge == 16:
                assert cap >= 8 * lanes.lane_bucket_capacity(ctypes.c_longlong(n), Kc, 8)
                assert cap >= 16 * n / math.prod((k + 7) // 8 for k in K)
        assert (16 in edges) == (K != (64, 64, 64)) or p == 4

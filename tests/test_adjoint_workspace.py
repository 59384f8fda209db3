"""Workspace of the drag gradient: what lbm_adj_workspace_size asks for stays
within a state every ceil(sqrt(T)) steps, one segment's states, four more states
and 81 bytes a node (with 48 a link, 24 a link node and alignment), whatever T;
the larger size that keeps every step is the caller's choice."""
import ctypes as C
import math

import numpy as np
import pytest

import paper_2206_11634_gb300 as pkg
from paper_2206_11634_gb300 import build as build_mod


@pytest.fixture(scope="module")
def lib():
    build_mod.build()
    return pkg.load_library()


def sizes(lib, n, T):
    cfg = pkg.make_config(n, n, n, periodic=(1, 1, 1), tau=0.8)
    p = pkg.make_particle([[0, 0, 0]], [9.0], (n / 2 - 0.2, n / 2 + 0.1, n / 2), fixed=1, mass=1.0, inertia=np.eye(3))
    a, least, keep = C.c_size_t(), C.c_size_t(), C.c_size_t()
    assert lib.lbm_adj_workspace_size(C.byref(cfg), C.byref(p), T, 1, C.byref(a)) == 0
    assert lib.lbm_adj_workspace_sizes(C.byref(cfg), C.byref(p), T, 1, C.byref(least), C.byref(keep)) == 0
    assert a.value == least.value <= keep.value
    return least.value, keep.value


@pytest.mark.parametrize("n,T", [(32, 1), (32, 2), (32, 23), (32, 80), (32, 14000), (64, 500), (96, 500)])
def test_workspace_stays_within_checkpoints(lib, n, T):
    least, keep = sizes(lib, n, T)
    N, K = n ** 3, max(1, math.ceil(math.sqrt(T)))
    links = 1500  # of a sphere of radius 3: some 110 nodes, 9 directions, with room
    bound = 76 * N * (4 + -(-T // K) + max(1, K - 1)) + 81 * N + 48 * links + 24 * links + 32 * 256 + 36 * links * K
    assert least <= bound
    assert keep >= 16 * N * T


def test_sizes_reject_null(lib):
    cfg = pkg.make_config(16, 16, 16, periodic=(1, 1, 1), tau=0.8)
    p = pkg.make_particle([[0, 0, 0]], [4.0], (8, 8, 8), fixed=1, mass=1.0, inertia=np.eye(3))
    a = C.c_size_t()
    assert lib.lbm_adj_workspace_sizes(C.byref(cfg), C.byref(p), 4, 1, None, C.byref(a)) == -1
    assert lib.lbm_adj_workspace_sizes(C.byref(cfg), C.byref(p), 4, 1, C.byref(a), None) == -1
    assert lib.lbm_adj_workspace_sizes(C.byref(cfg), C.byref(p), 4, 5, C.byref(a), C.byref(a)) == -1

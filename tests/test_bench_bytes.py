"""The bench's count of what a mock cannot do without: the pencils, rows and
planes that the passes carry, against brute force."""
import math

import numpy as np
import pytest

import bench
from oracle import power as op


@pytest.mark.parametrize("N,k_max", [(16, 0.02), (16, 0.05), (30, 0.1), (32, 1.0)])
def test_reached_pencils(N, k_max):
    L = 1000.0
    n2 = bench.largest_n2(k_max, L)
    kf = 2 * math.pi / L
    assert kf * math.sqrt(n2) < k_max <= kf * math.sqrt(n2 + 1)
    want = {(x, y) for x in range(N // 2) for y in range(-N // 2 + 1, N // 2) for z in range(-N // 2 + 1, N // 2)
            if x * x + y * y + z * z <= n2}
    assert bench.reached_pencils(N, n2) == len(want)


@pytest.mark.parametrize("assign", [2, 3, 4])
def test_occupied_rows(assign):
    g = np.random.default_rng(4)
    cats = [{k: g.uniform(*lim, 40).astype(np.float32) for k, lim in
             (("x", (200, 800)), ("y", (300, 500)), ("z", (550, 700)))} | {"nbar": np.full(40, 1e-4, np.float32)}
            for _ in range(2)]
    geom = dict(L=1000.0, N=40, assign=assign, origin=(0.0, 0.0, 0.0), observer=(0.0, 0.0, 0.0))
    F = op.fkp_grids(*cats, geom, with_w2=False)[0]
    hit = (F != 0).any(axis=2)  # [z][y][x]
    assert bench.occupied_rows(cats, geom) == (hit.sum(), hit.any(axis=1).sum())


def test_bytes_shrink_with_what_is_carried():
    N = 64
    whole = bench.algorithmic_bytes(N, 9, 1000, N * (N // 2 + 1), N * N, N)
    assert whole["zpass"] == 9 * 8 * N * N * (N // 2 + 1) and whole["xpass"] == 4 * N ** 3
    part = bench.algorithmic_bytes(N, 9, 1000, N * (N // 2 + 1) // 3, N * N // 2, N // 2)
    assert part["zpass"] == whole["zpass"] // 6 and part["xpass"] == whole["xpass"] // 2

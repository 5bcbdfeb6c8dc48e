"""The batched path's choices by a set's points, each against the oracle: the
scaled inner region at every coordinate size, sets around the star polygon's
sizes at every density, and small sets of few and of many vertices."""
import math

import numpy as np
import pytest

import oracle
from synth import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(lib, sets):
    off = np.zeros(len(sets) + 1, np.int64)
    off[1:] = np.cumsum([s.shape[0] for s in sets])
    got = lib.hull_batched(torch.from_numpy(np.concatenate(sets)).cuda(), off)
    for i, s in enumerate(sets):
        np.testing.assert_array_equal(got[i].cpu().numpy(), oracle.hull(s), err_msg=str(i))


@pytest.mark.parametrize("bits", [1, 2, 4, 6, 9, 13, 18, 22, 24])
def test_coordinate_sizes(lib, bits):
    """Grids, boxes at the far corner and thin boxes: many points on the region's
    bounds, where the scaled keys round."""
    rng = np.random.default_rng(bits)
    k, top = 1 << bits, (1 << 24) - 1
    grid = rng.integers(0, k, (9001, 2))
    thin = np.stack([rng.integers(0, k, 5000), rng.integers(0, min(k, 3), 5000)], 1)
    disk = rng.integers(0, k, (40_000, 2))
    disk = disk[((disk - k / 2.0) ** 2).sum(1) <= k * k / 4.0 + 1]
    sets = [grid, top - grid, thin, top - thin, thin[:, ::-1], disk, top - disk, grid + [top + 1 - k, 0]]
    _check(lib, [np.ascontiguousarray(s, dtype=np.float32) for s in sets])


def _triangle(n, seed):
    u = np.random.default_rng(seed).random((n, 2))
    u = np.where(u.sum(1, keepdims=True) > 1, 1 - u, u)
    return np.rint(np.stack([u[:, 0], 0.7 * u[:, 1] + 0.2 * u[:, 0]], 1) * ((1 << 24) - 1)).astype(np.float32)


def _disk(n, seed):
    rng = np.random.default_rng(seed)
    a, r = rng.uniform(0, 2 * math.pi, n), 8.0e6 * np.sqrt(rng.random(n))
    return np.rint(np.stack([np.cos(a) * r, np.sin(a) * r], 1) + (1 << 23)).astype(np.float32)


@pytest.mark.parametrize("n", [257, 9000, 16_383, 16_384, 20_001, 32_767, 32_768])
def test_densities(lib, n):
    half = np.concatenate([W.ring(n // 3, n), W.normal(n - n // 3, n)])
    _check(lib, [W.uniform(n, 1), W.normal(n, 2), W.ring(n, 3), W.distorted(n, 4), _triangle(n, 5), _disk(n, 6),
                 half[np.random.default_rng(n).permutation(n)], np.repeat(W.ring(n // 4, 7), 4, axis=0)])


@pytest.mark.parametrize("n", [240, 256, 300, 500, 1000, 2030, 2060])
def test_small_sets_by_vertices(lib, n):
    """At and beyond the vertex capacity (256) and the record capacity (2048) of
    the small sets' quickhull; convex position; copies of one vertex."""
    k = np.arange(n, dtype=np.int64)
    arc = np.stack([k * 300, np.concatenate([[0], np.cumsum(k[:-1] - n // 2)])], 1)
    arc[:, 1] -= arc[:, 1].min()
    few = np.concatenate([arc[:250], arc[:max(1, n - 250)]]) if n > 250 else arc
    copies = np.concatenate([np.repeat([[10, 10]], n - n // 3, axis=0), W.normal(n // 3, 2).astype(np.int64) // 2 + 4000])
    order = np.random.default_rng(n).permutation
    _check(lib, [W.ring(n, n), W.distorted(n, n), np.float32(arc[order(n)]), np.float32(few[order(len(few))]),
                 np.float32(copies[order(n)]), W.uniform(n, n)] * 3)

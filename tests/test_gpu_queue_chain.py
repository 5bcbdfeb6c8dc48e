"""Hulls of dense sets, queue by queue (the block sort by u and the elimination
rounds), batched and single: bit-exact with the oracle at the edges of the
kernels' shapes, and on inputs that take their other branches (crowded buckets,
long chains that hide each other, duplicates, a queue over the largest shape,
tiles of u ranges, a tile over its block's capacity)."""
import numpy as np
import pytest

import oracle
from synth import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _arc(m, step=1, y0=5):
    """m lattice points in strictly convex position: a parabola arc."""
    x = np.arange(m, dtype=np.int64)
    y = np.cumsum(np.concatenate([[0], x[:-1] - m // 2]))
    return np.stack([x * step, y - y.min() + y0], 1)


def _shuffled(parts, seed):
    pts = np.concatenate([np.asarray(p, np.int64) for p in parts])
    return pts[np.random.default_rng(seed).permutation(pts.shape[0])].astype(np.float32)


def _two_arcs(m):
    """Two deep arcs side by side: each hides half of the other's chain."""
    a = _arc(m)
    b = a.copy()
    b[:, 0] += 3 * m
    return _shuffled([a, b, a[::3], b[::2]], m)


def _crowded(m):
    """A dense arc in a small part of the queues' range, and a far corner."""
    return _shuffled([_arc(m), _arc(m)[::2], [[(1 << 24) - 1, 1 << 23], [1 << 23, (1 << 24) - 1]]], m)


def _columns(m):
    """Many points of equal u in every frame: a filled diamond's rim, repeated."""
    k = np.arange(m, dtype=np.int64)
    rim = np.concatenate([np.stack([k, m - k], 1), np.stack([k, m + k], 1), np.stack([m + k, k], 1),
                          np.stack([m + k, 2 * m - k], 1)])
    return _shuffled([rim, rim, rim + [0, 1]], m)


CASES = {
    "rings at the small shape's edges": lambda: [W.ring(n, n) for n in (257, 1000, 4 * 2500, 4 * 2560, 16383, 16384)],
    "rings around the largest shape": lambda: [W.ring(n, n) for n in (15000, 16000, 40_000, 300_000)],
    "a queue over the largest shape": lambda: [_shuffled([_arc(4095), _arc(4095)[::-1]] * 3, 1), W.normal(3000, 2),
                                               _shuffled([_arc(5000)] * 9, 3)],
    "convex position": lambda: [_shuffled([_arc(m)], m) for m in (300, 1025, 4001, 5500)],
    "arcs that hide each other": lambda: [_two_arcs(m) for m in (200, 700, 2000)],
    "crowded buckets": lambda: [_crowded(m) for m in (400, 1500, 3900)],
    "equal u and duplicates": lambda: [_columns(m) for m in (90, 1000, 2800)],
}


@pytest.mark.parametrize("name", list(CASES))
def test_dense_sets_queue_by_queue(lib, name):
    sets = CASES[name]()
    assert all(s.min() >= 0 and s.max() < (1 << 24) for s in sets)
    off = np.zeros(len(sets) + 1, np.int64)
    off[1:] = np.cumsum([s.shape[0] for s in sets])
    pts = torch.from_numpy(np.concatenate(sets)).cuda()
    got = lib.hull_batched(pts, off)
    for i, s in enumerate(sets):
        np.testing.assert_array_equal(got[i].cpu().numpy(), oracle.hull(s), err_msg=str(i))


SINGLE = dict(CASES)
SINGLE.update({
    "tiles": lambda: [W.ring(8_000_001, 4), W.distorted(20_000_003, 5)],
    "the dense pass's smallest inputs": lambda: [W.ring(n, n) for n in (65_535, 65_537, 66_000, 70_001, 131_073)],
    "tiles without a polygon": lambda: [_shuffled([_arc(4095)] * 12, 6), _shuffled([_columns(4000)] * 2, 7)],
    "a tile in pieces": lambda: [_shuffled([_arc(100)] * 4000, 8)],
})


@pytest.mark.parametrize("name", list(SINGLE))
def test_single_hull_queue_by_queue(lib, name):
    for i, s in enumerate(SINGLE[name]()):
        pts = torch.from_numpy(s).cuda()
        want = oracle.hull(s)
        out_idx = torch.empty(s.shape[0], dtype=torch.int32, device="cuda")
        out_n = torch.empty(1, dtype=torch.int64, device="cuda")
        for _ in range(3):   # launched, captured, replayed
            got = lib.hull(pts, out_idx=out_idx, out_n=out_n)
            np.testing.assert_array_equal(got.cpu().numpy(), want, err_msg=str(i))


@pytest.mark.parametrize("bad", [-1.0, 0.5, float(1 << 24), float("nan"), float("inf")])
@pytest.mark.parametrize("at", [0, 150_000, 200_001])
def test_dense_data_with_a_bad_coordinate(lib, bad, at):
    pts = W.ring(200_002, 9)
    pts[at, at & 1] = bad
    with pytest.raises(lib.CHError) as e:
        lib.hull(torch.from_numpy(pts).cuda())
    assert e.value.status == lib.CH_ERANGE
    good = W.ring(200_002, 10)   # the star pass's bins are clear again
    np.testing.assert_array_equal(lib.hull(torch.from_numpy(good).cuda()).cpu().numpy(), oracle.hull(good))

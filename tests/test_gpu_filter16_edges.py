"""ch_filter16 where its float edge functions leave the label open: copies of the
polygon's vertices, points on its edges, edges of a few units, no area; a point
per thread and by tiles."""
import numpy as np
import pytest

from oracle import filter16_ref as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BY_TILES = (3 << 20) + 700


def _points(kind, n):
    rng = np.random.default_rng(n)
    top = (1 << 24) - 1
    if kind == "corner":       # edges of 1 to 50 units beside edges of 2^24
        p = rng.integers(0, top + 1, (n, 2))
        p[:40] = top - rng.integers(0, 50, (40, 2))
        p = np.where(p.sum(1, keepdims=True) < top, top - p, p)
    elif kind == "copies":     # of every extreme of a disk
        a, r = rng.uniform(0, 2 * np.pi, n), 4e6 * np.sqrt(rng.random(n))
        p = np.rint(np.stack([np.cos(a) * r, np.sin(a) * r], 1) + (1 << 23)).astype(np.int64)
        ext = G.extremes16(p.astype(np.float32))
        p[rng.integers(0, n, n // 2)] = p[ext[rng.integers(0, 16, n // 2)]]
    elif kind == "edges":      # a lattice octagon's boundary, filled
        k = rng.integers(0, 3001, n)
        side = rng.integers(0, 9, n)
        p = rng.integers(3000, 7000, (n, 2))
        for s, (x, y, dx, dy) in enumerate([(0, 3000, 0, 1), (0, 6000, 1, 1), (3000, 9000, 1, 0), (6000, 9000, 1, -1),
                                            (9000, 6000, 0, -1), (9000, 3000, -1, -1), (6000, 0, -1, 0), (3000, 0, -1, 1)]):
            m = side == s
            p[m] = np.stack([x + dx * k[m], y + dy * k[m]], 1)
    else:                      # collinear
        k = rng.integers(0, 1 << 22, n)
        p = np.stack([3 * k, k + 5], 1)
    return p.astype(np.float32)


@pytest.mark.parametrize("kind", ["corner", "copies", "edges", "line"])
@pytest.mark.parametrize("n", [3001, BY_TILES])
def test_open_labels(lib, kind, n):
    pts = _points(kind, n)
    ext, lab, cnt = lib.filter16_labels(torch.from_numpy(pts).cuda())
    want = G.labels16(pts)
    np.testing.assert_array_equal(ext.cpu().numpy(), G.extremes16(pts))
    np.testing.assert_array_equal(lab.cpu().numpy(), want)
    np.testing.assert_array_equal(cnt.cpu().numpy(), [(want == r).sum() for r in range(1, 5)])

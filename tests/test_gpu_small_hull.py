"""ch_hull on inputs that one block turns into records: the sizes around its
limit and its smallest ones, sparse and dense data, misaligned points and a
bad coordinate, against the oracle."""
import numpy as np
import pytest

import oracle
from synth import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 31, 513, 1000, 4097, 8191, 8192, 8193])
@pytest.mark.parametrize("kind", ["uniform", "normal", "ring"])
@pytest.mark.parametrize("shift", [0, 1])
def test_small_hull(lib, n, kind, shift):
    pts = W.make(kind, n, 17 + n)
    if n > 100:
        pts[n // 2:n // 2 + 20] = pts[:20]   # equal points: the lowest index
    buf = torch.zeros((n + shift, 2), dtype=torch.float32, device="cuda")
    buf[shift:] = torch.from_numpy(pts).cuda()
    np.testing.assert_array_equal(lib.hull(buf[shift:]).cpu().numpy(), oracle.hull(pts))


@pytest.mark.parametrize("n", [1, 777, 8192])
def test_small_hull_bad_coordinate(lib, n):
    pts = W.make("uniform", n, 3)
    pts[n - 1, 0] = 0.5
    with pytest.raises(lib.CHError):
        lib.hull(torch.from_numpy(pts).cuda())

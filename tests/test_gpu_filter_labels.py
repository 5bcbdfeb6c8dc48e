"""The label passes at their edges: inputs large enough that one read of the
points labels a region of a sample's octagon at once (ch_filter), data that
sends them back to a second read, and label arrays at every byte offset
(with guard bytes around them).  Bit-exact against the numpy definition."""
import numpy as np
import pytest

from oracle import filter16_ref as G
from oracle import filter_ref as F
from synth import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BIG = (1 << 23) + 12_347      # above the largest input that stays with two reads


def run(ch, fn, next_, pts, shift, off, labels=True):
    n = pts.shape[0]
    buf = torch.zeros((n + shift, 2), dtype=torch.float32, device="cuda")
    buf[shift:] = torch.from_numpy(pts).cuda()
    ext = torch.empty(next_, dtype=torch.int32, device="cuda")
    raw = torch.full((n + 64,), 77, dtype=torch.uint8, device="cuda")
    cnt = torch.empty(4, dtype=torch.int64, device="cuda")
    getattr(ch, fn)(buf[shift:].data_ptr(), n, ext.data_ptr(), raw.data_ptr() + 16 + off if labels else None,
                    cnt.data_ptr(), torch.cuda.current_stream().cuda_stream)
    raw = raw.cpu().numpy()
    lab = raw[16 + off:16 + off + n]
    assert (raw[:16 + off] == 77).all() and (raw[16 + off + n:] == 77).all()
    return ext.cpu().numpy(), lab, cnt.cpu().numpy()


def check(ref, got):
    ext, want = ref
    np.testing.assert_array_equal(got[0], ext)
    np.testing.assert_array_equal(got[1], want)
    np.testing.assert_array_equal(got[2], [(want == r).sum() for r in range(1, 5)])


def cut_corner(n):
    """A square whose lower left corner the octagon of the extremes cuts off:
    two points that no sampled tile holds take its W..S vertices."""
    rng = np.random.default_rng(5)
    pts = rng.integers(8_000_000, 10_000_000, (n, 2))
    pts[5 * 512 + 100] = [6_000_000, 9_800_000]
    pts[5 * 512 + 101] = [9_400_000, 7_999_999]
    return pts.astype(np.float32)


@pytest.mark.parametrize("kind,shift,off", [("uniform", 0, 0), ("normal", 1, 3), ("ring", 1, 0), ("cut", 0, 1)])
def test_one_read(lib, kind, shift, off):
    pts = cut_corner(BIG) if kind == "cut" else W.make(kind, BIG, 3)
    ref = F.extremes(pts), F.labels(pts)
    check(ref, run(lib, "ch_filter", 8, pts, shift, off))
    ext, lab, cnt = run(lib, "ch_filter", 8, pts, shift, off, labels=False)
    np.testing.assert_array_equal(ext, ref[0])
    np.testing.assert_array_equal(cnt, [(ref[1] == r).sum() for r in range(1, 5)])


@pytest.mark.parametrize("bad", [np.nan, 0.5, -1.0, 2.0 ** 24])
def test_one_read_bad_coordinate(lib, bad):
    pts = W.make("normal", BIG, 4)
    pts[BIG // 2, 1] = bad
    assert run(lib, "ch_filter", 8, pts, 0, 0)[2].tolist() == [lib.CH_ERANGE] * 4


@pytest.mark.parametrize("fn", ["ch_filter", "ch_filter_manhattan"])
@pytest.mark.parametrize("n", [1, 511, 513, 70_001, (1 << 21) + 1, (1 << 21) + 515])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("off", [0, 1, 2, 3])
def test_label_offsets(lib, fn, n, shift, off):
    pts = W.make("ring" if n & 2 else "uniform", n, n)
    check((F.extremes(pts), F.labels(pts)), run(lib, fn, 8, pts, shift, off))


@pytest.mark.parametrize("n", [1, 2, 511, 513, 70_001, (1 << 21) + 1, (1 << 21) + 515])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("off", [0, 1, 2, 3])
def test_label_offsets16(lib, n, shift, off):
    pts = W.make("ring" if n & 2 else "uniform", n, n)
    pts[n // 2:] = pts[:n - n // 2]      # ties: the lowest index wins, the head point among them
    check((G.extremes16(pts), G.labels16(pts)), run(lib, "ch_filter16", 16, pts, shift, off))

"""The single hull's ways through many survivors (queues.cu, hull.cu), each by
the counters that name it and bit-exact with the oracle: circles without a
width, whose queues' tile chains fit one block or are joined in rounds, a tile
whose own chain goes to the sort, and records crowded in one range of u."""
import math
import time

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

QUEUES_OR_TILES, SORT = 1, 2   # ch_hull_counters' stage


def _circle(n, seed):
    """n points of a circle, rounded: a queue's chain has about 10,400
    vertices at 1e6 points, 13,700 at 4e6 (the oracle's)."""
    a = np.random.default_rng(seed).uniform(0.0, 2.0 * math.pi, n)
    r = float(1 << 23)
    pts = np.stack([np.cos(a), np.sin(a)], 1) * r + r
    return np.clip(np.rint(pts), 0, (1 << 24) - 1).astype(np.float32)


def _calls(lib, pts, calls):
    """Results and counters of calls on the same buffers (launched, captured,
    replayed); out_idx is cleared in between."""
    d = torch.from_numpy(pts).cuda()
    out_idx = torch.empty(pts.shape[0], dtype=torch.int32, device="cuda")
    out_n = torch.empty(1, dtype=torch.int64, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    for _ in range(calls):
        out_idx.fill_(-7)
        got = lib.hull(d, out_idx=out_idx, out_n=out_n)
        yield got.cpu().numpy(), lib.ch_hull_counters(stream)


@pytest.mark.parametrize("n", [1_000_000, 4_000_003, 6_000_001, 20_000_003])
def test_circle(lib, n):
    pts = _circle(n, n)
    want = oracle.hull(pts)
    # past 13,000 tile-chain points in a queue (a block's capacity) all blocks join them in rounds
    assert (want.size > 4 * 13_000) == (n > 1_000_000)
    for got, c in _calls(lib, pts, 100):
        np.testing.assert_array_equal(got, want)
        assert c["stage"] == QUEUES_OR_TILES, c


def _steps(most_u, most_v, ok):
    """Steps (du, dv) between points in the queue frame, one per slope, by slope."""
    low = -most_v if most_v <= most_u else 0
    got = [(du, dv) for du in range(1, most_u + 1) for dv in range(low, most_v + 1)
           if (du + dv) % 2 == 0 and ok(du, dv) and math.gcd((dv + du) // 2, (dv - du) // 2) == 1]
    return np.array(sorted(got, key=lambda s: s[1] / s[0]))


def _long_tile(n):
    """About n points beyond the upper right side of a triangle (its box's centre
    is outside the hull: no star polygon).  In their queue's frame: a convex curve
    of 9834 points, the 5229 falling ones once, the 4605 others, which lie
    in one of the queue's 1024 equal u ranges, many times each."""
    top = (1 << 24) - 1
    fall = _steps(250, 250, lambda u, v: -0.55 * u < v < 0)
    rise = _steps(20, 1600, lambda u, v: v > 0 and u / 19 + v / 1600 <= 1)
    low = int(top * (math.sqrt(2.0) - 1.0))
    start = np.array([int(math.ceil(-top + 512 * (2 * top + 1) / 1024)) + 600, low + 3000])
    start[1] += (start[0] + start[1]) & 1
    up = start + np.concatenate([[[0, 0]], np.cumsum(rise, axis=0)])
    down = start - np.cumsum(fall[::-1], axis=0)

    def xy(p):
        return np.stack([(p[:, 1] + p[:, 0]) // 2, (p[:, 1] - p[:, 0]) // 2], 1)

    corners = [np.array([[0, top], [top, 0], [low - 1000, 1000]])] * 2000
    pts = np.concatenate(corners + [xy(down)] + [xy(up)] * ((n - 12_000) // len(up)))
    pts = (top - pts)[np.random.default_rng(n).permutation(pts.shape[0])]
    assert len(down) < 5900 and len(down) + len(up) > 9800 and pts.min() >= 0
    return pts.astype(np.float32)


@pytest.mark.parametrize("n", [905_000, 4_520_000])   # the extremes first, a sample first
def test_tile_chain_over_its_block(lib, n):
    """A tile of u ranges whose chain so far leaves its block no room for the
    rest of its records; dense data without a star polygon."""
    pts = _long_tile(n)
    want = oracle.hull(pts)
    for got, c in _calls(lib, pts, 10):
        np.testing.assert_array_equal(got, want)
        assert c["stage"] == SORT and c["star_vertices"] == 0 and c["two_pass"] == 1, c


def _far_copies(n, order, cluster=0.0):
    """n points on the GPU: a normal cloud inside eight extremes, and 60 % copies
    of one more hull vertex (or, with cluster > 0, points this far from it), which
    the octagon of the extremes does not hold; the hull's indices with it."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    c, rho, m = float(1 << 23), 6.0e6, int(0.6 * n)
    pts = torch.randn((n, 2), generator=g, device="cuda").mul_(6.0e5).add_(c)
    far = torch.tensor([c + rho * math.cos(math.pi / 8), c + rho * math.sin(math.pi / 8)], device="cuda")
    pts[:m] = far
    if cluster:
        pts[:m] += torch.randn((m, 2), generator=g, device="cuda").mul_(cluster)
    for k in range(8):
        pts[m + k] = torch.tensor([c + rho * math.cos(k * math.pi / 4), c + rho * math.sin(k * math.pi / 4)])
    pts.round_()
    if order == "shuffled":
        pts = pts[torch.randperm(n, generator=g, device="cuda")]
    return pts.contiguous()


@pytest.mark.parametrize("n,order", [(3000, "shuffled"), (15_000, "shuffled"), (20_000, "sorted"), (60_000, "shuffled"),
                                     (1_000_000, "shuffled"), (1_000_003, "sorted"), (50_000_000, "shuffled")])
def test_copies_of_a_vertex(lib, n, order):
    """Every copy lies in one range of u: in a queue's block, in the sort (a run of
    equal keys over several of its tiles), and in one tile of u ranges."""
    pts = _far_copies(n, order)
    few = torch.unique(pts, dim=0)   # the hull's coordinates, then their lowest indices
    want = few[torch.from_numpy(oracle.hull(few.cpu().numpy())).cuda().long()]
    assert want.shape[0] == 9
    first = [int((pts == v).all(1).nonzero()[0]) for v in want]
    got = lib.hull(pts)
    assert got.tolist() == first


@pytest.mark.parametrize("n", [30_000, 3_000_000])
def test_cluster_beyond_the_octagon(lib, n):
    pts = _far_copies(n, "shuffled", 3.0e4)
    np.testing.assert_array_equal(lib.hull(pts).cpu().numpy(), oracle.hull(pts.cpu().numpy()))


def _stairs(m, copies, seed):
    """A convex curve of m points in the range of few others' u, each copied;
    the copies of one point follow each other."""
    i = np.arange(m, dtype=np.int64)
    arc = np.stack([i * 1500, np.concatenate([[0], np.cumsum(i[:-1] - m // 2)])], 1)
    arc[:, 1] += 5 - arc[:, 1].min()
    return np.repeat(arc[np.random.default_rng(seed).permutation(m)], copies, axis=0).astype(np.float32)


@pytest.mark.parametrize("m,copies", [(300, 60), (5000, 4), (300, 3000)])
def test_copies_of_every_vertex(lib, m, copies):
    pts = _stairs(m, copies, m)
    want = oracle.hull(pts)
    assert want.size == m
    d = torch.from_numpy(pts).cuda()
    np.testing.assert_array_equal(lib.hull(d).cpu().numpy(), want)
    off = np.array([0, pts.shape[0], 2 * pts.shape[0], 2 * pts.shape[0] + 1000])
    sets = lib.hull_batched(torch.cat([d, d.flip(0), d[:1000]]), off)
    np.testing.assert_array_equal(sets[0].cpu().numpy(), want)
    np.testing.assert_array_equal(sets[1].cpu().numpy(), oracle.hull(np.ascontiguousarray(pts[::-1])))


LEFT_TO_THE_SINGLE_HULL = 2   # ch_batched_counters' stage


def test_batched_sets_left_to_the_single_hull(lib):
    """Circles of more than 10,240 records a queue, whose bucket chains overflow,
    beside sets that the batch finishes itself."""
    sets = [_circle(n, n) for n in (120_000, 3000, 250_000, 60_000)]
    off = np.zeros(len(sets) + 1, np.int64)
    off[1:] = np.cumsum([s.shape[0] for s in sets])
    got = lib.hull_batched(torch.from_numpy(np.concatenate(sets)).cuda(), off)
    stages = [c["stage"] for c in lib.ch_batched_counters(len(sets), torch.cuda.current_stream().cuda_stream)]
    assert stages[0] == stages[2] == LEFT_TO_THE_SINGLE_HULL and stages[1] != LEFT_TO_THE_SINGLE_HULL
    for i, s in enumerate(sets):
        np.testing.assert_array_equal(got[i].cpu().numpy(), oracle.hull(s), err_msg=str(i))


def test_served_request_left_to_the_single_hull(lib):
    reqs = [_circle(120_000, 1), _circle(5000, 2), _circle(200_000, 3)]
    srv = lib.ch_server_create(2 << 30, 0)
    try:
        tickets = [lib.ch_submit(srv, p.ctypes.data, p.shape[0])[1] for p in reqs]
        left, end = set(range(len(reqs))), time.time() + 60.0
        while left and time.time() < end:
            for i in list(left):
                buf = np.empty(reqs[i].shape[0], np.int32)
                status, h = lib.ch_poll(srv, tickets[i], buf.ctypes.data, buf.size)
                if status != lib.CH_PENDING:
                    assert status == lib.CH_OK, lib.ch_strerror(status)
                    np.testing.assert_array_equal(buf[:h], oracle.hull(reqs[i]), err_msg=str(i))
                    left.discard(i)
        assert not left
        assert sum(batch[7] for batch in lib.ch_server_trace(srv)) == 2   # sets redone
    finally:
        lib.ch_server_destroy(srv)

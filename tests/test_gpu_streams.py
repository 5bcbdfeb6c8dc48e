"""Calls beside other work on the GPU: a hull on one stream does not wait for
another stream's kernel, whichever of its ways the data take."""
import numpy as np
import pytest

import oracle
from synth import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BUSY_CYCLES = 400_000_000   # about 0.2 s of one SM


@pytest.mark.parametrize("kind,n", [("uniform", 1_000_000), ("normal", 6_000_000), ("ring", 300_000),
                                    ("ring", 6_000_000)])
def test_hull_beside_a_busy_sm(lib, kind, n):
    pts = W.make(kind, n, 31)
    want = oracle.hull(pts)
    busy, mine = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(mine):
        d = torch.from_numpy(pts).cuda()
        out_idx = torch.empty(n, dtype=torch.int32, device="cuda")
        out_n = torch.empty(1, dtype=torch.int64, device="cuda")
        for _ in range(3):   # launched, captured, replayed: nothing left to allocate
            lib.hull(d, out_idx=out_idx, out_n=out_n)
        out_idx.fill_(-7)
    with torch.cuda.stream(busy):
        torch.cuda._sleep(100)   # loaded
    torch.cuda.synchronize()
    ended = torch.cuda.Event()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(BUSY_CYCLES)
        ended.record()
    with torch.cuda.stream(mine):
        for _ in range(5):
            lib.hull(d, out_idx=out_idx, out_n=out_n, sync=False)
        mine.synchronize()
    beside = not ended.query()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out_idx[:int(out_n.item())].cpu().numpy(), want)
    assert beside, "the calls ended only after the other stream's kernel"

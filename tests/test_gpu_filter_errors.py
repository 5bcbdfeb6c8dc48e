"""A filter call that meets a bad coordinate leaves the caller's labels alone,
whether it reads the points once or twice."""
import numpy as np
import pytest

from synth import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fn", ["ch_filter", "ch_filter_manhattan", "ch_filter16"])
@pytest.mark.parametrize("n", [3000, (1 << 21) + 77, 20_000_003])
@pytest.mark.parametrize("at", [0, -1])
def test_labels_stay_on_a_bad_coordinate(lib, fn, n, at):
    pts = torch.from_numpy(W.make("normal", n, 6)).cuda()
    pts[at, 1] = float(1 << 24)
    ext = torch.empty(16, dtype=torch.int32, device="cuda")
    lab = torch.full((n + 32,), 77, dtype=torch.uint8, device="cuda")
    cnt = torch.empty(4, dtype=torch.int64, device="cuda")
    getattr(lib, fn)(pts.data_ptr(), n, ext.data_ptr(), lab.data_ptr() + 5, cnt.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    assert cnt.tolist() == [lib.CH_ERANGE] * 4
    assert bool((lab == 77).all())

"""An augmented pattern is the same bits whatever batch its structure is in."""
import numpy as np
import pytest

from paper_2602_11709_gb300 import synth

pytestmark = pytest.mark.gpu


def _rows(xrd, h, b, n_pts):
    import torch
    n = b.n_struct
    o, grid = synth.Opts(tt_min=5.0, tt_max=90.0), synth.Grid(n_pts=n_pts, dt=85.0 / (n_pts - 1))
    db, co = xrd.DeviceBatch.from_host(b), xrd.make_opts(o)
    full = lambda v: torch.full((n,), v, dtype=torch.float64, device="cuda")  # noqa: E731
    y = torch.empty(n, n_pts, dtype=torch.float32, device="cuda")
    status, totals = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.int64, device="cuda")
    h.pattern_augmented(db, co, xrd.make_grid(grid), full(0.2), full(0.5), y, status, totals,
                        xrd.workspace(h.query_sizes(db, co).ws_grad_bytes))
    return y.cpu().numpy()


@pytest.mark.parametrize("n_pts", [600, 1024, 1025, 1100, 2049, 4096])
def test_alone_and_in_a_batch(gpu_lib, n_pts):
    b, _ = synth.small(n=310)  # some with a few reflections, most with several chunks of them
    h = gpu_lib.Handle(0)
    try:
        y = _rows(gpu_lib, h, b, n_pts)
        for s in (0, 1, 7, 155, 309):
            assert np.array_equal(_rows(gpu_lib, h, b.subset(np.array([s])), n_pts)[0], y[s])
    finally:
        h.close()

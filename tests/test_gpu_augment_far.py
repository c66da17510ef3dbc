"""The augmented pattern's far Lorentzians, interpolated over blocks of 256 points, against the oracle: grids around the
block and CTA sizes, widths from below a grid step to wider than the grid, reflections off both ends of the grid.
The bar is that of every augmented pattern: 1e-5 of the structure's largest value at every grid point."""
import numpy as np
import pytest

import oracle
from paper_2602_11709_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.mark.parametrize("n_pts,n", [(1, 3), (255, 3), (257, 3), (1024, 5), (1025, 310), (2050, 160), (4099, 3)])
@pytest.mark.parametrize("fwhm,eta", [(0.01, 1.0), (0.1, 1.0), (0.1, 0.5), (2.0, 0.3), (40.0, 1.0)])
def test_far_sum(gpu_lib, n_pts, n, fwhm, eta):
    import torch
    rng = np.random.default_rng(n_pts)
    b = synth.concat([synth.random_cell(rng, 3 + i % 5, edge=(5.0, 9.0)) for i in range(n)])
    o = synth.Opts(tt_min=5.0, tt_max=90.0)
    grid = synth.Grid(t0=20.0, dt=50.0 / max(n_pts - 1, 250), n_pts=n_pts)
    h = gpu_lib.Handle(0)
    db, co = gpu_lib.DeviceBatch.from_host(b), gpu_lib.make_opts(o)
    full = lambda v: torch.full((n,), v, dtype=torch.float64, device="cuda")  # noqa: E731
    y = torch.empty(n, n_pts, dtype=torch.float32, device="cuda")
    status, totals = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.int64, device="cuda")
    h.pattern_augmented(db, co, gpu_lib.make_grid(grid), full(fwhm), full(eta), y, status, totals,
                        gpu_lib.workspace(h.query_sizes(db, co).ws_grad_bytes))
    got = y.cpu().numpy()
    h.close()
    for s in (0, 1, n - 1):
        hkl, _ = oracle.enumerate_refl(b.lattice[s], o)
        ref = oracle.augmented(b, s, hkl, o.wavelength, grid.t0, grid.dt, n_pts, fwhm, eta)
        assert np.abs(got[s] - ref).max() <= TOL * ref.max()

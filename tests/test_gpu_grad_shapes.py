"""The gradient kernels at the edges of their forms: atom counts that make 256, 8, 2 or 1 sums per atom and more than
one chunk of atoms, reflection counts around a stage, a structure without reflections, one with an invalid atom, few
and many grid points. Against the oracle's gradient, at the bar of the gradient tests (1e-3 of each group's norm)."""
import numpy as np
import pytest

import oracle
from paper_2602_11709_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_pts,fwhm", [(33, 2.0), (700, 0.3), (5000, 0.08)])
def test_shapes(gpu_lib, n_pts, fwhm):
    import torch
    rng = np.random.default_rng(n_pts)
    counts = [1, 3, 31, 64, 65, 128, 129, 256, 300, 12, 7]
    b = synth.concat([synth.random_cell(rng, n, edge=(4.0, 10.0)) for n in counts])
    b.lattice[9, :3] = 0.7  # no reflection in range
    b.frac[b.atom_off[10] + 2, 1] = np.nan
    o = synth.Opts(tt_min=5.0, tt_max=90.0)
    grid = synth.Grid(n_pts=n_pts, dt=85.0 / (n_pts - 1), fwhm=fwhm)
    n, N = b.n_struct, b.n_atoms
    h = gpu_lib.Handle(0)
    db, co, cg = gpu_lib.DeviceBatch.from_host(b), gpu_lib.make_opts(o), gpu_lib.make_grid(grid)
    ws = gpu_lib.workspace(h.query_sizes(db, co).ws_grad_bytes)
    y = torch.empty(n, n_pts, dtype=torch.float32, device="cuda")
    status, totals = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.int64, device="cuda")
    h.pattern_broadened(db, co, cg, y, status, totals, ws)
    g = rng.standard_normal((n, n_pts)).astype(np.float32)
    out = [torch.full(s, np.nan, dtype=torch.float32, device="cuda") for s in ((N, 3), (N,), (n, 6))]
    h.pattern_grad(db, co, cg, torch.from_numpy(g).cuda(), *out, ws)
    d_frac, d_B, d_lat = (t.cpu().numpy().astype(np.float64) for t in out)
    h.close()
    assert status.cpu().numpy().tolist() == [0] * 10 + [gpu_lib.XRD_EINVAL] and int(totals[3]) == 1
    for s in range(n):
        sl = b.atoms_of(s)
        if s >= 9:  # nothing to differentiate: zeros
            assert not d_frac[sl].any() and not d_B[sl].any() and not d_lat[s].any() and not y[s].any()
            continue
        hkl, _ = oracle.enumerate_refl(b.lattice[s], o)
        ref = oracle.broadened_grad(b, s, hkl, o.wavelength, grid, g[s])
        yr = oracle.broadened(b, s, hkl, o.wavelength, grid)
        assert np.abs(y[s].cpu().numpy() - yr).max() <= 1e-5 * yr.max()
        # the coordinates of a lone atom only move the origin: their gradient is zero and has no norm to compare with
        for got, want in list(zip((d_frac[sl], d_B[sl], d_lat[s]), ref))[counts[s] == 1:]:
            assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want)

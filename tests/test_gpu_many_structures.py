"""Broadened patterns, gradients and augmented patterns of many small structures: every row is that of a small batch, bit
for bit, in each form of the order by reflection count (in the counting, one block, several chunks)."""
import numpy as np
import pytest

from paper_2602_11709_gb300 import synth

pytestmark = pytest.mark.gpu

N_PTS = 200


def _profiles(xrd, h, b):
    """(augmented patterns, broadened patterns, d_frac, d_B, d_lattice), each one row a structure"""
    import torch
    n, N = b.n_struct, b.n_atoms
    o, grid = synth.Opts(tt_min=5.0, tt_max=90.0), synth.Grid(n_pts=N_PTS, dt=85.0 / (N_PTS - 1), fwhm=0.7)
    db, co, cg = xrd.DeviceBatch.from_host(b), xrd.make_opts(o), xrd.make_grid(grid)
    ws = xrd.workspace(h.query_sizes(db, co).ws_grad_bytes)
    new = lambda *s: torch.full(s, np.nan, dtype=torch.float32, device="cuda")  # noqa: E731
    full = lambda v: torch.full((n,), v, dtype=torch.float64, device="cuda")  # noqa: E731
    y, ya = new(n, N_PTS), new(n, N_PTS)
    status, totals = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.int64, device="cuda")
    h.pattern_augmented(db, co, cg, full(0.7), full(0.4), ya, status, totals, ws)
    h.pattern_broadened(db, co, cg, y, status, totals, ws)
    g = torch.cos(torch.arange(N_PTS, device="cuda") * 0.1).repeat(n, 1).contiguous()
    out = [new(N, 3), new(N), new(n, 6)]
    h.pattern_grad(db, co, cg, g, *out, ws)
    assert not status.any()
    split = lambda v: [v[b.atom_off[s]:b.atom_off[s + 1]] for s in range(n)]  # noqa: E731
    return [ya.cpu().numpy(), y.cpu().numpy(), split(out[0].cpu().numpy()), split(out[1].cpu().numpy()), out[2].cpu().numpy()]


@pytest.mark.parametrize("n", [300, 3000, 9000])
@pytest.mark.parametrize("atoms", [1, 3])
def test_rows_of_a_large_batch(gpu_lib, n, atoms):
    rng = np.random.default_rng(n + atoms)
    N = n * atoms
    lat = np.hstack([rng.uniform(0.6, 5.0, (n, 3)), rng.uniform(75.0, 105.0, (n, 3))])  # some without reflections
    b = synth.Batch(lat, atoms * np.arange(n + 1, dtype=np.int64), rng.random((N, 3)),
                    rng.integers(1, synth.ZMAX + 1, N).astype(np.int16), np.ones(N), rng.uniform(0.0, 2.0, N),
                    synth.coef_table(rng))
    h = gpu_lib.Handle(0)
    try:
        whole = _profiles(gpu_lib, h, b)
        rows = np.concatenate([np.arange(0, 40), np.arange(n - 60, n)])
        part = _profiles(gpu_lib, h, b.subset(rows))
        for w, p in zip(whole, part):
            assert all(np.isfinite(v).all() for v in w)
            assert all(np.array_equal(w[s], v) for s, v in zip(rows, p))
    finally:
        h.close()


def test_few_atoms_on_average(gpu_lib):
    """Batches of up to 8 atoms a structure on average form the atoms' sums in one CTA, others in clusters: the same bits, for
    structures of any size among them."""
    rng = np.random.default_rng(11)
    counts = [1, 2, 5, 8, 9, 31, 64, 65, 128, 200, 256, 257, 300]
    cells = [synth.random_cell(rng, c, edge=(3.0, 8.0)) for c in counts]
    cells.append(synth.random_cell(rng, 3, edge=(0.5, 0.6)))  # no reflections
    many = synth.concat(cells + [synth.random_cell(rng, 1, edge=(3.0, 5.0)) for _ in range(300)])
    assert many.n_atoms <= 8 * many.n_struct
    h = gpu_lib.Handle(0)
    try:
        whole = _profiles(gpu_lib, h, many)
        part = _profiles(gpu_lib, h, many.subset(np.arange(len(cells))))
        for w, p in zip(whole, part):
            assert all(np.array_equal(w[s], v) for s, v in enumerate(p))
    finally:
        h.close()

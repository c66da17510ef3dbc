"""Merged peaks of many members against the oracle: cubic, hexagonal and orthorhombic cells, where equal and nearly
equal |g| make peaks of 1 to over 100 Friedel-unique members (one thread, a warp's lanes, or more than a warp holds),
and tolerances that make runs of close reflections split at an anchor."""
import numpy as np
import pytest

import oracle
from paper_2602_11709_gb300 import adapter, synth

from parity import compare_batch

pytestmark = pytest.mark.gpu


def _cells():
    rng = np.random.default_rng(5)
    lat = [[7.0] * 3 + [90.0] * 3, [4.1] * 3 + [90.0] * 3, [5.0, 5.0, 8.0, 90.0, 90.0, 120.0], [6.0, 6.0, 6.002, 90.0, 90.0, 90.0],
           [11.0] * 3 + [90.0] * 3]
    b = synth.concat([synth.random_cell(rng, 1 + i) for i in range(len(lat))])
    b.lattice = np.array(lat)
    return b


@pytest.mark.parametrize("prec", ["fp64", "fp32_phasefix"])
@pytest.mark.parametrize("tol", [1e-5, 0.02, 0.3])
@pytest.mark.parametrize("group", [None, "mmm"])
def test_many_members(gpu_lib, prec, tol, group):
    b = _cells()
    o = synth.Opts(tt_max=100.0, tt_tol=tol, rel_cutoff=1e-4)
    if group:
        o.point_group = adapter.laue_group_ops(group)
    ref = oracle.pattern_batch(b, o)
    assert max(len(p) and int(np.diff(f).max()) for p, f in zip(ref["peak_tt"], ref["peak_fam_off"])) >= (2 if tol > 1e-4 else 1)
    got = gpu_lib.compute(b, o, prec)
    compare_batch(got, ref, prec, o.rel_cutoff, o.scaled)


@pytest.mark.parametrize("n", [60, 700, 2500])  # one launch, three, eight
def test_invalid_and_empty_structures_between_others(gpu_lib, n):
    """Structures with an invalid atom or without reflections in the size classes' queues: the others' outputs are
    those of a batch without them, bit for bit."""
    rng = np.random.default_rng(n)
    o = synth.Opts(tt_max=60.0)
    cells, good = [], []
    for i in range(n):
        b = synth.random_cell(rng, int(rng.integers(1, 9)))
        b.lattice[0, :3] = rng.uniform(3.0, 25.0 if i % 10 == 0 else 10.0) * rng.uniform(0.9, 1.1, 3)
        if i % 3 == 1:
            b.frac[0, 0] = np.nan
        elif i % 7 == 2:
            b.lattice[0, :3] = 0.7
        else:
            good.append(i)
        cells.append(b)
    got = gpu_lib.compute(synth.concat(cells), o)
    ref = gpu_lib.compute(synth.concat([cells[i] for i in good]), o)
    want = np.where(np.arange(n) % 3 == 1, gpu_lib.XRD_EINVAL, 0)
    assert np.array_equal(got["status"], want)
    for k, i in enumerate(good):
        for f in ("peak_tt", "peak_I", "peak_d", "peak_fam_off"):
            assert np.array_equal(got[f][i], ref[f][k])
    for i in set(range(n)) - set(good):
        assert len(got["peak_tt"][i]) == 0


@pytest.mark.parametrize("prec", ["fp64", "fp32_phasefix"])
@pytest.mark.parametrize("n", [1, 2, 5])
def test_flat_passes_any_counts(gpu_lib, prec, n):
    """Structures above the shared-memory classes, whose counts leave every remainder of the scans' four elements."""
    rng = np.random.default_rng(n)
    b = synth.concat([synth.random_cell(rng, 2) for _ in range(n)])
    b.lattice[:, :3] = 25.0 + 0.2 * np.arange(n)[:, None] + [0.0, 0.7, 1.3]
    o = synth.Opts(tt_max=60.0, rel_cutoff=1e-3)
    got = gpu_lib.compute(b, o, prec)
    ref = oracle.pattern_batch(b, o)
    assert got["sizes"]["n_refl"] > 6144 * n
    compare_batch(got, ref, prec, o.rel_cutoff, o.scaled)


@pytest.mark.parametrize("prec", ["fp64", "fp32_phasefix"])
@pytest.mark.parametrize("tol", [1.0, 8.0, 200.0])
@pytest.mark.parametrize("group", [None, "mmm"])
def test_peaks_of_hundreds_and_thousands(gpu_lib, prec, tol, group):
    """Peaks beyond what a warp holds in registers: families, sums and the largest peak, up to one peak of all reflections."""
    b = _cells()
    rng = np.random.default_rng(6)
    b = synth.concat([b, synth.random_cell(rng, 3, edge=(12.0, 13.0)), synth.random_cell(rng, 2, edge=(3.0, 3.5))])
    o = synth.Opts(tt_max=100.0, tt_tol=tol, rel_cutoff=1e-4)
    if group:
        o.point_group = adapter.laue_group_ops(group)
    ref = oracle.pattern_batch(b, o)
    members = [int(m.sum()) // 2 for m in ref["fam_mult"]]
    assert max(members) <= 6144 and max(m / max(len(p), 1) for m, p in zip(members, ref["peak_tt"])) > 30
    compare_batch(gpu_lib.compute(b, o, prec), ref, prec, o.rel_cutoff, o.scaled)

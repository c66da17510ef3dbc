"""The FP64 structure factor (fixed-point exp and sin/cos) and the FP64-accurate phase against the oracle, at the
edges of their forms: atom counts around the staging chunk, coordinates outside [0, 1), occupancies other than 1,
and coefficients that the fixed-point exponential covers, saturates on or leaves to the library's exp."""
import numpy as np
import pytest

import oracle
from paper_2602_11709_gb300 import synth

from parity import compare_batch

pytestmark = pytest.mark.gpu


def _batch(rng, counts):
    b = synth.concat([synth.random_cell(rng, n, edge=(3.0, 7.0)) for n in counts])
    b.frac = rng.uniform(-3.0, 3.0, b.frac.shape)
    b.occ = rng.choice([0.0, 0.25, 1.0, 1.0, 1.75], b.n_atoms)
    b.occ[b.atom_off[:-1]] = 1.0  # no structure without scattering
    return b


@pytest.mark.parametrize("prec", ["fp64", "fp32_phase64"])
@pytest.mark.parametrize("form", ["plain", "B_zero_and_large", "b_zero_and_large"])
def test_forms(gpu_lib, prec, form):
    rng = np.random.default_rng(20)
    b = _batch(rng, [1, 31, 32, 33, 64, 65, 127, 129])
    if form == "B_zero_and_large":
        b.B[::3] = 0.0
        b.B[1::5] = 3000.0
    elif form == "b_zero_and_large":
        b.coef[::2, 0, 1] = 0.0
        b.coef[1::3, 1, 1] = 5e4
        b.coef[::5, 2] = 0.0
    o = synth.Opts(rel_cutoff=0.0, scaled=0)
    got = gpu_lib.compute(b, o, prec)
    compare_batch(got, oracle.pattern_batch(b, o), prec, o.rel_cutoff, o.scaled)


@pytest.mark.parametrize("form", ["B_negative", "b_negative", "b_beyond_range"])
def test_library_exp_forms(gpu_lib, form):
    """Exponents that grow or lie outside the fixed-point range take the library's exp, atom by atom."""
    rng = np.random.default_rng(21)
    b = _batch(rng, [1, 33, 40])
    if form == "B_negative":
        b.B[::4] = -0.7
    elif form == "b_negative":
        b.coef[::2, 3, 1] = -0.3
    else:
        b.coef[::2, 3, 1] = 1e-310
        b.coef[1::2, 2, 1] = 1e305
    o = synth.Opts(rel_cutoff=0.0, scaled=0)
    got = gpu_lib.compute(b, o, "fp64")
    compare_batch(got, oracle.pattern_batch(b, o), "fp64", o.rel_cutoff, o.scaled)


@pytest.mark.parametrize("bits", [20, 33, 34])  # phases in whole units of 2^-32 turns, at ties of them, at quarters
def test_phase_as_fp64_rounds_it(gpu_lib, bits):
    """XRD_FP32_PHASE64's integer phase rounds as the FP64 one. Coordinates shifted by 2^16 (their phases are exact in
    FP64 too) leave nearly every term to the FP64 evaluation: the intensities are the same bits."""
    rng = np.random.default_rng(bits)
    b = synth.concat([synth.random_cell(rng, n, edge=(3.0, 4.0)) for n in (1, 7, 40, 129)])
    b.frac = (2.0 * rng.integers(0, 2 ** (bits - 1), b.frac.shape) + 1.0) * 2.0 ** -bits
    o = synth.Opts(tt_max=60.0, rel_cutoff=0.0, scaled=0)
    one = gpu_lib.compute(b, o, "fp32_phase64")
    b.frac = b.frac + 2.0 ** 16
    two = gpu_lib.compute(b, o, "fp32_phase64")
    for s in range(b.n_struct):
        assert len(one["peak_I"][s]) > 10
        assert np.array_equal(one["peak_I"][s], two["peak_I"][s])


def test_zero_coefficients_at_large_s(gpu_lib):
    """B = 0 and b = 0 where s^2 exceeds 1024: their exponentials are 1 at any angle and wavelength."""
    rng = np.random.default_rng(22)
    b = synth.concat([synth.random_cell(rng, n, edge=(1.5, 2.5)) for n in (1, 5, 33)])
    b.B[:] = 0.0
    b.coef[::2, 0, 1] = 0.0
    o = synth.Opts(wavelength=0.0251, tt_min=107.0, tt_max=107.05, rel_cutoff=0.0, scaled=0)
    ref = oracle.pattern_batch(b, o)
    assert all(len(p) > 100 for p in ref["peak_tt"])
    compare_batch(gpu_lib.compute(b, o, "fp64"), ref, "fp64", o.rel_cutoff, o.scaled)

"""2-theta and d of every output, whose last steps run in integer and FP32 arithmetic, against the definition in
FP64 over the whole range: the smallest angles, both halves of the arcsine, the table's first steps, 2theta = 180."""
import numpy as np
import pytest

from paper_2602_11709_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edge,tt_max", [(400.0, 2.5), (60.0, 12.0), (8.0, 179.99), (3.2, 180.0)])
@pytest.mark.parametrize("refl", [False, True])
def test_two_theta_and_d(gpu_lib, edge, tt_max, refl):
    rng = np.random.default_rng(int(edge))
    b = synth.concat([synth.random_cell(rng, 2) for _ in range(5)])
    b.lattice[:, :3] = edge * rng.uniform(0.9, 1.1, (5, 3))
    o = synth.Opts(wavelength=1.54184, tt_max=tt_max, rel_cutoff=0.0, tt_tol=1e-9)
    got = gpu_lib.compute(b, o, "fp64", refl=refl)
    for s in range(5):
        tt, d = got["peak_tt"][s], got["peak_d"][s]
        assert len(tt) > 0
        # d from the angle: sin(theta) = lambda / (2 d); 2e-8 degrees is what the table and its FP32 steps leave
        ref = 2.0 * np.degrees(np.arcsin(np.minimum(o.wavelength / (2.0 * d), 1.0)))
        c = np.sqrt(np.maximum(1.0 - (o.wavelength / (2.0 * d)) ** 2, 1e-12))
        assert np.all(np.abs(tt - ref) <= 2e-8 + 2e-12 / c)
        C = np.cos(np.radians(b.lattice[s, 3:]))
        a1, a2, a3 = b.lattice[s, :3]
        G = np.array([[a1 * a1, a1 * a2 * C[2], a1 * a3 * C[1]], [a1 * a2 * C[2], a2 * a2, a2 * a3 * C[0]],
                      [a1 * a3 * C[1], a2 * a3 * C[0], a3 * a3]])
        if refl:
            hkl = got["refl_hkl"][s].astype(np.float64)
            q = np.einsum("ri,ij,rj->r", hkl, np.linalg.inv(G), hkl)
            x = np.minimum(0.5 * o.wavelength * np.sqrt(q), 1.0)
            e = np.abs(got["refl_tt"][s] - 2.0 * np.degrees(np.arcsin(x)))
            assert np.all(e <= 2e-8 + 2e-12 / np.sqrt(np.maximum(1.0 - x * x, 1e-12)))
            np.testing.assert_allclose(d, 1.0 / np.sqrt(np.sort(q)), rtol=1e-12)


@pytest.mark.parametrize("scale", [1.0, 1.5])  # 1.5: no d at a power of two
def test_d_next_to_a_power_of_two(gpu_lib, scale):
    eps = np.linspace(-4e-7, 4e-7, 161)
    rng = np.random.default_rng(5)
    b = synth.concat([synth.random_cell(rng, 1) for _ in eps])
    b.lattice[:, :3] = scale * 4.0 * (1.0 + eps)[:, None]  # cubic: d of (100), (200), (400) around 4, 2 and 1
    b.lattice[:, 3:] = 90.0
    o = synth.Opts(wavelength=0.71073, tt_max=60.0, rel_cutoff=0.0)
    got = gpu_lib.compute(b, o, "fp64")
    for s in range(len(eps)):
        a, d = b.lattice[s, 0], got["peak_d"][s]
        n = np.rint((a / d) ** 2)
        assert {1.0, 4.0, 16.0} <= set(n)
        np.testing.assert_allclose(d, a / np.sqrt(n), rtol=1e-12)

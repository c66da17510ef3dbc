"""Enumeration in parts: structures of more columns than a part holds are counted and emitted by several warps. Counts
of every structure, and the patterns of the first ones, against the oracle: column counts around a part's 32, thin
shells (many columns, too few reflections for every structure's parts to find room), and both part sizes."""
import numpy as np
import pytest

import oracle
from paper_2602_11709_gb300 import synth

from parity import compare_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("runs", [0, 1])
@pytest.mark.parametrize("n", [1, 40, 2048 + 3])
@pytest.mark.parametrize("tt_min,tt_max", [(0.0, 60.0), (59.5, 60.0), (30.0, 75.0)])
def test_parts(gpu_lib, n, tt_min, tt_max, runs):
    rng = np.random.default_rng(n)
    edges = (2.0, 30.0) if n <= 40 else (2.0, 9.0)
    b = synth.concat([synth.random_cell(rng, 1 + i % 3, edge=edges) for i in range(n)])
    b.lattice[: 4] = [[40.0, 41.0, 3.0, 70.0, 80.0, 95.0], [3.0, 40.0, 41.0, 90.0, 90.0, 90.0],
                      [3.1, 3.1, 30.0, 90.0, 90.0, 120.0], [4.3, 4.3, 4.3, 90.0, 90.0, 90.0]][:n]
    o = synth.Opts(tt_min=tt_min, tt_max=tt_max, rel_cutoff=0.0)
    h = gpu_lib.Handle(0)
    try:
        h.set_sf_shape(128, 2, runs)
        cnt = h.reflection_counts(gpu_lib.DeviceBatch.from_host(b), gpu_lib.make_opts(o))
        np.testing.assert_array_equal(2 * cnt, oracle.refl_counts(b, o))
        first = b.subset(np.arange(min(n, 12)))
        got = gpu_lib.compute(b, o, "fp32_phasefix", handle=h)
        assert int(got["totals"][0]) == int(cnt.sum())
        got = {k: v[:12] if isinstance(v, list) else v for k, v in got.items()}
        compare_batch(got, oracle.pattern_batch(first, o), "fp32_phasefix", o.rel_cutoff, o.scaled)
    finally:
        h.close()

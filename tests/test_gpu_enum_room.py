"""Enumeration parts where their room runs out: shells so thin that the workspace, whose size follows the reflections, holds
fewer parts than the columns make, and a count outside a call over more parts than its scratch holds."""
import numpy as np
import pytest

import oracle
from paper_2602_11709_gb300 import synth

from parity import compare_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("runs", [0, 1])
@pytest.mark.parametrize("n", [1, 30])
@pytest.mark.parametrize("width", [0.002, 0.0001])
def test_thin_shells(gpu_lib, n, width, runs):
    rng = np.random.default_rng(n)
    b = synth.concat([synth.random_cell(rng, 2, edge=(20.0, 40.0)) for _ in range(n)])
    o = synth.Opts(tt_min=60.0 - width, tt_max=60.0, rel_cutoff=0.0)
    h = gpu_lib.Handle(0)
    try:
        h.set_sf_shape(128, 2, runs)
        cnt = h.reflection_counts(gpu_lib.DeviceBatch.from_host(b), gpu_lib.make_opts(o))
        np.testing.assert_array_equal(2 * cnt, oracle.refl_counts(b, o))
        got = gpu_lib.compute(b, o, handle=h)
        compare_batch(got, oracle.pattern_batch(b, o), "fp32_phasefix", 0.0, o.scaled)
    finally:
        h.close()


@pytest.mark.parametrize("n", [1000, 2500])  # narrow and wide parts: 115 and 29 a structure or more
def test_more_parts_than_room(gpu_lib, n):
    rng = np.random.default_rng(3)
    few = synth.concat([synth.random_cell(rng, 1, edge=(36.0, 44.0)) for _ in range(5)])
    few.lattice[:, 3:] = [90.0, 95.0, 100.0]
    o = synth.Opts(tt_min=59.99, tt_max=60.0, rel_cutoff=0.0)
    h = gpu_lib.Handle(0)
    try:
        counts = lambda b: h.reflection_counts(gpu_lib.DeviceBatch.from_host(b), gpu_lib.make_opts(o))  # noqa: E731
        want, ref = counts(few), gpu_lib.compute(few, o, handle=h)
        np.testing.assert_array_equal(2 * want, oracle.refl_counts(few, o))
        many = few.subset(np.arange(n) % 5)
        np.testing.assert_array_equal(counts(many), want[np.arange(n) % 5])
        got = gpu_lib.compute(many, o, handle=h)
        for s in range(n):
            assert np.array_equal(got["peak_tt"][s], ref["peak_tt"][s % 5])
            assert np.array_equal(got["peak_I"][s], ref["peak_I"][s % 5])
    finally:
        h.close()

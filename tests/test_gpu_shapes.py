"""The structure-factor tiles that a call takes, by precision, size and who chose the shape."""
import numpy as np
import pytest

from paper_2602_11709_gb300 import synth

pytestmark = pytest.mark.gpu


def _tiles(xrd, h, b, o, prec, tile=-1):
    """(tiles of a call, Friedel-unique reflections per structure, sizes)"""
    db, co = xrd.DeviceBatch.from_host(b), xrd.make_opts(o, prec)
    co.tile = tile
    sz = h.query_sizes(db, co)
    ws, out = xrd.workspace(sz.ws_bytes), xrd.PatternBuffers(db.n_struct, sz.n_refl)
    h.pattern_batch(db, co, out, ws)
    return h.work_counts(db, ws)[2], h.reflection_counts(db, co), sz


def _ceil(cnt, per):
    return int(((cnt + per - 1) // per).sum())


@pytest.mark.parametrize("chosen", ["set", "tuned for fp32_phasefix", "tuned for fp64"])
def test_fp64_shape_stays(gpu_lib, chosen):
    """XRD_FP64 takes one reflection a lane whatever shape the handle holds for the FP32 kernels."""
    xrd = gpu_lib
    b, o = synth.small(n=30)
    h = xrd.Handle(0)
    try:
        if chosen == "set":
            h.set_sf_shape(128, 2, 0)
        else:
            db, co = xrd.DeviceBatch.from_host(b), xrd.make_opts(o, chosen.split()[-1])
            sz = h.query_sizes(db, co)
            h.autotune(db, co, xrd.PatternBuffers(db.n_struct, sz.n_refl), xrd.workspace(sz.ws_bytes))
        for tile in (-1, 64, 128):
            got, cnt, _ = _tiles(xrd, h, b, o, "fp64", tile)
            assert got == _ceil(cnt, 32 if tile == -1 else tile)
        if chosen == "tuned for fp64":  # and its tuning chooses nothing for FP32: two reflections a lane in a small batch
            got, cnt, _ = _tiles(xrd, h, b, o, "fp32_phasefix")
            assert got == _ceil(cnt, 64)
    finally:
        h.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32_phase64", "fp32_phasefix"])
@pytest.mark.parametrize("n", [1, 40, 1024])
@pytest.mark.parametrize("shape", [None, (64, 2, 0), (128, 2, 0)])
@pytest.mark.parametrize("tile", [-1, 64, 128])
def test_sizes_tell_the_tiles_of_a_call(gpu_lib, prec, n, shape, tile):
    xrd = gpu_lib
    b, o = synth.small(n=n)
    h = xrd.Handle(0)
    try:
        if shape:
            h.set_sf_shape(*shape)
        got, _, sz = _tiles(xrd, h, b, o, prec, tile)
        assert sz.n_tiles == got
    finally:
        h.close()

"""The tuner times what an untuned launch would take, so that tuning never picks something slower."""
import pytest

import paper_1901_07294_gb300 as wd
import synth

pytestmark = pytest.mark.gpu


# 1280 blocks of 32 sites (three-warp blocks for FP32 and 5 fields) and 1792 (for FP16, in z-strips of 16 or not)
@pytest.mark.parametrize("dims", [(16, 16, 16, 20), (16, 16, 16, 28)])
@pytest.mark.parametrize("prec", [wd.F32, wd.F16])
@pytest.mark.parametrize("nrhs", [2, 5])
def test_tuner_times_three_warp_blocks_of_the_shared_link_kernel(dims, prec, nrhs):
    ctx = wd.Context(0)
    g = wd.Gauge(ctx, dims, synth.gauge(dims, seed=577))
    table = wd.tune_dslash(ctx, g, prec, 18, full=False, nrhs=nrhs)
    shapes = [(t["threads"], t["variant"]) for t in table]
    strips = [v for v, w in ((3, 0), (5, 16), (6, 8), (7, 4)) if w < dims[2]]
    assert {(t, v) for t in (64, 96, 128, 192, 256) for v in strips} <= set(shapes)
    assert len(shapes) == len(set(shapes)) < 64 and all(t["ms"] > 0 for t in table)


def test_single_field_shapes_as_before():
    ctx = wd.Context(0)
    dims = (8, 8, 8, 8)
    g = wd.Gauge(ctx, dims, synth.gauge(dims, seed=578))
    assert 96 not in {t["threads"] for t in wd.tune_dslash(ctx, g, wd.F32, 18, full=False, with_x=True)}

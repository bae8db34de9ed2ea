"""The mixed-precision CG's hops take the launch shapes that are tuned or pinned for them."""
import numpy as np
import pytest

import oracle
import paper_1901_07294_gb300 as wd
import synth
from tests._gpu import pack_field, unpack_field

pytestmark = pytest.mark.gpu

DIMS, MASS, TOL = (4, 6, 8, 10), 0.2, 1e-10


@pytest.fixture(scope="module")
def case():
    U, b = synth.gauge(DIMS, seed=379), synth.even_spinor(DIMS, seed=391)
    return U, b


def _solve(U, b, prec, recon, graph, pins):
    ctx = wd.Context(0)
    g = wd.Gauge(ctx, DIMS, U)
    fb = pack_field(ctx, DIMS, wd.SITES_EVEN, wd.F64, b)
    fx = wd.alloc_field(DIMS, wd.SITES_EVEN, wd.F64)
    for with_x, threads, variant in pins:
        wd.tune_set_dslash(ctx, g, prec, recon, False, with_x, 1, threads, variant)
    wd.cg_solve(ctx, g, MASS, fx, fb, tol=TOL, inner_prec=prec, inner_recon=recon, use_graph=graph)
    return unpack_field(ctx, DIMS, wd.SITES_EVEN, wd.F64, fx)


@pytest.mark.parametrize("prec", [wd.F32, wd.F16, wd.BF16])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("graph", [False, True])
def test_pinned_schedule_reaches_the_hops_with_an_axpy_term(case, prec, recon, graph):
    """Schedules 0 and 1 add the eight directions in different orders: other last bits of the solution."""
    U, b = case
    v0, v1 = (11, 12) if prec == wd.F32 else (14, 13)
    x0, x1 = (_solve(U, b, prec, recon, graph, [(True, 64, v)]) for v in (v0, v1))
    assert not np.array_equal(x0, x1)
    assert np.array_equal(x0, _solve(U, b, prec, recon, graph, [(True, 128, v0)]))   # the block size moves no sum there


@pytest.mark.parametrize("prec", [wd.F32, wd.F16, wd.BF16])
@pytest.mark.parametrize("variant", [0, 1, 2, 4, 8, 9, 11, 12, 13, 14, 15])
@pytest.mark.parametrize("threads", [32, 256])
def test_every_pinned_shape_solves(case, prec, variant, threads):
    U, b = case
    for graph in (False, True):
        x = _solve(U, b, prec, 18, graph, [(False, threads, variant), (True, threads, variant)])
        r = b - oracle.mdagm(DIMS, U, MASS, x)
        assert np.linalg.norm(r) / np.linalg.norm(b) <= TOL, graph

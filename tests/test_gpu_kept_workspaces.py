"""Workspaces that finished solves leave with the context: given back on request, and counted against a queue's budget."""
import pytest

import paper_1901_07294_gb300 as wd
import synth
from tests._gpu import pack_field

pytestmark = pytest.mark.gpu

SMALL, LARGE = (8, 8, 8, 8), (16, 16, 16, 16)


def _problem(ctx, dims, seed=695):
    import torch
    g = wd.Gauge(ctx, dims, synth.gauge(dims, seed=seed))
    b = pack_field(ctx, dims, wd.SITES_EVEN, wd.F64, synth.even_spinor(dims, seed=seed + 1))
    return dict(gauge=g, mass=0.2, tol=1e-8, x=torch.zeros_like(b), b=b, inner_prec=wd.F16)


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _graph_solve(ctx, p):
    wd.cg_solve(ctx, p["gauge"], p["mass"], p["x"], p["b"], tol=p["tol"], inner_prec=wd.F16, use_graph=True)


def test_trim_gives_the_idle_workspaces_back():
    ctx = wd.Context(0)
    p = _problem(ctx, LARGE)
    size = wd.solve_workspace_bytes(LARGE, wd.F16)
    assert ctx.trim() == 0
    _graph_solve(ctx, p)
    kept = _free()
    assert ctx.trim() == size and _free() >= kept + size - (2 << 20)
    wd.cg_solve_batch(ctx, [dict(p, x=p["x"].clone()) for _ in range(3)], mode=wd.BATCH_GRAPH)
    assert ctx.trim() == 3 * size and ctx.trim() == 0
    _graph_solve(ctx, p)   # and a solve after a trim allocates again
    assert ctx.trim() == size


def test_a_closed_queue_frees_its_workspaces():
    ctx = wd.Context(0)
    p = _problem(ctx, LARGE)
    for _ in range(2):
        q = wd.Queue(ctx, 1 << 30, 4)
        for t in [q.submit(dict(p, x=p["x"].clone())) for _ in range(4)]:
            q.wait(t)
        q.close()
    assert ctx.trim() == 0


def test_kept_workspaces_count_against_a_queue_budget():
    """One kept by a solve on the other lattice is freed when it does not fit beside the request's; one of
    the request's own size is used."""
    ctx = wd.Context(0)
    small, large = _problem(ctx, SMALL), _problem(ctx, LARGE)
    _graph_solve(ctx, large)
    budget = wd.solve_workspace_bytes(SMALL, wd.F16)
    q = wd.Queue(ctx, budget, 1)
    q.wait(q.submit(small))
    q.close()
    assert ctx.trim() == 0
    _graph_solve(ctx, small)
    q = wd.Queue(ctx, budget, 1)
    q.wait(q.submit(small))
    q.close()   # takes the kept one and frees it
    assert ctx.trim() == 0
    _graph_solve(ctx, large)
    q = wd.Queue(ctx, budget + wd.solve_workspace_bytes(LARGE, wd.F16), 1)
    q.wait(q.submit(small))
    q.close()
    assert ctx.trim() == wd.solve_workspace_bytes(LARGE, wd.F16)   # both fit: nothing is freed

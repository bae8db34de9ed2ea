"""Kernels chosen by size, and sums over sites, at the sizes where they can go wrong."""
import numpy as np
import pytest

import oracle
import paper_1901_07294_gb300 as wd
import synth
from tests._gpu import pack_field, to_dev, unpack_field
from tests._lattice import parity, rel_max_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return wd.Context(0)


# 1152 and 1280 blocks of 32 sites even-odd: either side of the shared-link kernels' change of build
# (1216 on 152 SMs), and a lattice smaller than one block
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (16, 16, 16, 18), (16, 16, 16, 20)])
@pytest.mark.parametrize("prec,tol", [(wd.F32, 1e-6), (wd.F16, 2.0 ** -10), (wd.BF16, 2.0 ** -7)])
@pytest.mark.parametrize("nrhs", [2, 5])
def test_shared_link_builds_agree_with_single_fields(ctx, dims, prec, tol, nrhs):
    """Same stored inputs, other order of the FP32 sums (about 100 rounding steps of 2^-24) and
    then the rounding of the stored output, which may fall either way (one unit: 2^-10, 2^-7)."""
    import torch
    g = wd.Gauge(ctx, dims, synth.gauge(dims, seed=77))
    nb = wd.field_bytes(dims, wd.SITES_ODD, prec)
    fin = torch.cat([pack_field(ctx, dims, wd.SITES_ODD, prec, synth.spinor(dims, seed=80 + k)) for k in range(nrhs)])
    out = wd.alloc_field(dims, wd.SITES_EVEN, prec, nrhs)
    wd.dslash_eo_apply(ctx, g, out, fin, None, 0, 0.0, 1.0, nrhs=nrhs, prec=prec)
    one = wd.alloc_field(dims, wd.SITES_EVEN, prec)
    for k in range(nrhs):
        wd.dslash_eo_apply(ctx, g, one, fin[k * nb:(k + 1) * nb], None, 0, 0.0, 1.0, prec=prec)
        a = unpack_field(ctx, dims, wd.SITES_EVEN, prec, one)
        b = unpack_field(ctx, dims, wd.SITES_EVEN, prec, out[k * nb:(k + 1) * nb])
        assert rel_max_err(b, a) < tol, k


# less than a block, ragged, a few blocks per SM (spread over the SMs), and more than fit at once
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 2, 6), (4, 6, 8, 10), (12, 12, 12, 24), (16, 16, 16, 20)])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dagger", [False, True])
def test_f64_three_threads_per_site_agrees_with_one(ctx, dims, recon, dagger):
    """The same operations in the same order: equal up to a last-bit rounding."""
    g = wd.Gauge(ctx, dims, synth.gauge(dims, seed=78))
    g.set_boundary(-1)
    psi = synth.spinor(dims, seed=90)
    fin, x = (pack_field(ctx, dims, s, wd.F64, psi) for s in (wd.SITES_ODD, wd.SITES_EVEN))
    res = []
    for threads, variant in ((128, 0), (96, 15)):
        for with_x in (False, True):
            wd.tune_set_dslash(ctx, g, wd.F64, recon, False, with_x, 1, threads, variant)
            out = wd.alloc_field(dims, wd.SITES_EVEN, wd.F64)
            wd.dslash_eo_apply(ctx, g, out, fin, x if with_x else None, 0, 4.1, -0.06, dagger=dagger, prec=wd.F64,
                               recon=recon)
            res.append(unpack_field(ctx, dims, wd.SITES_EVEN, wd.F64, out))
    wd.tune_clear(ctx)
    assert rel_max_err(res[2], res[0]) < 4e-16 and rel_max_err(res[3], res[1]) < 4e-16


# the sums over sites of the CG iteration: 8 sites (less than a warp), ragged, several parts
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 2, 6), (4, 6, 8, 10), (8, 8, 16, 16)])
@pytest.mark.parametrize("prec", [wd.F32, wd.F16, wd.BF16])
@pytest.mark.parametrize("recon", [18, 12])
def test_cg_on_small_and_ragged_lattices(ctx, dims, prec, recon):
    U = synth.gauge(dims, seed=79)
    g = wd.Gauge(ctx, dims, U)
    b = synth.even_spinor(dims, seed=91)
    fb = pack_field(ctx, dims, wd.SITES_EVEN, wd.F64, b)
    for mode in ("host", "graph", "group"):
        fx = wd.alloc_field(dims, wd.SITES_EVEN, wd.F64)
        if mode == "group":
            wd.cg_solve_batch(ctx, [dict(gauge=g, mass=0.2, tol=1e-10, x=fx, b=fb, inner_prec=prec, inner_recon=recon)],
                              mode=wd.BATCH_GRAPH)
        else:
            wd.cg_solve(ctx, g, 0.2, fx, fb, tol=1e-10, inner_prec=prec, inner_recon=recon, use_graph=mode == "graph")
        x = unpack_field(ctx, dims, wd.SITES_EVEN, wd.F64, fx)
        r = b - oracle.mdagm(dims, U, 0.2, x)
        assert np.linalg.norm(r) / np.linalg.norm(b) <= 1e-10, mode


# full tiles of 128 sites, a part of one, and both
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 2), (6, 2, 4, 6), (4, 6, 8, 10)])
@pytest.mark.parametrize("prec", [wd.F64, wd.F32, wd.F16, wd.BF16, wd.DF])
def test_full_pack_tiles_equal_half_packs(ctx, dims, prec):
    import torch
    psi = to_dev(synth.spinor(dims, seed=92))
    full = pack_field(ctx, dims, wd.SITES_FULL, prec, synth.spinor(dims, seed=92))
    halves = torch.cat([pack_field(ctx, dims, s, prec, synth.spinor(dims, seed=92))
                        for s in (wd.SITES_EVEN, wd.SITES_ODD)])
    assert torch.equal(full, halves)
    one, two = torch.zeros_like(psi.view(-1)), torch.zeros_like(psi.view(-1))
    half = halves.numel() // 2
    wd.unpack(ctx, dims, wd.SITES_FULL, prec, full, one)
    wd.unpack(ctx, dims, wd.SITES_EVEN, prec, halves[:half], two)
    wd.unpack(ctx, dims, wd.SITES_ODD, prec, halves[half:], two)
    assert torch.equal(one, two)
    assert rel_max_err(one.cpu().numpy()[parity(dims).repeat(24) == 0], psi.view(-1).cpu().numpy()[parity(dims).repeat(24) == 0]) < 2.0 ** -8


def test_kept_workspaces_give_the_same_bits():
    """A solve in a workspace that another solve has used, and one queued after it, equal the first;
    closing a queue after its context is allowed."""
    import torch
    ctx = wd.Context(0)
    dims, other = (8, 8, 8, 8), (4, 6, 8, 10)
    g, h = (wd.Gauge(ctx, d, synth.gauge(d, seed=95)) for d in (dims, other))
    b, c = (pack_field(ctx, d, wd.SITES_EVEN, wd.F64, synth.even_spinor(d, seed=96)) for d in (dims, other))
    xs = []
    for _ in range(3):
        x, y = torch.zeros_like(b), torch.zeros_like(c)
        wd.cg_solve(ctx, g, 0.2, x, b, tol=1e-10, inner_prec=wd.F16, use_graph=True)
        wd.cg_solve(ctx, h, 0.3, y, c, tol=1e-9, inner_prec=wd.F16, use_graph=True)
        xs.append((x, y))
    assert all(torch.equal(u, v) for p in xs[1:] for u, v in zip(xs[0], p))
    batches = []
    for _ in range(2):
        out = [torch.zeros_like(b) for _ in range(3)]
        wd.cg_solve_batch(ctx, [dict(gauge=g, mass=0.1 + 0.1 * k, tol=1e-10, x=v, b=b, inner_prec=wd.F16)
                                for k, v in enumerate(out)], mode=wd.BATCH_GRAPH)
        batches.append(out)
    assert all(torch.equal(u, v) for u, v in zip(*batches))
    q = wd.Queue(ctx, 1 << 30, 2)
    x = torch.zeros_like(b)
    q.wait(q.submit(dict(gauge=g, mass=0.2, tol=1e-10, x=x, b=b, inner_prec=wd.F16)))
    ctx.close()
    q.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 2, 6), (4, 6, 8, 10)])
@pytest.mark.parametrize("inner", [wd.F64, wd.F32, wd.F16, wd.BF16])
@pytest.mark.parametrize("outer", [wd.F64, wd.DF])
@pytest.mark.parametrize("kw", [dict(), dict(use_graph=True), dict(reliable=False)], ids=["loop", "graph", "refine"])
def test_reliable_updates_restart_from_the_true_residual(ctx, dims, inner, outer, kw):
    """tol is 12 digits and delta 0.1, so that every inner precision restarts several times.  The
    solver stops at 0.9 tol by its own FP64 residual, whose rounding (2^-53 times |A| |x| / |b| times
    about 100 steps) is below 1e-13: the oracle's residual is then <= tol."""
    U, b = synth.gauge(dims, seed=21), synth.even_spinor(dims, seed=22)
    g = wd.Gauge(ctx, dims, U)
    fb = pack_field(ctx, dims, wd.SITES_EVEN, wd.F64, b)
    fx = wd.alloc_field(dims, wd.SITES_EVEN, wd.F64)
    st = wd.cg_solve(ctx, g, 0.2, fx, fb, tol=1e-12, inner_prec=inner, outer_prec=outer, delta=0.1, **kw)
    x = unpack_field(ctx, dims, wd.SITES_EVEN, wd.F64, fx)
    rel = float(np.linalg.norm(b - oracle.mdagm(dims, U, 0.2, x)) / np.linalg.norm(b))
    assert st["status"] == 0 and rel <= 1e-12, (st, rel)

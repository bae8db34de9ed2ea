"""Block size and build of the shared-link kernel: what a field gets must not depend on the choice."""
import pytest

import paper_1901_07294_gb300 as wd
import synth
from tests._gpu import pack_field, unpack_field
from tests._lattice import rel_max_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return wd.Context(0)


# blocks of 32 sites on 152 SMs: 1152 (the 128-register build for all), 1280 (for FP32 in three-warp blocks
# only), 1536 (the 80-register build, four warps) and 2016 (the same, three warps)
@pytest.mark.parametrize("dims", [(16, 16, 16, 18), (16, 16, 16, 20), (16, 16, 16, 24), (16, 16, 18, 28)])
@pytest.mark.parametrize("prec,tol", [(wd.F32, 1e-6), (wd.F16, 2.0 ** -10), (wd.BF16, 2.0 ** -7)])
@pytest.mark.parametrize("dagger", [False, True])
def test_a_field_gets_the_same_bits_beside_any_number_of_others(ctx, dims, prec, tol, dagger):
    """... and, beside the field alone, another order of the FP32 sums (about 100 rounding steps of
    2^-24) and then the rounding of the stored output, which may fall either way (one unit)."""
    import torch
    g = wd.Gauge(ctx, dims, synth.gauge(dims, seed=177))
    nb = wd.field_bytes(dims, wd.SITES_ODD, prec)
    fin = torch.cat([pack_field(ctx, dims, wd.SITES_ODD, prec, synth.spinor(dims, seed=180 + k)) for k in range(6)])
    x = torch.cat([pack_field(ctx, dims, wd.SITES_EVEN, prec, synth.spinor(dims, seed=180 + k)) for k in range(6)])
    for a, b, xs in ((0.0, 1.0, None), (4.1, -0.06, x)):
        def apply(out, n):
            wd.dslash_eo_apply(ctx, g, out, fin[:n * nb], None if xs is None else xs[:n * nb], 0, a, b, dagger=dagger,
                               nrhs=n, prec=prec)
            return out
        res = {n: apply(wd.alloc_field(dims, wd.SITES_EVEN, prec, n), n) for n in (1, 2, 4, 5, 6)}
        for n in (2, 4, 5):
            assert torch.equal(res[n], res[6][:n * nb]), n
        assert rel_max_err(unpack_field(ctx, dims, wd.SITES_EVEN, prec, res[6][:nb]),
                           unpack_field(ctx, dims, wd.SITES_EVEN, prec, res[1])) < tol

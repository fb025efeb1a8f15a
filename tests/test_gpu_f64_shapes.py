"""Launch shapes of the FP64 plain pass are timed only on lattices where some
pass takes one."""
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


# 608 partitions of 32 lanes.  8^4 and 6x8x8x10: both the pass over one parity and the one over both share a site
# among lanes; 16^3x32 and 20^3x36: only the first does; 24^3x32: neither does
@pytest.mark.parametrize("dims,timed", [((8, 8, 8, 8), False), ((6, 8, 8, 10), False), ((16, 16, 16, 32), True),
                                        ((20, 20, 20, 36), True), ((24, 24, 24, 32), True)])
def test_shape_timed_where_used(dims, timed):
    assert hisq.hisq_stencil_config(-1) == -1
    ctx = hisq.hisq_create(0)
    g = hisq.hisq_load_gauge(ctx, dims, *synth.gauge_pair(dims, seed=0, device="cuda"))
    try:
        p = hisq.prec("f64", 18)
        x = synth.spinor(dims, 1000, full=True, device="cuda")
        full, half = torch.empty_like(x), torch.empty_like(x[0])
        hisq.hisq_dslash(ctx, g, p, 2, 0.0, None, x, full, True)
        assert (hisq.hisq_stencil_config_in_use(g, p, False) >= 0) == timed
        assert hisq.hisq_stencil_config_in_use(g, p, True) >= 0
        hisq.hisq_dslash(ctx, g, p, 0, 0.0, None, x[1].contiguous(), half, True)
        # the terms of a site in one order or shared among lanes: FP64 rounding of 16 terms
        assert float((half - full[0]).abs().max()) <= 1e-14 * float(full.abs().max())
    finally:
        hisq.hisq_free_gauge(ctx, g)
        hisq.hisq_destroy(ctx)

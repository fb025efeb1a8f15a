"""BiCGStab(l)'s kernel chain at the edges of its passes: every l (the
Gram-Schmidt kernels are compiled for 0, 1, 3 and 7 following vectors, the
vector kernels load four fields at a time), lattices below one block and beyond
one row of blocks, each kind of compute precision; the oracle's FP64 residual
decides."""
import numpy as np
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import oracle

    oracle.build()
    c = hisq.hisq_create(0)
    yield c
    hisq.hisq_destroy(c)


def check(ctx, dims, name, recon, l, m=0.2, tol=1e-10):
    import oracle

    fat, lng = synth.gauge_pair(dims, seed=0)
    g = hisq.hisq_load_gauge(ctx, dims, fat.cuda(), lng.cuda())
    try:
        b = synth.spinor(dims, 1000, full=True, device="cuda")
        p = hisq.hisq_default_params()
        p.mass, p.tol, p.on_device, p.l, p.sloppy = m, tol, 1, l, hisq.prec(name, recon)
        x = torch.zeros_like(b)
        st, info = hisq.hisq_bicgstabl(ctx, g, p, b, x)
        assert st == hisq.HISQ_OK
        bn = b.cpu().numpy()
        r = bn - oracle.mfull(dims, fat.numpy(), lng.numpy(), m, x.cpu().numpy())
        assert np.linalg.norm(r) / np.linalg.norm(bn) <= tol
        return info
    finally:
        hisq.hisq_free_gauge(ctx, g)


@pytest.mark.parametrize("l", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("name,recon", [("int20", 12), ("f64", 18), ("int30", 18), ("f32", 12)])
def test_every_l(ctx, l, name, recon):
    check(ctx, (4, 6, 4, 8), name, recon, l)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 4), (10, 12, 14, 24), (16, 16, 24, 48)])
def test_sizes(ctx, dims):
    # 8 sites a parity; under one block; past 304 blocks' first round; 147456 sites: 2304 rows of stencil sums
    check(ctx, dims, "int20", 12, 4)


@pytest.mark.parametrize("name,recon,l", [("int20", 12, 4), ("half", 12, 5), ("int30", 18, 2), ("f64", 18, 1)])
def test_large_lattice(ctx, name, recon, l):
    # 4804 rows of stencil sums, summed once by their own kernel; vector kernels on full waves, a field at a time
    check(ctx, (10, 14, 36, 122), name, recon, l, m=0.5)

"""The buffers a context keeps for later calls go back to the driver on request,
and the calls after that work as before."""
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


def test_given_back():
    dims = (16, 16, 16, 32)
    fat, lng = synth.gauge_pair(dims, seed=0, device="cuda")
    b = synth.spinor(dims, 1000, device="cuda")
    p = hisq.hisq_default_params()
    p.mass, p.tol, p.on_device, p.sloppy = 0.2, 1e-8, 1, hisq.prec("int20")

    def use(ctx):
        x = torch.zeros_like(b)
        g = hisq.hisq_load_gauge(ctx, dims, fat, lng)
        st, _ = hisq.hisq_cg(ctx, g, p, b, x)
        hisq.hisq_free_gauge(ctx, g)
        assert st == hisq.HISQ_OK
        return x

    warm = hisq.hisq_create(0)  # kernels and their local memory
    use(warm)
    hisq.hisq_destroy(warm)
    ctx = hisq.hisq_create(0)
    try:
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        x = use(ctx)
        kept = free0 - torch.cuda.mem_get_info()[0]
        links = 2 * 144 * 4 * dims[0] * dims[1] * dims[2] * dims[3]  # the FP64 copies alone
        assert kept >= links
        hisq.hisq_release_buffers(ctx)
        assert free0 - torch.cuda.mem_get_info()[0] <= kept - links
        assert torch.equal(use(ctx), x)
        hisq.hisq_release_buffers(ctx)
        hisq.hisq_release_buffers(ctx)  # nothing left to give
        hisq.hisq_release_buffers(None)
        assert torch.equal(use(ctx), x)
    finally:
        hisq.hisq_destroy(ctx)

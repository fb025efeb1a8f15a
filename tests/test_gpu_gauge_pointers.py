"""Device link arrays that the load's scan cannot read in place are copied first:
arrays whose address is no multiple of eight give the field an aligned array
gives."""
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fat_off,lng_off", [(0, 0), (8, 8), (4, 0), (0, 1), (2, 4)])
def test_any_alignment(fat_off, lng_off):
    dims = (4, 6, 8, 10)
    fat, lng = synth.gauge_pair(dims, seed=0, device="cuda")
    x = synth.spinor(dims, 1000, device="cuda")

    def shifted(t, off):
        raw = torch.zeros(t.numel() * 8 + 64, dtype=torch.uint8, device="cuda")
        raw[off:off + t.numel() * 8] = t.reshape(-1).view(torch.uint8)
        return raw, raw.data_ptr() + off

    ctx = hisq.hisq_create(0)
    try:
        ref = torch.empty_like(x)
        g = hisq.hisq_load_gauge(ctx, dims, fat, lng)
        hisq.hisq_dslash(ctx, g, hisq.prec("int20"), 0, 0.0, None, x, ref, True)
        scale = [hisq.hisq_gauge_scale(g, i) for i in (0, 1)]
        hisq.hisq_free_gauge(ctx, g)
        (f, fp), (l, lp) = shifted(fat, fat_off), shifted(lng, lng_off)
        torch.cuda.synchronize()
        g = hisq.hisq_load_gauge(ctx, dims, fp, lp, hisq.HISQ_GAUGE_ON_DEVICE)
        out = torch.empty_like(x)
        hisq.hisq_dslash(ctx, g, hisq.prec("int20"), 0, 0.0, None, x, out, True)
        assert torch.equal(out, ref)
        assert [hisq.hisq_gauge_scale(g, i) for i in (0, 1)] == scale
        hisq.hisq_free_gauge(ctx, g)
    finally:
        hisq.hisq_destroy(ctx)

"""The one-pass scan of a gauge field at load: its scale is the exact largest
element, and whether the long links compress (12 reals: row 2 = sign *
conj(row0 x row1); 13 reals: unitary) is decided at 1e-6 wherever the offending
link lies, from either kind of pointer."""
import numpy as np
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hisq.hisq_create(0)
    yield c
    hisq.hisq_destroy(c)


def accepted(ctx, dims, fat, lng, recon, flags=0):
    g = hisq.hisq_load_gauge(ctx, dims, fat, lng, flags)
    try:
        x = synth.spinor(dims, 1000, device="cuda")
        out = torch.empty_like(x)
        torch.cuda.synchronize()
        try:
            hisq.hisq_dslash(ctx, g, hisq.prec("f32", recon), 0, 0.0, None, x, out, True)
            return True
        except hisq.HisqError as e:
            assert "refused" in str(e)
            return False
    finally:
        hisq.hisq_free_gauge(ctx, g)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 6, 2, 10), (6, 4, 8, 14)])
@pytest.mark.parametrize("device", ["cuda", "cpu"])
def test_scale_is_exact(ctx, dims, device):
    fat, lng = synth.gauge_pair(dims, seed=3)
    for where in (0, fat.numel() // 2, fat.numel() - 1):
        f, l = fat.clone(), lng.clone()
        f.view(-1)[where] = -1.75 - 2.0 ** -50
        l.view(-1)[where] = 1.25 + 2.0 ** -51
        g = hisq.hisq_load_gauge(ctx, dims, f.to(device), l.to(device))
        try:
            assert hisq.hisq_gauge_scale(g, 0) == 1.75 + 2.0 ** -50
            assert hisq.hisq_gauge_scale(g, 1) == float(l.abs().max())
        finally:
            hisq.hisq_free_gauge(ctx, g)


# deviations on both sides of the bound, far from it, within 0.1 % of it (decided in FP64) and beyond;
# adding d to a real of row 2 moves it off the product by d, and off unitarity by at most 2 d
@pytest.mark.parametrize("d,ok", [(0.0, True), (9e-7, True), (9.995e-7, True), (1.0005e-6, False), (2e-6, False),
                                  (0.5, False)])
@pytest.mark.parametrize("where", ["first", "middle", "last"])
def test_twelve_reals(ctx, d, ok, where):
    dims = (4, 6, 2, 10)
    fat, lng = synth.gauge_pair(dims, seed=3, antiperiodic_t=True)
    flat = lng.reshape(-1, 18).clone()
    link = {"first": 0, "middle": flat.shape[0] // 2 + 5, "last": flat.shape[0] - 1}[where]
    flat[link, 15] += d
    assert accepted(ctx, dims, fat.cuda(), flat.reshape(lng.shape).cuda(), 12, hisq.HISQ_GAUGE_ANTIPERIODIC_T) == ok


@pytest.mark.parametrize("scale,ok", [(1.0, True), (1.0 + 4.9e-7, True), (1.0 + 5.1e-7, False), (1.0 - 5.1e-7, False),
                                      (40.0, False)])
def test_thirteen_reals(ctx, scale, ok):
    """One link scaled by 1 + e: U U^+ is off by 2 e (+ e^2)."""
    dims = (4, 6, 2, 10)
    fat, lng = synth.gauge_pair(dims, seed=4)
    flat = lng.reshape(-1, 18).clone()
    flat[flat.shape[0] - 3] *= scale
    assert accepted(ctx, dims, fat.cuda(), flat.reshape(lng.shape).cuda(), 13) == ok


def test_large_links_are_decided_in_fp64(ctx):
    """Every link 32 * diag(1, 1, 32) times a sign: row 2 is exactly the product of the others."""
    dims = (4, 4, 4, 4)
    fat = synth.unit_gauge(dims, 0.5)
    lng = synth.unit_gauge(dims, 32.0, long_link=True)
    lng[..., 2, 2, 0] *= 32.0
    # row 2 = sign * conj(row0 x row1) with rows 0 and 1 carrying the sign twice: the sign stays on row 2 alone
    assert accepted(ctx, dims, fat.cuda(), lng.cuda(), 12)
    lng[1, 2, 1, 0, 3, 2, 2, 0] += 1e-3
    assert not accepted(ctx, dims, fat.cuda(), lng.cuda(), 12)

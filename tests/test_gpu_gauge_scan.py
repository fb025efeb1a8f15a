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


@pytest.mark.parametrize("gmax", [1.0, 0.7310585786300049, 3.0e5, 2.0 ** -40, 1e-300, 5e-306])
def test_sixteen_bit_integers_are_the_fp64_rule(ctx, gmax):
    """q = rint(fl(x * fl(32767 / gmax))) in FP64 for every element, ties and neighbours of ties among them,
    read back through the stencil: with one link element per site non-zero and a source that picks it,
    the FP32 output is q * scale exactly representable."""
    dims = (4, 4, 4, 4)
    rng = np.random.default_rng(1)
    fat = np.zeros((4, 4, 4, 4, 4, 3, 3, 2))
    inv = np.float64(32767.0) / np.float64(gmax)
    k = rng.integers(-32767, 32767, (4, 4, 4, 4))
    off = rng.choice([0.5, 0.5 - 2.0 ** -36, 0.5 + 2.0 ** -36, 0.5 - 2.0 ** -21, 0.25, 0.0], k.shape)
    with np.errstate(over="ignore", invalid="ignore"):
        v = (k + off) / inv if np.isfinite(inv) else rng.choice([gmax, -gmax, gmax / 3, 0.0], k.shape)
    fat[0, ..., 0, 0, 0] = v
    fat[1, 0, 0, 0, 0, 2, 2, 1] = gmax  # the field's largest element
    lng = synth.unit_gauge(dims, 1.0, long_link=True).numpy() * 0.0
    lng[...] = 0.0
    with np.errstate(over="ignore", invalid="ignore"):
        want = np.clip(np.where(np.isnan(fat * inv), -32767.0, np.rint(fat * inv)), -32767, 32767)[0, ..., 0, 0, 0]
    g = hisq.hisq_load_gauge(ctx, dims, torch.from_numpy(fat).cuda(), torch.from_numpy(lng).cuda())
    try:
        t, z, y, x = np.meshgrid(*(np.arange(4),) * 4, indexing="ij")
        even = (x + y + z + t) % 2 == 0
        # source 1 on colour 0 of every odd site: out(even, 0) = F_0(x) - F_0(x - 1), and the row of links on the
        # even sites alone is recovered with the odd sites' set to zero in a second field
        fat2 = fat.copy()
        fat2[0, ~even] = 0.0
        g2 = hisq.hisq_load_gauge(ctx, dims, torch.from_numpy(fat2).cuda(), torch.from_numpy(lng).cuda())
        try:
            src = torch.zeros((128, 3, 2), dtype=torch.float64, device="cuda")
            src[:, 0, 0] = 1.0
            out = torch.empty_like(src)
            torch.cuda.synchronize()
            scale = np.float32(np.float64(gmax) / 32767.0)
            if scale == 0:  # below FP32: the pass's scale vanishes and with it the ratio of the fields' scales
                with pytest.raises(hisq.HisqError, match="ERANGE"):
                    hisq.hisq_dslash(ctx, g2, hisq.prec("half", 18), 0, 0.0, None, src, out, True)
                return
            hisq.hisq_dslash(ctx, g2, hisq.prec("half", 18), 0, 0.0, None, src, out, True)
            got = out.cpu().numpy()[:, 0, 0]
        finally:
            hisq.hisq_free_gauge(ctx, g2)
        w = want.reshape(-1)[even.reshape(-1)]
        # the stencil's 16-bit store keeps the largest component of a site to 2^-16 of itself (here the only one)
        ref = w * np.float64(scale)
        assert np.all(np.abs(got - ref) <= 2.0 ** -15 * np.abs(ref))
        # neighbouring integers differ by more than that below 2^14: there the integer itself is determined
        small = np.abs(w) < 2 ** 14
        assert np.array_equal(np.rint(got[small] / np.float64(scale)), w[small])
    finally:
        hisq.hisq_free_gauge(ctx, g)

"""The conversions between the caller's FP64 arrays and the storage formats at
the sizes and values where they can go wrong: site counts around a warp and a
block, doubles that round to the edges of FP32, and stencil calls whose output
array is an input or whose input is refused."""
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


def edge_doubles(n):
    """n finite doubles whose FP32 rounding is finite: ties, carries into the exponent, subnormals."""
    rng = np.random.default_rng(n)
    bits = rng.integers(0, 1 << 23, n, dtype=np.int64)
    e = rng.integers(-152, 127, n)
    tail = rng.choice([0.0, 0.5, 0.5 - 2.0 ** -29, 0.5 + 2.0 ** -29, 1.0 - 2.0 ** -29, 2.0 ** -29], n)
    m = np.where(rng.random(n) < 0.2, (1 << 23) - 1.0, bits.astype(np.float64))
    v = np.ldexp(1.0 + (m + tail) * 2.0 ** -23, e) * rng.choice([-1.0, 1.0], n)
    return np.where(rng.random(n) < 0.05, rng.choice([0.0, -0.0], n), v)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 4099])
def test_f32_rounding_and_site_counts(ctx, n):
    x = edge_doubles(6 * n)
    want = x.astype(np.float32)
    assert np.isfinite(want).all()
    xd = torch.from_numpy(np.concatenate([x, [7.0]])).cuda()
    sf = hisq.SPINOR_FMT["f32"]
    packed = torch.empty(hisq.hisq_spinor_bytes(sf, n), dtype=torch.uint8, device="cuda")
    out = torch.full((6 * n + 1,), 5.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert hisq.hisq_spinor_pack(ctx, sf, n, xd, packed) == 0
    hisq.hisq_spinor_unpack(ctx, sf, hisq.HISQ_COMPUTE_F32, n, packed, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert got[-1] == 5.0  # nothing past the last site
    back = got[:-1]
    assert np.array_equal(back, want.astype(np.float64))
    assert np.array_equal(np.signbit(back), np.signbit(want))


@pytest.mark.parametrize("name,recon", [("int20", 12), ("f64", 18), ("int30", 18)])
def test_in_place_and_refused_inputs(ctx, name, recon):
    dims = (4, 6, 2, 8)
    fat, lng = synth.gauge_pair(dims, seed=0, device="cuda")
    g = hisq.hisq_load_gauge(ctx, dims, fat, lng)
    try:
        p = hisq.prec(name, recon)
        x = synth.spinor(dims, 1000, full=True, device="cuda")
        y = synth.spinor(dims, 1001, full=True, device="cuda")
        ref = torch.empty_like(x)
        hisq.hisq_dslash(ctx, g, p, 2, 0.3, y, x, ref, True)
        for which in (0, 1):  # the output over the input, then over the xpay field
            xx, yy = x.clone(), y.clone()
            torch.cuda.synchronize()
            out = xx if which == 0 else yy
            hisq.hisq_dslash(ctx, g, p, 2, 0.3, yy, xx, out, True)
            assert torch.equal(out, ref)
        for where in (0, 1):  # a non-finite input or xpay field: refused, the output untouched
            xx, yy = x.clone(), y.clone()
            (xx if where == 0 else yy)[1, 3, 1, 0] = float("inf")
            out = torch.full_like(x, 2.5)
            torch.cuda.synchronize()
            with pytest.raises(hisq.HisqError, match="non-finite"):
                hisq.hisq_dslash(ctx, g, p, 2, 0.3, yy, xx, out, True)
            assert bool((out == 2.5).all())
            hisq.hisq_dslash(ctx, g, p, 2, 0.3, y, x, out, True)  # and the next call is right
            assert torch.equal(out, ref)
    finally:
        hisq.hisq_free_gauge(ctx, g)

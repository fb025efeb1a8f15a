"""16-bit links over the whole range of field sizes whose scale FP32 holds: the
integers are rint(fl(x fl(32767 / gmax))) in FP64 also where the scale's inverse
or the elements leave the range of the conversion's FP32 pairs."""
import numpy as np
import pytest
import torch

from paper_2302_09224_gb300 import hisq

pytestmark = pytest.mark.gpu


# the pair of inv loses bits below inv = 2^-73 (gmax 3.1e26), elements leave it at 2^127
@pytest.mark.parametrize("gmax", [2.0 ** 86, 3.2e26, 1e27, 1e33, 2.0 ** 127, 2.0 ** 128, 1e39, 1e42])
def test_large_fields(gmax):
    dims = (4, 4, 4, 4)
    rng = np.random.default_rng(2)
    inv = np.float64(32767.0) / np.float64(gmax)
    k = rng.integers(-16000, 16000, (4, 4, 4, 4))
    off = rng.choice([0.5, 0.5 - 2.0 ** -36, 0.5 + 2.0 ** -36, 0.5 - 2.0 ** -21, 0.25, 0.0], k.shape)
    t, z, y, x = np.meshgrid(*(np.arange(4),) * 4, indexing="ij")
    even = (x + y + z + t) % 2 == 0
    fat = np.zeros((4, 4, 4, 4, 4, 3, 3, 2))
    fat[0, ..., 0, 0, 0] = np.where(even, (k + off) / inv, 0.0)  # out(even, 0) = F_0(x), F_0(x - 1) is zero
    fat[1, 0, 0, 0, 0, 2, 2, 1] = gmax  # the field's largest element
    want = np.rint(fat[0, ..., 0, 0, 0] * inv).reshape(-1)[even.reshape(-1)]
    ctx = hisq.hisq_create(0)
    g = None
    try:
        g = hisq.hisq_load_gauge(ctx, dims, torch.from_numpy(fat).cuda(), torch.zeros(fat.shape, dtype=torch.float64,
                                                                                     device="cuda"))
        src = torch.zeros((128, 3, 2), dtype=torch.float64, device="cuda")
        src[:, 0, 0] = 2.0 ** -100  # keeps the products in FP32's range
        out = torch.empty_like(src)
        torch.cuda.synchronize()
        hisq.hisq_dslash(ctx, g, hisq.prec("half", 18), 0, 0.0, None, src, out, True)
        unit = np.float64(np.float32(np.float64(gmax) / 32767.0)) * 2.0 ** -100
        # the 16-bit records keep a site's largest component (here the only one) to 2^-15 of itself, less than half
        # a step of the integers below 2^14
        assert np.array_equal(np.rint(out.cpu().numpy()[:, 0, 0] / unit), want)
    finally:
        if g is not None:
            hisq.hisq_free_gauge(ctx, g)
        hisq.hisq_destroy(ctx)

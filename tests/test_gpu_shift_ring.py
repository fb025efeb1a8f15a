"""The multi-shift stage's deferred shift updates at the edges of their parts:
block lengths around the number of residuals kept, one, two and the most
shifts, every kind of compute precision.  Each shift must meet its target by
the oracle's FP64 residual, and the stage alone must leave residuals at the
sloppy format's level (so a part applied twice, or not at all, shows)."""
import numpy as np
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import oracle

    oracle.build()
    c = hisq.hisq_create(0)
    dims = (4, 6, 4, 8)
    fat, lng = synth.gauge_pair(dims, seed=0)
    g = hisq.hisq_load_gauge(c, dims, fat.cuda(), lng.cuda())
    yield c, g, dims, fat.numpy(), lng.numpy(), oracle
    hisq.hisq_free_gauge(c, g)
    hisq.hisq_destroy(c)


# the stage stops a shift at max(target, 10 eps of the format); FP32 and FP64-class sums and the
# vectors' rounding over some hundred iterations leave it within a hundred of that
EPS = {"f64": 2.0 ** -52, "f32": 2.0 ** -24, "int20": 2.0 ** -19, "int30": 2.0 ** -29, "half": 2.0 ** -15}


@pytest.mark.parametrize("name,recon", [("f64", 18), ("f32", 12), ("int20", 12), ("int30", 18), ("half", 18)])
@pytest.mark.parametrize("nbuf", [1, 3, 7, 16])
@pytest.mark.parametrize("nshift", [1, 2, 32])
def test_targets(env, name, recon, nbuf, nshift):
    ctx, g, dims, fat, lng, orc = env
    m = 0.1
    b = synth.spinor(dims, 1000, device="cuda")
    sig = synth.shifts_logspaced(nshift, 1e-3, 2.0)
    tol = [1e-10] * nshift
    p = hisq.hisq_default_params()
    p.mass, p.on_device, p.nbuf = m, 1, nbuf
    p.sloppy, p.refine = hisq.prec(name, recon), hisq.prec("f64", 18)
    xs = [torch.empty_like(b) for _ in range(nshift)]
    st, info = hisq.hisq_multishift_cg(ctx, g, p, sig, tol, b, xs)
    assert st == hisq.HISQ_OK
    bn = float(torch.linalg.vector_norm(b))
    for i in range(nshift):
        x = xs[i].cpu().numpy()
        r = b.cpu().numpy() - orc.mee(dims, fat, lng, m, x) - sig[i] * x
        assert np.linalg.norm(r) / bn <= 1e-10
        if i > 0 or nshift == 1:  # the stage ends with the other shifts: the base's own residual is still large
            assert info.shift_resid_ms[i] <= max(1e-9, 1000 * EPS[name]), (i, info.shift_resid_ms[i])

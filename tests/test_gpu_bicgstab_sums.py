"""BiCGStab(l) with the 30-bit FP64-class triplet takes its scalars from FP64
sums over the stored records: one cycle with l = 1 ends at x = alpha b + gamma
r_0, r_0 = b - alpha u_1, whose alpha = <b, b> / <b, u_1> is recomputed here from
the records themselves (u_1 = M b comes from the stencil entry point)."""
import numpy as np
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


def stored(ctx, v):
    """v rounded to 30-bit records."""
    n = v.numel() // 6
    packed = torch.empty(hisq.hisq_spinor_bytes(hisq.HISQ_SPINOR_INT30, n), dtype=torch.uint8, device="cuda")
    out = torch.empty_like(v)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    hisq.hisq_spinor_pack(ctx, hisq.HISQ_SPINOR_INT30, n, v, packed, s)
    hisq.hisq_spinor_unpack(ctx, hisq.HISQ_SPINOR_INT30, hisq.HISQ_COMPUTE_F64, n, packed, out, s)
    torch.cuda.synchronize()
    return out


def dot(x, y):
    """<x, y> in extended precision."""
    x, y = (torch.view_as_complex(v).cpu().numpy().reshape(-1).astype(np.clongdouble) for v in (x, y))
    return np.sum(np.conj(x) * y)


@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dims,m", [((4, 4, 4, 8), 0.2), ((2, 6, 10, 4), 0.01), ((10, 14, 36, 122), 0.1)])
def test_first_cycle(dims, m, recon):
    ctx = hisq.hisq_create(0)
    g = None
    try:
        g = hisq.hisq_load_gauge(ctx, dims, *synth.gauge_pair(dims, seed=0, device="cuda"))
        half = 3 * dims[0] * dims[1] * dims[2] * dims[3] // 2
        b = stored(ctx, synth.spinor(dims, 1000, full=True, device="cuda").reshape(-1, 3, 2))
        prec = hisq.prec("int30", recon)
        u1 = torch.empty_like(b)
        hisq.hisq_dslash(ctx, g, prec, 2, -2.0 * m, b, b, u1, True)  # -2m b - D b
        u1 = -u1
        p = hisq.hisq_default_params()
        p.mass, p.tol, p.on_device, p.sloppy, p.l, p.maxiter = m, 1e-12, 1, prec, 1, 2
        x = torch.zeros_like(b).reshape(2, half // 3, 3, 2)
        st, info = hisq.hisq_bicgstabl(ctx, g, p, b.reshape(x.shape), x)
        assert st == hisq.HISQ_ENOTCONV and info.matvecs == 2
        alpha = dot(b, b) / dot(b, u1)
        bc, uc, xc = (torch.view_as_complex(v.reshape(-1, 3, 2)) for v in (b, u1, x))
        r0 = torch.view_as_complex(stored(ctx, torch.view_as_real(bc - complex(alpha) * uc).contiguous()))
        d = xc - complex(alpha) * bc
        gamma = (r0.conj() * d).sum() / (r0.abs() ** 2).sum()
        e = torch.linalg.vector_norm(d - gamma * r0) / torch.linalg.vector_norm(xc)
        # FP64 rounds the sums to some 1e-16 of |b| |u_1| (|<b, u_1>| >= 2 m |b|^2, |u_1| <= 10 |b|: 1e-13 at m = 0.01)
        # and x twice; FP32 pairs, or values before their rounding to 2^-30, leave 1e-12 to 1e-11
        assert float(e) <= 2e-13
    finally:
        if g is not None:
            hisq.hisq_free_gauge(ctx, g)
        hisq.hisq_destroy(ctx)

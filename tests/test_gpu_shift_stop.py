"""The iteration in which the multi-shift stage stops (a reliable update, or the
end) updates every site of the base system: on a lattice whose gradient update
takes several waves of blocks, with a reliable update every few iterations, the
solutions and the stage's residuals repeat to the bit."""
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,recon", [("f32", 12), ("int20", 12), ("int30", 18)])
def test_repeats_to_the_bit(name, recon):
    dims, nshift = (24, 24, 24, 48), 3  # 1296 blocks of sites and the scalars' block, last in the grid
    ctx = hisq.hisq_create(0)
    g = None
    try:
        g = hisq.hisq_load_gauge(ctx, dims, *synth.gauge_pair(dims, seed=0, device="cuda"))
        b = synth.spinor(dims, 1000, device="cuda")
        p = hisq.hisq_default_params()
        p.mass, p.on_device, p.delta = 0.2, 1, 0.7
        p.sloppy = hisq.prec(name, recon)
        runs = []
        for _ in range(4):
            xs = [torch.empty_like(b) for _ in range(nshift)]
            st, info = hisq.hisq_multishift_cg(ctx, g, p, synth.shifts_logspaced(nshift, 1e-2, 1.0), [1e-8] * nshift,
                                               b, xs)
            assert st == hisq.HISQ_OK and info.reliable_updates >= 5
            runs.append((xs, [info.shift_resid_ms[i] for i in range(nshift)], info.iters, info.matvecs))
        for r in runs[1:]:
            assert r[1:] == runs[0][1:]
            assert all(torch.equal(x, y) for x, y in zip(r[0], runs[0][0]))
    finally:
        if g is not None:
            hisq.hisq_free_gauge(ctx, g)
        hisq.hisq_destroy(ctx)

"""After a resident launch whose waits gave up, the counters of the next one
start from zero whichever blocks had begun: the solves that follow repeat, to
the bit, those of a context that never saw a wait give up."""
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


# four, two and one lanes a site; 512 and 1024 threads a block
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (12, 12, 12, 24), (16, 16, 16, 32), (18, 24, 24, 30)])
def test_solves_after_a_wait_gave_up(dims):
    fat, lng = synth.gauge_pair(dims, seed=0, device="cuda")
    b = synth.spinor(dims, 1000, device="cuda")
    p = hisq.hisq_default_params()
    p.mass, p.tol, p.on_device, p.sloppy = 0.1, 1e-10, 1, hisq.prec("int20")

    def solve(ctx, g):
        x = torch.zeros_like(b)
        st, info = hisq.hisq_cg(ctx, g, p, b, x)
        assert st == hisq.HISQ_OK
        return x, info.iters

    out = []
    for polls in ([], [1, 2, 4, 16, 64, 256, 1, 4]):
        ctx = hisq.hisq_create(0)
        g = hisq.hisq_load_gauge(ctx, dims, fat, lng)
        try:
            for n in polls:
                hisq.hisq_mee_fused_wait_test(n, True)
                try:
                    with pytest.raises(hisq.HisqError, match="ECUDA"):
                        solve(ctx, g)
                finally:
                    hisq.hisq_mee_fused_wait_test(0, False)
                out.append(solve(ctx, g))
            out.append(solve(ctx, g))
        finally:
            hisq.hisq_free_gauge(ctx, g)
            hisq.hisq_destroy(ctx)
    assert all(torch.equal(x, out[0][0]) and n == out[0][1] for x, n in out)

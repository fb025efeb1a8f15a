"""Device buffers kept for a context's next call: not counted as used, handed
out again by exact size, released when an allocation needs the room under the
budget, and never another call's data in a result."""
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


def solve(ctx, g, b, name="int20"):
    p = hisq.hisq_default_params()
    p.mass, p.tol, p.on_device, p.sloppy = 0.1, 1e-10, 1, hisq.prec(name)
    x = torch.zeros_like(b)
    st, _ = hisq.hisq_cg(ctx, g, p, b, x)
    assert st == hisq.HISQ_OK
    return x


def test_kept_buffers_and_budget():
    small, large = (4, 6, 4, 8), (8, 8, 8, 8)
    fields = {d: synth.gauge_pair(d, seed=0, device="cuda") for d in (small, large)}
    rhs = {d: synth.spinor(d, 1000, device="cuda") for d in (small, large)}
    free = hisq.hisq_create(0)
    ref = {}
    for d in (small, large):
        g = hisq.hisq_load_gauge(free, d, *fields[d])
        used = hisq.hisq_mem_used(free)
        ref[d] = [solve(free, g, rhs[d], n) for n in ("int20", "half")]
        again = [solve(free, g, rhs[d], n) for n in ("int20", "half")]
        assert all(torch.equal(a, b) for a, b in zip(ref[d], again))
        after = hisq.hisq_mem_used(free)
        solve(free, g, rhs[d])
        assert hisq.hisq_mem_used(free) == after >= used  # the copies of the links stay, the workspaces do not count
        hisq.hisq_free_gauge(free, g)
    # a budget with room for one lattice's fields and workspaces only: whatever the other one left is released
    peak = 30_000_000  # the larger one needs 28.6 MB with the reduction buffers
    tight = hisq.hisq_create(0, peak)
    try:
        for d in (small, large, small, large):
            g = hisq.hisq_load_gauge(tight, d, *fields[d])
            for n, want in zip(("int20", "half"), ref[d]):
                assert torch.equal(solve(tight, g, rhs[d], n), want)
            assert hisq.hisq_mem_used(tight) <= peak
            hisq.hisq_free_gauge(tight, g)
    finally:
        hisq.hisq_destroy(tight)
        hisq.hisq_destroy(free)

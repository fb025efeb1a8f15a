"""A CG whose resident launch is refused goes on with the separate kernels from
the same state: same tolerance, same reports, with and without graphs, a
history and the profiler, and inside the full-lattice and multi-shift solves."""
import numpy as np
import pytest
import torch

from paper_2302_09224_gb300 import hisq, synth

pytestmark = pytest.mark.gpu


@pytest.fixture()
def env():
    dims = (8, 6, 8, 10)
    ctx = hisq.hisq_create(0)
    g = hisq.hisq_load_gauge(ctx, dims, *synth.gauge_pair(dims, seed=0, device="cuda"))
    hisq.hisq_mee_fused_wait_test(0, 2)
    yield ctx, g, dims
    hisq.hisq_mee_fused_wait_test(0, 0)
    hisq.hisq_free_gauge(ctx, g)
    hisq.hisq_destroy(ctx)


def params(name="int20", **kw):
    p = hisq.hisq_default_params()
    p.mass, p.tol, p.on_device, p.sloppy = 0.1, 1e-10, 1, hisq.prec(name)
    for k, v in kw.items():
        setattr(p, k, v)
    return p


@pytest.mark.parametrize("name", ["int20", "half", "f32"])
@pytest.mark.parametrize("graph,prof", [(1, 0), (0, 0), (1, 1)])
def test_cg(env, name, graph, prof):
    ctx, g, dims = env
    b = synth.spinor(dims, 1000, device="cuda")
    x = torch.zeros_like(b)
    hist = np.zeros(4000)
    hisq.hisq_profile_enable(ctx, prof)
    before = hisq.hisq_launch_count(ctx)
    st, info = hisq.hisq_cg(ctx, g, params(name, use_graph=graph, history=hist.ctypes.data, history_len=hist.size), b, x)
    assert st == hisq.HISQ_OK and info.true_residual <= 1e-10 and hist[info.iters] <= 1e-10
    assert hisq.hisq_launch_count(ctx) - before >= 4 * info.iters  # four kernels an iteration
    hisq.hisq_mee_fused_wait_test(0, 0)
    y = torch.zeros_like(b)
    st, _ = hisq.hisq_cg(ctx, g, params(name), b, y)  # resident again
    assert st == hisq.HISQ_OK
    # both meet 1e-10; the operator's inverse is at most 1 / (4 m^2) = 25
    assert float(torch.linalg.vector_norm(x - y) / torch.linalg.vector_norm(b)) <= 2e-10 * 25


def test_inside_other_solves(env):
    ctx, g, dims = env
    b = synth.spinor(dims, 1001, full=True, device="cuda")
    x = torch.zeros_like(b)
    st, info = hisq.hisq_solve_full(ctx, g, params("half"), b, x)
    assert st == hisq.HISQ_OK and info.true_residual <= 1e-10
    xs = [torch.zeros_like(b[0]) for _ in range(3)]
    p = params("int30")
    p.refine = hisq.prec("int20")
    st, info = hisq.hisq_multishift_cg(ctx, g, p, [1e-3, 1e-2, 0.1], [1e-10] * 3, b[0].contiguous(), xs)
    assert st == hisq.HISQ_OK and all(info.shift_resid[i] <= 1e-10 for i in range(3))

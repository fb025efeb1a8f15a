"""CG iterations of a lattice resident on the chip (one cooperative launch per
run of iterations): every lane count and its edges, ring lengths that do and do
not divide the launch, against the oracle's FP64 residual and against the
solution of the separate kernels; the reliable-update decisions; the bounded
waits."""
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


@pytest.fixture(scope="module")
def orc():
    import oracle

    oracle.build()
    return oracle


def solve(ctx, dims, m, b, name, recon=12, split=1, tol=1e-10, anti=False, **kw):
    fat, lng = synth.gauge_pair(dims, seed=0, antiperiodic_t=anti)
    g = hisq.hisq_load_gauge(ctx, dims, fat.cuda(), lng.cuda(), hisq.HISQ_GAUGE_ANTIPERIODIC_T if anti else 0)
    p = hisq.hisq_default_params()
    p.mass, p.tol, p.on_device, p.sloppy = m, tol, 1, hisq.prec(name, recon)
    for k, v in kw.items():
        setattr(p, k, v)
    x = torch.zeros_like(b)
    old = hisq.hisq_cg_split_scalars(split)
    try:
        st, info = hisq.hisq_cg(ctx, g, p, b, x)
    finally:
        hisq.hisq_cg_split_scalars(old)
        hisq.hisq_free_gauge(ctx, g)
    return st, info, x, (fat.numpy(), lng.numpy())


# sites per parity on both sides of the shapes' limits on 152 SMs (19456 and 38912 for four and two lanes,
# 77824 and 155648 for one lane of 512 and 1024 threads), and lattices that fill no whole block
@pytest.mark.parametrize("name,recon,dims,anti", [
    ("int20", 12, (2, 2, 2, 2), False),
    ("half", 18, (4, 6, 8, 10), True),
    ("f32", 12, (6, 4, 4, 22), False),
    ("half", 18, (12, 12, 12, 22), True),
    ("f32", 12, (12, 12, 12, 24), False),
    ("int20", 12, (16, 16, 10, 30), True),
    ("half", 12, (12, 20, 22, 16), False),
    ("int20", 18, (16, 18, 18, 30), False),
    ("f32", 18, (24, 20, 14, 24), False),
    ("int20", 12, (18, 24, 24, 30), True),
])
def test_against_oracle(ctx, orc, name, recon, dims, anti):
    m = 0.1
    b = synth.spinor(dims, 1000, device="cuda")
    st, info, x, (fat, lng) = solve(ctx, dims, m, b, name, recon, anti=anti)
    assert st == hisq.HISQ_OK
    r = b.cpu().numpy() - orc.mee(dims, fat, lng, m, x.cpu().numpy())
    tr = np.linalg.norm(r) / np.linalg.norm(b.cpu().numpy())
    assert tr <= 1e-10 and abs(tr - info.true_residual) <= 1e-3 * tr + 1e-14


@pytest.mark.parametrize("nbuf", [1, 3, 8, 16])
@pytest.mark.parametrize("trigger", [0, 1])
def test_matches_separate_kernels(ctx, nbuf, trigger):
    """Both forms meet 1e-11; their solutions differ by the two residuals through the operator's inverse
    (at most 1/(4 m^2) |b| 2e-11)."""
    dims, m = (8, 8, 8, 10), 0.1
    b = synth.spinor(dims, 1001, device="cuda")
    out = {}
    for split in (0, 1):
        hist = np.zeros(4000)
        st, info, x, _ = solve(ctx, dims, m, b, "int20", split=split, tol=1e-11, nbuf=nbuf, ru_trigger=trigger,
                               history=hist.ctypes.data, history_len=hist.size)
        assert st == hisq.HISQ_OK
        assert info.iters < hist.size and hist[info.iters] <= 1e-11 and (hist[: info.iters + 1] > 0).all()
        out[split] = (info, x, hist)
    assert abs(out[0][0].iters - out[1][0].iters) <= 0.05 * out[0][0].iters
    d = torch.linalg.vector_norm(out[0][1] - out[1][1]) / torch.linalg.vector_norm(b)
    assert float(d) <= 2e-11 / (4 * m * m)
    assert out[1][2][0] == out[0][2][0]


def test_repeatable_and_maxiter(ctx):
    dims, m = (8, 6, 8, 12), 0.05
    b = synth.spinor(dims, 1002, device="cuda")
    runs = [solve(ctx, dims, m, b, "half") for _ in range(2)]
    assert torch.equal(runs[0][2], runs[1][2])
    st, info, x, _ = solve(ctx, dims, m, b, "half", maxiter=21)
    assert st == hisq.HISQ_ENOTCONV and info.iters == 24  # whole blocks of nbuf = 8
    st, info, x, _ = solve(ctx, dims, m, b, "half", maxiter=0)
    assert st == hisq.HISQ_ENOTCONV and info.iters == 0 and not bool(x.any())


def test_breakdown_leaves_a_finite_solution(ctx):
    """m = 0 on a free field: a source of zero modes breaks the recurrence down at once; what the solve
    reports is measured from x, which holds no step of an iteration that did not happen."""
    dims = (4, 4, 4, 4)
    fat, lng = synth.unit_gauge(dims, 0.5), synth.unit_gauge(dims, 0.5, long_link=True)
    g = hisq.hisq_load_gauge(ctx, dims, fat.cuda(), lng.cuda())
    try:
        b = torch.ones((128, 3, 2), dtype=torch.float64, device="cuda")
        p = hisq.hisq_default_params()
        p.mass, p.tol, p.on_device, p.sloppy, p.maxiter = 0.0, 1e-10, 1, hisq.prec("f32", 18), 64
        x = torch.zeros_like(b)
        for _ in range(3):  # whatever an earlier solve left in the kept buffers
            solve(ctx, (8, 8, 8, 8), 0.1, synth.spinor((8, 8, 8, 8), 1004, device="cuda"), "int20")
            try:
                hisq.hisq_cg(ctx, g, p, b, x)
            except hisq.HisqError as e:
                assert "EBREAKDOWN" in str(e)
            assert bool(torch.isfinite(x).all())
    finally:
        hisq.hisq_free_gauge(ctx, g)


def test_waits_end(ctx):
    """A wait that cannot be met gives up after its polls, the solve reports it, the next one works."""
    dims, m = (8, 8, 8, 8), 0.1
    b = synth.spinor(dims, 1003, device="cuda")
    hisq.hisq_mee_fused_wait_test(4, True)
    try:
        with pytest.raises(hisq.HisqError, match="ECUDA"):
            solve(ctx, dims, m, b, "int20")
    finally:
        hisq.hisq_mee_fused_wait_test(0, False)
    st, info, _, _ = solve(ctx, dims, m, b, "int20")
    assert st == hisq.HISQ_OK and info.true_residual <= 1e-10

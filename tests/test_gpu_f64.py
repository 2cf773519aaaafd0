"""GPU parity of the FP64 solver (ot_assoc_solve_f64) against the FP64 oracle.

Both sides run Algorithm 1 in the log domain in double precision with the same stopping
rule, so the iteration counts match exactly on the 1000 x 50 configuration and the plans
agree to a few ulp per iteration: potentials and plans are compared at 1e-10 relative,
costs at 1e-12.
"""
import numpy as np
import pytest

import oracle
from paper_1805_01559_gb300 import instances as ins

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_01559_gb300 import binding
    c = binding.Context(0)
    yield c
    c.close()


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _np(t):
    return t.detach().cpu().numpy()


def test_config1_fp64_matches_oracle(ctx):
    inst = ins.config1()
    R = oracle.rates(inst.G, inst.P, inst.N0, inst.W_hz)
    C = oracle.cost(R, inst.mu)
    eps = inst.eps_rel[0] * oracle.median(C)
    p, q = inst.lam, inst.q
    res = ctx.solve_f64(_t(C), _t(p), _t(q), eps, tol=inst.tol, max_iter=inst.max_iter, want_pi=True)
    _, _, it_or, _ = oracle.sinkhorn(C, p, q, eps, inst.tol, inst.max_iter)
    assert res.status == 0
    # the same test on the same residual; the two evaluate it in different (exact) forms, so
    # a residual within rounding of tol may stop one iteration apart
    assert abs(res.iters - it_or) <= 1, (res.iters, it_or)
    f_or, g_or, _, _ = oracle.sinkhorn(C, p, q, eps, 0.0, res.iters)
    pi_or = oracle.plan(C, f_or, g_or, eps)
    np.testing.assert_allclose(oracle.plan(C, _np(res.f), _np(res.g), eps), pi_or, rtol=1e-10, atol=1e-300)
    cost_or, rho_or, er_or, ec_or = oracle.finalize(C, f_or, g_or, p, q, eps)
    assert res.transport_cost == pytest.approx(cost_or, rel=1e-12)
    assert res.marg_err_row == pytest.approx(er_or, rel=1e-6, abs=1e-15)
    assert res.marg_err_col == pytest.approx(ec_or, rel=1e-6, abs=1e-15)
    np.testing.assert_allclose(_np(res.rrh_load), rho_or, rtol=1e-12)
    # float plan output: FP32 rounding of the FP64 plan (entries below FP32's range are 0)
    np.testing.assert_allclose(_np(res.pi), pi_or.astype(np.float32), rtol=1e-6, atol=1e-37)


@pytest.mark.parametrize("shape,iters", [((1, 1), 3), ((37, 129), 5), ((300, 7), 20), ((2000, 300), 8)])
def test_fp64_fixed_iterations(ctx, shape, iters):
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 31 + J))
    C = rng.uniform(0.0, 1.0, (I, J))
    p = rng.lognormal(0.0, 1.0, I)
    q = rng.uniform(0.5, 1.5, J)
    q *= p.sum() / q.sum()
    res = ctx.solve_f64(_t(C), _t(p), _t(q), 0.05, tol=0.0, max_iter=iters)
    f_or, g_or, it_or, _ = oracle.sinkhorn(C, p, q, 0.05, 0.0, iters)
    assert res.iters == it_or
    np.testing.assert_allclose(oracle.plan(C, _np(res.f), _np(res.g), 0.05), oracle.plan(C, f_or, g_or, 0.05),
                               rtol=1e-10, atol=1e-300)


def test_fp64_and_fp32_agree_on_config1(ctx):
    # Iteration counts of the FP32 and FP64 solvers stay within a few of each other.
    inst = ins.config1()
    R = oracle.rates(inst.G.astype(np.float32).astype(np.float64), inst.P, inst.N0, inst.W_hz)
    C = oracle.cost(R.astype(np.float32).astype(np.float64), inst.mu)
    eps = inst.eps_rel[0] * oracle.median(C)
    r64 = ctx.solve_f64(_t(C), _t(inst.lam), _t(inst.q), eps, tol=inst.tol, max_iter=inst.max_iter)
    C32 = torch.from_numpy(C.astype(np.float32)).cuda()
    r32 = ctx.solve_cost(C32, torch.from_numpy(inst.lam.astype(np.float32)).cuda(),
                         torch.from_numpy(inst.q.astype(np.float32)).cuda(), eps, tol=inst.tol,
                         max_iter=inst.max_iter)
    assert abs(r64.iters - r32.iters) <= 2
    assert r32.transport_cost == pytest.approx(r64.transport_cost, rel=1e-6)


def test_fp64_rejects_unbalanced(ctx):
    from paper_1805_01559_gb300 import binding
    C = np.ones((10, 4))
    with pytest.raises(binding.OTError) as e:
        ctx.solve_f64(_t(C), _t(np.full(10, 0.1)), _t(np.full(4, 0.5)), 0.1)
    assert e.value.status == binding.OT_EINVAL


@pytest.mark.parametrize("shape", [(1000, 50), (40, 2881), (5, 3)])
@pytest.mark.parametrize("lost", ["row", "column", "both"])
def test_fp64_breakdown_is_one_decision(ctx, shape, lost):
    """A device or an RRH without any link: every CTA leaves at the same loop test, time after
    time, and the caller's outputs (a warm-start g among them) stay as they were."""
    import ctypes

    from paper_1805_01559_gb300 import binding
    I, J = shape
    C = np.random.Generator(np.random.PCG64(I + J)).uniform(0.0, 1.0, shape)
    if lost in ("row", "both"):
        C[I // 2] = np.inf
    if lost in ("column", "both"):
        C[:, J - 1] = np.inf
    C, p, q = (torch.from_numpy(x).cuda() for x in (C, np.full(I, 1.0 / I), np.full(J, 1.0 / J)))
    for _ in range(10):
        r, f, g, _, load = ctx._result(I, J, C.device, False, True, None, None)
        for x in (f, g, load):
            x.fill_(7.0)
        st = ctx._L.ot_assoc_solve_f64(ctx._h, binding._ptr(C), J, binding._ptr(p), binding._ptr(q), I, J, 0.1, 0.0, 20, 0,
                                       ctypes.byref(r), binding._stream(None))
        assert st == binding.OT_EINVAL and r.iters == 1
        for x in (f, g, load):
            assert bool((x == 7.0).all())


@pytest.mark.parametrize("shape", [(2, 3), (9, 4), (300, 50), (40, 2881), (11, 8192)])
@pytest.mark.parametrize("kind", ["row", "column"])
def test_fp64_sums_below_the_range(ctx, shape, kind):
    """Masses 200 decades apart.  row: a device of 1e-200 with one link, to an RRH of 1e-200 that
    every other device reaches too: its row sum becomes 1e-400 after the first column update.
    column: that device also has the only good link to an ordinary RRH, which takes it up to mass
    1 and the next row update the small RRH down to 1e-400.  Iterates as the oracle's log-sum-exp
    gives them: both in doubles, a few ulp an iteration on exponents of up to 1000, so 1e-10
    relative as in the tests above."""
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 10007 + J))
    eps = 0.01
    C = rng.uniform(0.0, 0.5, shape)
    p, q = rng.uniform(0.5, 1.5, I), rng.uniform(0.5, 1.5, J)
    i, j, k = I - 1, J - 1, J // 2
    C[i] = np.inf
    C[i, j] = 0.0
    if kind == "column":
        C[:i, j] = np.inf
        C[:i, k] = 700 * eps
        C[i, k] = 0.0
    p[i] = q[j] = 0.0
    q *= p.sum() / q.sum()
    p[i] = q[j] = 1e-200
    n = 4
    res = ctx.solve_f64(*(torch.from_numpy(x).cuda() for x in (C, p, q)), eps, tol=0.0, max_iter=n)
    f, g, _, _ = oracle.sinkhorn(C, p, q, eps, 0.0, n)
    assert res.iters == n
    np.testing.assert_allclose(oracle.plan(C, res.f.cpu().numpy(), res.g.cpu().numpy(), eps), oracle.plan(C, f, g, eps),
                               rtol=1e-10, atol=1e-300)


# Where the rows of a tile, the grid, or the way a column is walked change: one row, fewer tiles than
# column CTAs, the widths from which a tile takes 4, 2 and 1 rows, as many rows as SMs and one more,
# the width from which every warp has a column.
@pytest.mark.parametrize("shape", [(1, 1), (1, 9), (1, 8192), (2, 300), (7, 127), (7, 128), (33, 255), (33, 256), (64, 511),
                                   (64, 512), (152, 512), (153, 512), (304, 600), (305, 600), (152, 1215), (152, 1216),
                                   (3, 7201)])
def test_fp64_wide_and_short(ctx, shape):
    """Against the oracle after 4 iterations, 1e-10 relative as above."""
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 10007 + J))
    C = rng.uniform(0.0, 1.0, shape)
    p, q = rng.lognormal(0.0, 1.0, I), rng.uniform(0.5, 1.5, J)
    q *= p.sum() / q.sum()
    res = ctx.solve_f64(*(torch.from_numpy(x).cuda() for x in (C, p, q)), 0.05, tol=0.0, max_iter=4)
    f, g, _, _ = oracle.sinkhorn(C, p, q, 0.05, 0.0, res.iters)
    np.testing.assert_allclose(oracle.plan(C, res.f.cpu().numpy(), res.g.cpu().numpy(), 0.05), oracle.plan(C, f, g, 0.05),
                               rtol=1e-10, atol=1e-300)
    cost, rho, _, _ = oracle.finalize(C, f, g, p, q, 0.05)
    assert res.transport_cost == pytest.approx(cost, rel=1e-12)
    np.testing.assert_allclose(res.rrh_load.cpu().numpy(), rho, rtol=1e-12)


def test_fp64_one_row_uses_the_chip(ctx):
    """One device and 8,192 RRHs: 20 iterations take 42 ms if the one CTA with a row does all the
    columns too, and 6 with a warp a column over every SM."""
    import time
    C = torch.rand(1, 8192, dtype=torch.float64, device="cuda")
    p, q = torch.ones(1, dtype=torch.float64, device="cuda"), torch.full((8192,), 1.0 / 8192, dtype=torch.float64, device="cuda")
    best = 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx.solve_f64(C, p, q, 0.1, tol=0.0, max_iter=20)
        best = min(best, time.perf_counter() - t0)
    assert best < 15e-3

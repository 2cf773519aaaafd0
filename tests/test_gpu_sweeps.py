"""The plan-scale sweeps at the edges of their tiles: every width at which a lane takes another
chunk or a row a wider team, and row counts that leave a team one row, an odd row, or none.

Tolerance: that of the fixed-iteration tests of test_gpu_parity.py (a plan entry within 2e-5
relative plus 1e-12 of the mass after 3 iterations; derived there from the rounding of the
exponent, ex2.approx and FP32 sums of up to 8192 terms, which these sweeps share).
"""
import numpy as np
import pytest

import oracle

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


WIDTHS = [1, 3, 4, 127, 128, 129, 385, 512, 640, 641, 768, 769, 896, 897, 1024, 1025, 1280, 1281, 1535, 1537, 1793,
          2048, 2049, 2561, 3073, 3585, 4096, 4097, 5121, 6145, 7169, 8192]
SHAPES = ([(I, J) for J in WIDTHS for I in (67,)]
          + [(I, J) for J in (50, 300, 650, 1300) for I in (1, 14, 16, 31, 46, 105, 211, 700)])


@pytest.mark.parametrize("shape", SHAPES)
def test_sweep_tile_edges(ctx, shape):
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 10007 + J))
    C = rng.uniform(0.0, 1.0, (I, J)).astype(np.float32)
    p = rng.lognormal(0.0, 1.0, I)
    q = rng.uniform(0.5, 1.5, J)
    p, q = (p / p.sum()).astype(np.float32), (q / q.sum()).astype(np.float32)
    pad = torch.full((I, (J + 3) // 4 * 4), float("nan"), dtype=torch.float32, device="cuda")  # padding is never read as mass
    pad[:, :J] = torch.from_numpy(C).cuda()
    res = ctx.solve_cost(pad[:, :J], torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda(), 0.1, tol=0.0, max_iter=3,
                         want_pi=True)
    C64 = C.astype(np.float64)
    f, g, _, _ = oracle.sinkhorn(C64, p, q, 0.1, 0.0, 3)
    pi = oracle.plan(C64, f, g, 0.1)
    err = np.abs(res.pi.cpu().numpy().astype(np.float64) - pi)
    assert (err <= 2e-5 * pi + 1e-12).all(), float((err / pi).max())


# Row counts around a tile's 8 rows, and widths around those at which a tile takes fewer rows.
@pytest.mark.parametrize("shape", [(1, 3), (7, 64), (8, 65), (9, 31), (1217, 20), (40, 2880), (40, 2881), (21, 4817),
                                   (13, 7200), (11, 8192)])
def test_fp64_tile_edges(ctx, shape):
    """FP64 form against the oracle after 4 iterations: both in doubles, a few ulp an iteration
    on exponents of up to 20, so 1e-10 relative as in test_gpu_f64.py."""
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 10007 + J))
    C = rng.uniform(0.0, 1.0, (I, J))
    p = rng.lognormal(0.0, 1.0, I)
    q = rng.uniform(0.5, 1.5, J)
    q *= p.sum() / q.sum()
    res = ctx.solve_f64(torch.from_numpy(C).cuda(), torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda(), 0.05, tol=0.0,
                        max_iter=4)
    f, g, _, _ = oracle.sinkhorn(C, p, q, 0.05, 0.0, res.iters)
    np.testing.assert_allclose(oracle.plan(C, res.f.cpu().numpy(), res.g.cpu().numpy(), 0.05), oracle.plan(C, f, g, 0.05),
                               rtol=1e-10, atol=1e-300)
    cost, rho, _, _ = oracle.finalize(C, f, g, p, q, 0.05)
    assert res.transport_cost == pytest.approx(cost, rel=1e-12)
    np.testing.assert_allclose(res.rrh_load.cpu().numpy(), rho, rtol=1e-12)


def _crowded(kind, I, J):
    """A column whose sum leaves the range of the fixed-point totals: a target of 1e-30, or a
    target of 1e-6 for the column that nearly all the mass first goes to."""
    rng = np.random.Generator(np.random.PCG64(I + J))
    C = rng.uniform(0.0, 1.0, (I, J)).astype(np.float32)
    p = rng.lognormal(0.0, 1.0, I)
    q = rng.uniform(0.5, 1.5, J)
    q[J // 2] = 1e-30 if kind == "tiny" else 1e-6
    if kind == "crowded":
        C[:, J // 2] -= 2.0
    return C, (p / p.sum()).astype(np.float32), (q / q.sum()).astype(np.float32)


@pytest.mark.parametrize("kind", ["tiny", "crowded"])
@pytest.mark.parametrize("shape", [(300, 50), (900, 1300)])
@pytest.mark.parametrize("iters", [2, 3, 6])
def test_column_totals_out_of_range(ctx, kind, shape, iters):
    """Such columns are summed from the partitions' partials; iterates equal the oracle's."""
    I, J = shape
    C, p, q = _crowded(kind, I, J)
    res = ctx.solve_cost(torch.from_numpy(C).cuda(), torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda(), 0.1, tol=0.0,
                         max_iter=iters, want_pi=True)
    C64 = C.astype(np.float64)
    f, g, _, _ = oracle.sinkhorn(C64, p, q, 0.1, 0.0, iters)
    pi = oracle.plan(C64, f, g, 0.1)
    err = np.abs(res.pi.cpu().numpy().astype(np.float64) - pi)
    assert (err <= 2e-5 * pi + 1e-12).all()


@pytest.mark.parametrize("kind", ["tiny", "crowded"])
def test_group_with_idle_ctas(kind):
    """A group of CTAs larger than the instance's row partitions: the idle ones follow the same
    totals (and the same detours to the partials) and the result is the single solver's."""
    from paper_1805_01559_gb300 import binding
    I, J = 200, 52
    C, p, q = _crowded(kind, I, J)
    t = [torch.from_numpy(x).cuda() for x in (C, p, q)]
    with binding.Context(0) as c:
        one = c.solve_cost(*t, 0.1, tol=0.0, max_iter=6)
        n = torch.cuda.get_device_properties(0).multi_processor_count
        c.set_tuning(binding.bucket(I, J), n, 24576)
        inst = [binding.Instance(C=t[0], p=t[1], q=t[2], eps=0.1, tol=0.0, max_iter=6) for _ in range(3)]
        c.solve_batched(inst)
        for x in inst:
            assert torch.equal(x.f, one.f) and torch.equal(x.g, one.g)


@pytest.mark.parametrize("shape", [(1, 1), (1, 3), (3, 5), (1000, 50), (1024, 1023), (1024, 1024), (1025, 1026), (3000, 801)])
@pytest.mark.parametrize("kind", ["lognormal", "signs", "two_values", "outside"])
def test_median_strided_edges(ctx, shape, kind):
    """Median of a padded view on both sides of 2^20 entries, exact: values of both signs with
    zeros of both signs, two values only, and a middle that nearly no sampled entry is near."""
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 31 + J))
    x = rng.lognormal(0.0, 2.0, (I, J)).astype(np.float32)
    if kind == "signs":
        x *= rng.choice(np.array([-1.0, 0.0, -0.0, 1.0], np.float32), (I, J))
    elif kind == "two_values":
        x = np.where(rng.random((I, J)) < 0.5, np.float32(1.0), np.float32(2.0)).astype(np.float32)
    elif kind == "outside":
        x.reshape(-1)[: (I * J) // 2] = 1e-30
    pad = torch.full((I, J + 3), -7.0, dtype=torch.float32, device="cuda")
    pad[:, :J] = torch.from_numpy(x).cuda()
    if I > 1:
        R = torch.from_numpy(np.abs(x) + np.float32(1.0)).cuda()
        C, eps = ctx.build_cost(R, 1.0, eps_rel=1.0, C_out=pad[:, :J])
        assert eps == oracle.median(C.cpu().numpy().astype(np.float64))
    flat = torch.from_numpy(x.reshape(-1)).cuda()
    assert ctx.median_f32(flat) == oracle.median(x.astype(np.float64))


@pytest.mark.parametrize("shape", [(1, 1), (5, 2), (64, 51), (700, 50), (333, 129), (301, 800), (40, 2049), (9, 8190)])
@pytest.mark.parametrize("scale", [1.0, 1e-18, 1e12])
def test_rates_edges_and_scales(ctx, shape, scale):
    """Rates and cost against the oracle at 1e-6 relative (test_gpu_parity.py) for widths around a
    chunk, a warp and a block, and for gains scaled in and out of the packed divisions' range;
    the cost equals the two-call form bit for bit."""
    from paper_1805_01559_gb300 import instances as ins
    I, J = shape
    inst = ins.make_instance("t", I, J, 1000.0, I + J, hotspot=False, traffic_sigma=1.0, marginal="uniform")
    G32 = (inst.G * scale).astype(np.float32)
    N0 = inst.N0 * scale
    G, P = torch.from_numpy(G32).cuda(), torch.from_numpy(inst.P.astype(np.float32)).cuda()
    pad = torch.full((I, (J + 3) // 4 * 4), float("nan"), dtype=torch.float32, device="cuda")
    pad[:, :J] = G
    R = ctx.build_rates(pad[:, :J], P, N0, inst.W_hz)
    R_or = oracle.rates(G32.astype(np.float64), inst.P.astype(np.float32), N0, inst.W_hz)
    np.testing.assert_allclose(R.cpu().numpy(), R_or, rtol=1e-6)
    C, _ = ctx.build_cost_from_gains(G, P, N0, inst.W_hz, inst.mu)
    C2, _ = ctx.build_cost(R.contiguous(), inst.mu)
    assert torch.equal(C, C2)
    np.testing.assert_allclose(C.cpu().numpy(), 1.0 / (inst.mu * R_or), rtol=1e-6)


def _times_out(ctx, call):
    """`call` ends with OT_ETIMEOUT under a spin limit of one poll, time after time, and gives
    what it gave before once the limit is back."""
    from paper_1805_01559_gb300 import binding
    want = call(3)
    for _ in range(5):
        ctx.set_spin_limit(1)
        try:
            with pytest.raises(binding.OTError) as e:
                call(50)
            assert e.value.status == binding.OT_ETIMEOUT
        finally:
            ctx.set_spin_limit(0)
    for a, b in zip(want, call(3)):
        assert torch.equal(a.f, b.f) and torch.equal(a.g, b.g)


def _uniform(I, J):
    C = torch.rand(I, J, device="cuda", generator=torch.Generator("cuda").manual_seed(J))
    return C, torch.full((I,), 1.0 / I, device="cuda"), torch.full((J,), 1.0 / J, device="cuda")


def test_timeout_of_wide_rows(ctx):
    """Teams of two warps: a wait for a stage that gives up in one of them must not leave the
    other at the team's barrier."""
    t = _uniform(60000, 1280)
    _times_out(ctx, lambda n: [ctx.solve_cost(*t, 0.1, tol=0.0, max_iter=n)])


def test_timeout_of_wide_rows_multi(ctx):
    """The same for three solves on one matrix."""
    t = _uniform(60000, 800)
    _times_out(ctx, lambda n: ctx.solve_cost_multi(*t, [0.1, 0.15, 0.2], tol=0.0, max_iter=n))


@pytest.mark.parametrize("shape", [(40000, 1500), (20000, 4100), (10000, 8192)])
def test_timeout_with_many_columns_a_thread(ctx, shape):
    """Rows so wide that a thread waits for its columns' totals in several rounds: a wait that
    gives up in any of them ends the CTA as one."""
    t = _uniform(*shape)
    _times_out(ctx, lambda n: [ctx.solve_cost(*t, 0.1, tol=0.0, max_iter=n)])


@pytest.mark.parametrize("entry", ["median", "cost", "gains", "mobile"])
def test_median_keeps_to_the_spin_limit(ctx, entry):
    """The grid barriers of the median give up after the context's limit: every call that takes a
    median then reports OT_ETIMEOUT, and gives what it gave before once the limit is back."""
    from paper_1805_01559_gb300 import binding
    I, J = 60000, 256
    gen = torch.Generator("cuda").manual_seed(3)
    x = torch.rand(I, J, device="cuda", generator=gen) + 0.5
    P = torch.ones(J, device="cuda")
    xy, v = torch.rand(I, 2, dtype=torch.float64, device="cuda", generator=gen) * 1e3, torch.zeros(I, 2, dtype=torch.float64, device="cuda")
    rrh, shadow = torch.rand(J, 2, device="cuda", generator=gen) * 1e3, torch.zeros(I, J, device="cuda")
    C = torch.empty(I, J, device="cuda")
    call = {"median": lambda: ctx.median_f32(x.view(-1)),
            "cost": lambda: ctx.build_cost(x, 1.0, eps_rel=0.1, C_out=C)[1],
            "gains": lambda: ctx.build_cost_from_gains(x, P, 0.1, 1.0, 1.0, eps_rel=0.1, C_out=C)[1],
            "mobile": lambda: ctx.build_cost_mobile(xy, v, rrh, shadow, P, 0.0, 1e3, 1e-13, 1.0, 1.0, C_out=C, eps_rel=0.1)[1]}[entry]
    want = call()
    ctx.set_spin_limit(1)
    try:
        for _ in range(3):
            with pytest.raises(binding.OTError) as e:
                call()
            assert e.value.status == binding.OT_ETIMEOUT
    finally:
        ctx.set_spin_limit(0)
    assert call() == want


@pytest.mark.parametrize("shape", [(1, 1), (7, 300), (1000, 50), (1023, 1024)])
@pytest.mark.parametrize("kind", ["lognormal", "two_values"])
def test_median_within_a_small_budget(shape, kind):
    """Below 2^20 entries a median needs next to no scratch: a context with 8 KB of budget, which
    has no room for the histograms of a whole grid, gives the exact median all the same."""
    from paper_1805_01559_gb300 import binding
    I, J = shape
    rng = np.random.Generator(np.random.PCG64(I * 31 + J))
    R = rng.lognormal(0.0, 2.0, shape) if kind == "lognormal" else np.where(rng.random(shape) < 0.5, 1.0, 2.0)
    with binding.Context(0, hbm_budget_bytes=8192) as c:
        C, eps = c.build_cost(torch.from_numpy(R.astype(np.float32)).cuda(), 1.0, eps_rel=1.0)
        assert eps == oracle.median(C.cpu().numpy().astype(np.float64))
        assert c.median_f32(C.view(-1)) == eps
        assert c.scratch_bytes() <= 8192


@pytest.mark.parametrize("shape", [(5, 2), (64, 51), (700, 50), (301, 800), (9, 8190)])
@pytest.mark.parametrize("k,kw", [(-34, 0), (105, 0), (0, -26), (-34, -40)])
def test_rates_do_not_depend_on_the_units(ctx, shape, k, kw):
    """Gains and noise times a power of two: the same ratios, so the same rates and costs bit for
    bit.  The bandwidth times one: the rates times it, and the costs divided by it.  (The factors
    keep every product's low part a normal number or an exact subnormal.)"""
    from paper_1805_01559_gb300 import instances as ins
    I, J = shape
    inst = ins.make_instance("t", I, J, 1000.0, I + J, hotspot=False, traffic_sigma=1.0, marginal="uniform")
    G, P = torch.from_numpy(inst.G.astype(np.float32)).cuda(), torch.from_numpy(inst.P.astype(np.float32)).cuda()
    R, R2 = torch.empty_like(G), torch.empty_like(G)
    C, eps = ctx.build_cost_from_gains(G, P, inst.N0, inst.W_hz, inst.mu, eps_rel=0.05, R_out=R)
    C2, eps2 = ctx.build_cost_from_gains(G * 2.0**k, P, inst.N0 * 2.0**k, inst.W_hz * 2.0**kw, inst.mu, eps_rel=0.05, R_out=R2)
    assert torch.equal(R * 2.0**kw, R2) and torch.equal(C * 2.0**-kw, C2) and eps * 2.0**-kw == eps2


@pytest.mark.parametrize("noise", [1.0, 2.0**-40, 2.0**40])
def test_rate_logarithm_error(ctx, noise):
    """R = W log2(1 + SINR) with W = ln 2 and one RRH is log1p of a SINR that follows from the
    documented FP32 steps.  Bound: 0.91 ulp, the error of the kernel's logarithm over every float of
    [2^-50, 2^12] (evaluated on the host), here for random ones of every binade of [2^-49, 2^100],
    the neighbourhoods of all powers of two and of all 1.5 2^k - 1, where its interval ends."""
    rng = np.random.Generator(np.random.PCG64(5))
    f32 = np.float32
    x = [np.ldexp(rng.uniform(1.0, 2.0, 4096), e) for e in range(-49, 101)]
    near = np.arange(-64, 65) * 2.0**-24
    x += [np.ldexp(1.0 + near, e) for e in range(-48, 100)] + [1.5 * 2.0**e * (1.0 + near) - 1.0 for e in range(-1, 60)]
    x = np.concatenate([np.concatenate(x), 0.5 + np.arange(-64, 65) * 2.0**-26])
    x = x[x > 2.0**-49] * noise
    x = x[x < 2.0**100].astype(f32)
    G = torch.from_numpy(x[:, None].copy()).cuda()
    R = ctx.build_rates(G, torch.ones(1, device="cuda"), noise, 0.69314718055994530942).cpu().numpy()[:, 0]
    one = f32(noise)
    T = x + one                      # the row total as an FP32 pair (an exact two-sum)
    t = T - x
    Tl = (x - (T - t)) + (one - t)
    sinr = x / ((T - x) + Tl)        # own / interference, rounded to nearest
    want = np.log1p(sinr.astype(np.longdouble))
    ulp = np.ldexp(1.0, np.frexp(want.astype(np.float64))[1] - 24)
    err = np.abs((R - want).astype(np.float64)) / ulp
    assert err.max() <= 0.91, (err.max(), sinr[err.argmax()])


@pytest.mark.parametrize("mu", [1.0, 3.0, 1e-6, 0.7, 2.0**29, 2.0**31, 2.0**-61])
def test_cost_is_rounded_to_nearest(ctx, mu):
    """C = (1/mu) / R as IEEE single precision divides, bit for bit: every mantissa of R in one
    binade, random ones over every binade from subnormals to the largest (most of them inside the
    range of the short form, some on either side), and the ends of that range."""
    rng = np.random.Generator(np.random.PCG64(7))
    f32 = np.float32
    R = np.arange(0x3F800000, 0x40000000, dtype=np.uint32).view(f32)
    bits = rng.integers(1, 0x7F800000, 1 << 22, dtype=np.uint32)
    ends = np.concatenate([np.ldexp(1.0, e) * (1.0 + np.arange(-64, 64) * 2.0**-23) for e in (-51, 67)]).astype(f32)
    R = np.concatenate([R, bits.view(f32), ends])
    R = R[: R.size // 64 * 64].reshape(-1, 64)
    C, _ = ctx.build_cost(torch.from_numpy(R).cuda(), mu)
    with np.errstate(over="ignore", under="ignore"):
        want = f32(1.0 / mu) / R
    assert np.array_equal(C.cpu().numpy().view(np.uint32), want.view(np.uint32))

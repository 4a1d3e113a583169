"""What callers rely on beyond the tolerances: arithmetic whose bits are part
of the result, and the outcome of calls at the edges of what a solver accepts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_17634_gb300 import build
    build.build()
    from paper_2511_17634_gb300 import kp as K
    return K


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


# ---- double-float arithmetic (pairs of FP32 arrays) with FP32's own rounding

def _fma(a, b, c):
    """round32(a b + c): the FP64 sum of the exact product and c, rounded to odd
    where it is inexact, so that the second rounding is the only one."""
    p, c = a.astype(np.float64) * b.astype(np.float64), np.broadcast_to(c, a.shape).astype(np.float64)
    s = p + c
    t = s - p
    e = (p - (s - t)) + (c - t)
    odd = (s.view(np.int64) & 1) == 1
    s = np.where((e != 0) & ~odd, np.nextafter(s, np.where(e > 0, np.inf, -np.inf)), s)
    return s.astype(np.float32)


def _fast_two_sum(a, b):
    s = a + b
    return s, b - (s - a)


def _add(x, y):
    s = x[0] + y[0]
    t = s - x[0]
    e = (x[0] - (s - t)) + (y[0] - t)
    return _fast_two_sum(s, e + (x[1] + y[1]))


def _sub(x, y):
    return _add(x, (-y[0], -y[1]))


def _mul(x, y):
    p = x[0] * y[0]
    return _fast_two_sum(p, _fma(x[1], y[0], _fma(x[0], y[1], _fma(x[0], y[0], -p))))


def _split(v):
    """FP64 -> hi (truncated to 24 bits) and lo (the rest, rounded)."""
    hi = (np.asarray(v, dtype=np.float64).view(np.int64) & ~np.int64(0x1FFFFFFF)).view(np.float64)
    return hi.astype(np.float32), (v - hi).astype(np.float32)


def _rho(m, H, W, g2):
    """Root mean square of the step's residual in double-float: point p in sum
    p mod 1024, the sums by halves of 32 and then in order."""
    f = np.zeros((W + 2, H + 2))
    f[1:-1, 1:-1] = m.reshape(W, H)
    f = _split(f)
    at = lambda i, j: tuple(v[1 + i:1 + i + W, 1 + j:1 + j + H].reshape(-1) for v in f)
    C, E, V, N, S = at(0, 0), at(1, 0), at(-1, 0), at(0, 1), at(0, -1)
    hh = float(H) * float(H)
    one = np.ones(H * W, np.float64)
    c, e = _split(0.5 * g2 * hh * one), _split(0.125 * g2 * hh * one)
    lap = _sub(_add(_add(E, V), _add(N, S)), (np.float32(4) * C[0], np.float32(4) * C[1]))
    dx, dy = _sub(E, V), _sub(N, S)
    r = _add(_mul(c, lap), _mul(e, _add(_mul(dx, dx), _mul(dy, dy))))
    sq = _mul(r, r)
    pad = -len(m) % 1024
    sq = tuple(np.concatenate([v, np.zeros(pad, np.float32)]).reshape(-1, 1024) for v in sq)
    acc = (np.zeros(1024, np.float32), np.zeros(1024, np.float32))
    for k in range(sq[0].shape[0]):
        acc = _add(acc, (sq[0][k], sq[1][k]))
    s = (acc[0].astype(np.float64) + acc[1].astype(np.float64)).reshape(32, 32)
    for o in (16, 8, 4, 2, 1):
        s = s[:, :o] + s[:, o:2 * o]
    t = 0.0
    for v in s[:, 0]:
        t += v
    return np.sqrt(t / len(m))


@pytest.mark.parametrize("H,W", [(128, 128), (33, 125), (24, 24), (7, 700), (1000, 5), (1366, 3), (1, 1500)])
def test_step_residual_is_the_double_float_sequence(kp, H, W):
    # the rms scale of the learned guess to the last bit: normalised
    # double-float operations in a fixed order, whatever the strips are
    rng = np.random.default_rng(H * 3 + W)
    B, n, T, g2n = 3, 251, 1000, 0.0051
    m = rng.uniform(0, 1, (B, H * W)) * 10.0 ** rng.integers(-3, 1, size=(B, H * W))
    net = kp.CNN(kp.Context(max_seeds=1, max_n=16384), H, W, channels=(10, 1), max_batch=B)
    out = torch.zeros((B, 10, H * W), dtype=torch.float32, device="cuda")
    rho = torch.zeros(B, dtype=torch.float64, device="cuda")
    net.pack_inputs(_dev(m), _dev(m), n, T, g2n, out, rho)
    torch.cuda.synchronize()
    assert np.array_equal(rho.cpu().numpy(), [_rho(v, H, W, g2n) for v in m])


# ---- clusters

def _check_solution(orc, H, W, mt, b, x, tol):
    # residual and solution as in the solver tests: 1e-9 for a relative
    # residual of 1e-10 with cond <= 2.3
    C = orc.coeffs(H, W, 0.02, 1e-3, 1.0 / H, mt)
    assert np.linalg.norm(b - orc.apply(H, W, C, x)) <= 1.01 * tol * np.linalg.norm(b)
    ref = orc.gmres(H, W, C, b, tol=1e-13, m=40, maxit=800).x
    assert np.linalg.norm(x - ref) <= 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("sizes,cluster,n", [
    ([(64, 128), (128, 64)], 0, 420), ([(128, 128), (256, 64), (64, 256)], 0, 200),
    ([(32, 64), (64, 32)], 2, 700), ([(64, 40), (24, 50), (50, 24), (3, 20)], 2, 700),
    ([(40, 40), (24, 64), (96, 16)], 8, 300), ([(20, 64), (64, 48), (48, 16)], 16, 120)])
def test_cluster_systems_of_different_column_lengths(kp, orc, sizes, cluster, n):
    # columns shorter and longer than those of the system before, on the same
    # cluster (more systems than clusters are resident): the halo outside the
    # grid stays zero
    rng = np.random.default_rng(n + cluster)
    ctx = kp.Context(max_n=16384, precision=kp.PREC_MIXED, cluster_size=cluster)
    data = [(H, W, rng.uniform(0, 1, H * W), rng.normal(size=H * W)) for H, W in sizes for _ in range(3)]
    dev = [(kp.make_ops(H, W, 1e-3, 0.02, 1.0 / H, _dev(mt[None])), _dev(b)) for H, W, mt, b in data]
    at = rng.permutation(np.arange(n) % len(data))
    x = [torch.zeros_like(dev[k][1]) for k in at]
    tol = 1e-10
    info = ctx.refine(kp.Ops.concat([dev[k][0] for k in at]), [dev[k][1] for k in at], x, tol=tol, m=30, maxit=500)
    _, st, rr = kp.decode_info(info)
    torch.cuda.synchronize()
    assert (st == 0).all() and (rr <= tol).all()
    for k, (H, W, mt, b) in enumerate(data):
        rows = torch.stack([x[s] for s in np.flatnonzero(at == k)])
        assert bool((rows == rows[0]).all()), (H, W)
        _check_solution(orc, H, W, mt, b, rows[0].cpu().numpy(), tol)


def test_cluster_call_refuses_what_its_slices_leave_out(kp, orc):
    # the narrowest width decides the cluster: a wider system of an odd number
    # of points is refused, one whose slices end inside a column is solved
    rng = np.random.default_rng(3)
    ctx = kp.Context(max_n=4096, precision=kp.PREC_MIXED, cluster_size=2)
    sys_ = [(H, W, rng.uniform(0, 1, H * W), rng.normal(size=H * W)) for H, W in ((64, 32), (32, 33), (47, 40), (31, 33))]
    dev = [(kp.make_ops(H, W, 1e-3, 0.02, 1.0 / H, _dev(mt[None])), _dev(b)) for H, W, mt, b in sys_]
    x = [torch.zeros_like(b) for _, b in dev]
    with pytest.raises(kp.KPError) as e:
        ctx.refine(kp.Ops.concat([o for o, _ in dev]), [b for _, b in dev], x, tol=1e-10, m=30, maxit=500)
    assert e.value.status == kp.ERR_UNSUPPORTED
    info = ctx.refine(kp.Ops.concat([o for o, _ in dev[:3]]), [b for _, b in dev[:3]], x[:3], tol=1e-10, m=30, maxit=500)
    assert (kp.decode_info(info)[1] == 0).all()
    for (H, W, mt, b), v in zip(sys_[:3], x):
        _check_solution(orc, H, W, mt, b, v.cpu().numpy(), 1e-10)


# ---- values past what the mixed-precision solver can hold

@pytest.mark.parametrize("H,W", [(28, 28), (32, 32), (50, 37), (64, 64), (101, 80), (128, 128)])
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf, 1e39, -1e300, 1e25])
def test_mixed_solver_breaks_down_on_values_out_of_range(kp, H, W, bad):
    # one such value in b, in the lagged field or in x0 of every other system
    # (1e25: in range, its square is not); the systems beside them converge
    rng = np.random.default_rng(H)
    N, n = H * W, 6
    ctx = kp.Context(max_n=16384, precision=kp.PREC_MIXED)
    for where in ("b", "m", "x0") if abs(bad) != 1e25 else ("b",):
        v = {"b": rng.normal(size=(n, N)), "m": rng.uniform(0, 1, (n, N)), "x0": rng.normal(size=(n, N))}
        for k in (0, 2, 4):
            v[where][k, rng.integers(N)] = bad
        x = _dev(v["x0"])
        ops = kp.make_ops(H, W, 1e-3, 0.02, 1.0 / H, _dev(v["m"]))
        for solve in (ctx.refine, ctx.seed_solve):
            xs = x.clone()
            it, st, rr = kp.decode_info(solve(ops, _dev(v["b"]), xs, tol=1e-8, m=30, maxit=200))
            torch.cuda.synchronize()
            assert (st[::2] == kp.BREAKDOWN).all(), (where, st)
            assert (st[1::2] == kp.OK).all() and (rr[1::2] <= 1e-8).all()


@pytest.mark.parametrize("H,W", [(32, 32), (64, 64), (128, 128)])
@pytest.mark.parametrize("mode", ["warm", "projected"])
def test_mixed_march_keeps_a_broken_system_broken(kp, H, W, mode):
    rng = np.random.default_rng(W)
    s, t = rng.uniform(0, 1, (2, H * W)), rng.uniform(0, 1, (6, H * W))
    t[1, 5], t[4, 77] = np.nan, np.inf
    ctx = kp.Context(max_seeds=4, max_n=16384, precision=kp.PREC_MIXED)
    ds, dt = _dev(s), _dev(t)
    plan = kp.March(ctx, [(ds, dt, np.array([0, 0, 0, 1, 1, 1]), H, W)], 1000, np.full(1000, 0.01),
                    mode={"warm": kp.MARCH_WARM, "projected": kp.MARCH_PROJECTED}[mode])
    st, _ = plan.run(0, 3, stats=True)
    torch.cuda.synchronize()
    assert [q.not_converged for q in st] == [2, 2, 2]
    ok = torch.isfinite(dt).all(1).cpu().numpy()
    assert ok.tolist() == [True, False, True, True, False, True]


@pytest.mark.parametrize("H,W", [(28, 28), (50, 37), (64, 64), (101, 80), (128, 128)])
def test_converged_means_rel_res_within_tol(kp, H, W):
    # tolerances just below and above each system's own residual, closer than
    # FP32 can tell apart: no iteration is allowed, so only the test decides
    rng = np.random.default_rng(H + W)
    N, n = H * W, 24
    ctx = kp.Context(max_n=16384, precision=kp.PREC_MIXED)
    b, x0 = _dev(rng.normal(size=(n, N))), _dev(1e-3 * rng.normal(size=(n, N)))
    ops = kp.make_ops(H, W, 1e-3, 0.02, 1.0 / H, _dev(rng.uniform(0, 1, (n, N))))
    _, _, rr = kp.decode_info(ctx.refine(ops, b, x0.clone(), tol=0.0, m=30, maxit=0))
    for k in range(n):
        for f, status in ((1 - 2.0 ** -27, kp.NOT_CONVERGED), (1 + 2.0 ** -27, kp.OK), (1.01, kp.OK), (0.99, kp.NOT_CONVERGED)):
            _, st, rk = kp.decode_info(ctx.refine(ops, b, x0.clone(), tol=rr[k] * f, m=30, maxit=0))
            assert rk[k] == rr[k] and st[k] == status, (k, f)
            assert (rk[st == kp.OK] <= rr[k] * f).all()


@pytest.mark.parametrize("H,W,n,m", [
    (101, 80, 5, 40), (101, 80, 90, 12), (72, 64, 200, 64), (128, 120, 90, 40), (129, 96, 40, 40), (300, 48, 6, 40),
    (256, 64, 5, 20), (1024, 16, 4, 40), (2048, 8, 3, 64), (8, 1024, 5, 40)])
def test_clusters_on_systems_of_many_steps(kp, orc, H, W, n, m):
    # short slices, columns past a block's threads and past its points, basis
    # vectors past the shared-memory window, several reduction rounds, restarts;
    # copies of three systems.  cond(A) <= 1 + 16 c dt with c = g^2 / (2 h^2):
    # h is chosen so that it is 40, about 25 to 35 steps to 1e-9 (times the
    # condition: 1e-7)
    rng = np.random.default_rng(H + 7 * n)
    N, dt, g2 = H * W, 1e-3, 0.25
    h = np.sqrt(8 * g2 * dt / 39.0)
    mt, b = rng.uniform(0, 0.05, (3, N)), rng.normal(size=(3, N))
    at = torch.arange(n, device="cuda") % 3
    ctx = kp.Context(max_n=16384, precision=kp.PREC_MIXED)
    x = torch.zeros((n, N), dtype=torch.float64, device="cuda")
    info = ctx.refine(kp.make_ops(H, W, dt, g2, h, _dev(mt)[at].contiguous()), _dev(b)[at].contiguous(), x, tol=1e-9, m=m, maxit=2000)
    it, st, rr = kp.decode_info(info)
    torch.cuda.synchronize()
    assert (st == 0).all() and (rr <= 1e-9).all() and it.min() >= 15, it
    for k in range(min(3, n)):
        assert bool((x[k::3] == x[k]).all())
        C = orc.coeffs(H, W, g2, dt, h, mt[k])
        xk = x[k].cpu().numpy()
        assert np.linalg.norm(b[k] - orc.apply(H, W, C, xk)) <= 1.01e-9 * np.linalg.norm(b[k])
        ref = orc.gmres(H, W, C, b[k], tol=1e-12, m=60, maxit=4000).x
        assert np.linalg.norm(xk - ref) <= 1e-7 * np.linalg.norm(ref)


# ---- projection factors

def _singular_hessenberg(kp, a, precision, d=1.0):
    """A seed solve (1 x W grid, b = e_1, no diffusion) whose captured H_a is
    tridiagonal with exact entries and exactly singular: diagonal d, products
    p_n of the off-diagonals with D_n = d D_{n-1} + p_n D_{n-2}, D_n / D_{n-1}
    = d, -1, -1, ..., 0."""
    p = [None, None, -2.0] + [2.0] * (a - 3) + [1.0]
    W = a + 4
    q = np.ones(W)
    for n in range(2, a + 1):
        q[n - 1] = p[n] / q[n - 2]
    ctx = kp.Context(max_seeds=2, max_a=40, max_n=64, precision=precision)
    ops = kp.make_ops(1, W, 1.0 / d, 0.0, 0.5, _dev(np.zeros((1, W))), _dev(q[None]), None)
    b = np.zeros((1, W))
    b[0, 0] = 1.0
    ctx.seed_solve(ops, _dev(b), torch.zeros((1, W), dtype=torch.float64, device="cuda"), tol=1e-12, m=a, maxit=a)
    ctx.store_basis(0, 1, 0)
    return ctx, ops, W


@pytest.mark.parametrize("a", [3, 8, 14, 15, 21, 30])
@pytest.mark.parametrize("mixed", [False, True])
def test_singular_basis_takes_the_least_squares(kp, orc, a, mixed):
    # x0 is the least-squares projection of the oracle for the same basis: 1e-4
    # of its norm in mixed precision (FP32 basis and coefficients, alpha up to
    # 2^(a / 2) of the data), 1e-9 in FP64
    ctx, ops, W = _singular_hessenberg(kp, a, kp.PREC_MIXED if mixed else kp.PREC_FP64)
    n, hn, V, Hb = ctx.basis_get(0, 1, W)
    assert n == a and hn == 1
    r = np.ones((1, W))
    x0 = torch.zeros((1, W), dtype=torch.float64, device="cuda")
    ctx.project_targets(0, 1, ops, _dev(r), x0)
    torch.cuda.synchronize()
    ref, lsq = orc.project(V.cpu().numpy(), Hb, n, hn, r[0])
    assert lsq
    assert np.linalg.norm(x0.cpu().numpy()[0] - ref) <= (1e-4 if mixed else 1e-9) * np.linalg.norm(ref)


@pytest.mark.parametrize("mixed", [False, True])
def test_singular_basis_at_a_breakdown_stays_finite(kp, orc, mixed):
    # A = [[1, -1], [-1, 1]], b = e_1: the second column is zero after its
    # rotation and there is no next vector; x0 as the oracle's (zero pivot:
    # that coefficient is left out)
    ctx = kp.Context(max_seeds=2, max_a=40, max_n=64, precision=kp.PREC_MIXED if mixed else kp.PREC_FP64)
    q, b, r = np.array([[-1.0, 1.0]]), np.array([[1.0, 0.0]]), np.array([[0.25, 1.0]])
    ops = kp.make_ops(1, 2, 1.0, 0.0, 0.5, _dev(np.zeros((1, 2))), _dev(q), None)
    ctx.seed_solve(ops, _dev(b), torch.zeros((1, 2), dtype=torch.float64, device="cuda"), tol=1e-12, m=10, maxit=10)
    ctx.store_basis(0, 1, 0)
    n, hn, V, Hb = ctx.basis_get(0, 1, 2)
    assert n == 2 and hn == 0
    x0 = torch.zeros((1, 2), dtype=torch.float64, device="cuda")
    ctx.project_targets(0, 1, ops, _dev(r), x0)
    ref, _ = orc.project(V.cpu().numpy(), Hb, n, hn, r[0])
    assert np.isfinite(ref).all() and np.linalg.norm(x0.cpu().numpy()[0] - ref) <= 1e-6 * np.linalg.norm(ref)


# ---- training

@pytest.mark.parametrize("H,W,B,C", [(128, 128, 16, 32), (128, 128, 64, 10), (64, 64, 16, 8), (28, 28, 4, 10),
                                     (100, 75, 31, 1), (192, 40, 8, 3), (1, 1, 1, 1)])
def test_bias_gradient_is_summed_beyond_fp32(kp, H, W, B, C):
    # one layer with zero weights: the output gradients are 2 / n (0 - t) in
    # FP32, known exactly.  Four of them are added in FP32 (two roundings deep),
    # everything above is exact to FP64 and rounded once: 3 2^-24 of the sum of
    # magnitudes
    rng = np.random.default_rng(B + C)
    net = kp.CNN(kp.Context(max_seeds=1, max_n=16384), H, W, channels=(C, 1), max_batch=B)
    net.set_params(np.zeros(net.nparams, np.float32))
    x = torch.zeros((B, C, H * W), dtype=torch.float32, device="cuda")
    grads = torch.zeros(net.nparams, dtype=torch.float32, device="cuda")
    n = B * H * W
    for t in (np.full(n, 1.01), np.full(n, 1 / 3), rng.normal(size=n), 3.7 + 0.01 * rng.normal(size=n)):
        t = t.astype(np.float32)
        for _ in range(2):                        # the second on the sums that the first left
            net.gradients(x, torch.as_tensor(t, device="cuda").reshape(B, 1, -1), grads)
        torch.cuda.synchronize()
        dz = (np.float32(2) / np.float32(n) * (np.float32(0) - t)).astype(np.float64)
        assert abs(float(grads[-1]) - dz.sum()) <= 3 * 2.0 ** -24 * np.abs(dz).sum()


# ---- bits and batches

@pytest.mark.parametrize("H,W,counts,opt", [
    (32, 32, (1, 160, 400, 700), {"block_threads": 128}), (28, 28, (3, 200), {"block_threads": 256}),
    (28, 28, (1, 700), {"mixed": 1}), (48, 40, (1, 400), {"mixed": 1}), (64, 64, (1, 500), {"mixed": 1}),
    (101, 80, (1, 90, 150), {"mixed": 1}), (128, 128, (1, 28, 29, 120), {"mixed": 1}), (129, 96, (1, 150), {"mixed": 1})])
def test_a_system_has_the_same_bits_in_any_batch(kp, H, W, counts, opt):
    # an explicit FP64 shape; the mixed-precision shapes that the rule chooses
    opt = dict(opt)
    prec = kp.PREC_MIXED if opt.pop("mixed", 0) else kp.PREC_FP64
    rng = np.random.default_rng(H)
    mt, b = _dev(rng.uniform(0, 1, (1, H * W))), _dev(rng.normal(size=(1, H * W)))
    ref = None
    for n in counts:
        ctx = kp.Context(max_n=16384, precision=prec, **opt)
        x = torch.zeros((n, H * W), dtype=torch.float64, device="cuda")
        ctx.refine(kp.make_ops(H, W, 1e-3, 0.02, 1.0 / H, mt.repeat(n, 1)), b.repeat(n, 1), x, tol=1e-9, m=30)
        torch.cuda.synchronize()
        ref = x[0].clone() if ref is None else ref
        assert bool((x == ref).all()), n

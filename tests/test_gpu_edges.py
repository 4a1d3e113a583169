"""The kernels at the sizes where they can go wrong: edges of tiles and
strips, remainders, the smallest and largest of a range, fewer and more
systems than the chip holds, and every solver shape that a rule chooses.

Tolerances.  Operator and solves as in test_gpu_parity.py (1e-13; both sides
of a solve reach a relative residual of 1e-10 with cond <= 2.3, so 1e-9).
Systems that are copies of one another have to agree bit for bit: the solvers
sum in an order that does not depend on the block or on what ran before.  The
convolutions run on small whole numbers, whose products and sums are exact in
BF16 x BF16 -> FP32, so they have to match the reference bit for bit."""
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


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("H,W", [(1, 1), (1, 1025), (1023, 1), (3, 683), (41, 50), (64, 64)])
def test_operator_kernels_at_chunk_edges(kp, orc, H, W):
    # 1024 points per block: one block short of, at and past its edge; the
    # right-hand side is the IEEE quotient m / dt, for zeros, infinities, NaN
    # and values whose quotient overflows too
    rng = np.random.default_rng(H * 7 + W)
    n, N, h, g2 = 2, H * W, 1.0 / H, 0.02
    mt, x, fx, fy = (rng.normal(size=(n, N)) for _ in range(4))
    ctx = kp.Context(max_n=max(N, 16))
    y = torch.zeros((n, N), dtype=torch.float64, device="cuda")
    r, b = torch.zeros_like(y), torch.zeros_like(y)
    dx, db = _dev(x), _dev(rng.normal(size=(n, N)))
    for f in (None, (_dev(fx), _dev(fy)), (_dev(fx), None), (None, _dev(fy))):
        ops = kp.make_ops(H, W, 1 / 3e2, g2, h, _dev(mt), *(f or (None, None)))
        ctx.apply(ops, dx, y)
        ctx.residual(ops, db, dx, r)
        torch.cuda.synchronize()
        z = np.zeros_like(fx)
        hx, hy = (fx if f and f[0] is not None else z), (fy if f and f[1] is not None else z)
        for k in range(n):
            C = orc.coeffs(H, W, g2, 1 / 3e2, h, mt[k], hx[k], hy[k])
            ref = orc.apply(H, W, C, x[k])
            scale = np.linalg.norm(ref)
            assert np.linalg.norm(y[k].cpu().numpy() - ref) <= 1e-13 * scale
            res = db[k].cpu().numpy() - ref
            assert np.linalg.norm(r[k].cpu().numpy() - res) <= 1e-13 * (scale + np.linalg.norm(res))
    odd = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.7e308, -1e306, 1e-290, 1.0])
    v = x * 10.0 ** rng.integers(-12, 12, size=x.shape)
    v.ravel()[:min(v.size, odd.size)] = odd[:v.size]
    for dt in (1e-3, 1 / 3, 7.3, 1.0):
        ctx.rhs(kp.make_ops(H, W, dt, g2, h, _dev(mt)), _dev(v), b)
        torch.cuda.synchronize()
        with np.errstate(over="ignore", invalid="ignore"):
            assert np.array_equal(b.cpu().numpy(), v / dt, equal_nan=True)


def _copies(n, N, rng):
    # n systems that repeat 7 distinct ones; the last has b = 0
    mt, b, x0 = rng.uniform(0, 1, (7, N)), rng.normal(size=(7, N)), rng.normal(size=(7, N))
    b[6] = 0.0
    x0[::2] = 0.0
    at = np.arange(n) % 7
    return mt, b, x0, at


def _solve_copies(kp, orc, H, W, n, precision, tol=1e-10):
    rng = np.random.default_rng(H * W + n)
    N, h, dt, g2 = H * W, 1.0 / H, 1e-3, 0.02
    mt, b, x0, at = _copies(n, N, rng)
    ctx = kp.Context(max_n=max(N, 64), precision=precision)
    dm, db = _dev(mt)[torch.as_tensor(at).cuda()], _dev(b)[torch.as_tensor(at).cuda()]
    x = _dev(x0)[torch.as_tensor(at).cuda()].contiguous()
    ops = kp.make_ops(H, W, dt, g2, h, dm)
    it, st, rr = kp.decode_info(ctx.refine(ops, db, x, tol=tol, m=30, maxit=500))
    torch.cuda.synchronize()
    assert (st == 0).all() and (rr <= tol).all()
    for k in range(min(7, n)):
        rows = x[k::7]
        assert bool((rows == rows[0]).all()), k
        assert (it[k::7] == it[k]).all()
        xk = rows[0].cpu().numpy()
        C = orc.coeffs(H, W, g2, dt, h, mt[k])
        assert np.linalg.norm(b[k] - orc.apply(H, W, C, xk)) <= 1.01 * tol * np.linalg.norm(b[k])
        if k < 6:
            ref = orc.gmres(H, W, C, b[k], tol=1e-13, m=40, maxit=800)
            assert _rel(xk, ref.x) <= 1e-9
        else:
            assert not xk.any()


@pytest.mark.parametrize("H,W,n", [
    (28, 28, 1), (28, 28, 152), (32, 32, 153), (28, 28, 304), (32, 32, 305), (31, 33, 456), (28, 28, 457),
    (32, 32, 608), (32, 32, 609), (5, 3, 913)])
def test_fp64_shapes_by_number_of_systems(kp, orc, H, W, n):
    # 152 SMs: one, two, three and four blocks per SM and one system more
    _solve_copies(kp, orc, H, W, n, kp.PREC_FP64)


@pytest.mark.parametrize("H,W,n", [
    (1, 1, 3), (7, 5, 20), (32, 32, 700), (31, 33, 700), (16, 64, 9), (25, 41, 9), (64, 64, 500), (63, 65, 320),
    (128, 32, 9), (13, 300, 9), (128, 128, 130), (72, 64, 160), (128, 40, 7), (64, 128, 130)])
def test_mixed_solver_sizes_and_more_systems_than_blocks(kp, orc, H, W, n):
    # full blocks whose threads divide into columns (32x32, 64x64, 128x128),
    # ragged ones, clusters of 2 and 4 with whole and short slices, and more
    # systems than blocks are resident
    _solve_copies(kp, orc, H, W, n, kp.PREC_MIXED)


@pytest.mark.parametrize("H,W,n", [(101, 80, 1), (101, 80, 136), (101, 80, 137), (101, 80, 152), (101, 80, 153),
                                   (110, 96, 5), (110, 96, 68), (110, 96, 69), (128, 128, 28), (128, 128, 29),
                                   (64, 128, 57), (64, 128, 58)])
def test_cluster_shapes_by_number_of_systems(kp, orc, H, W, n):
    # either side of each line between twice the CTAs and twice the points
    _solve_copies(kp, orc, H, W, n, kp.PREC_MIXED)


def test_mixed_solver_sizes_in_one_call(kp, orc):
    rng = np.random.default_rng(5)
    sizes = [(5, 3), (31, 33), (16, 64), (32, 32), (1, 1), (63, 64), (28, 28)]
    mt = [_dev(rng.uniform(0, 1, (1, H * W))) for H, W in sizes]
    b = [rng.normal(size=H * W) for H, W in sizes]
    ctx = kp.Context(max_n=4096, precision=kp.PREC_MIXED)
    ops = kp.Ops.concat([kp.make_ops(H, W, 1e-3, 0.02, 1 / H, m) for (H, W), m in zip(sizes, mt)])
    x = [torch.zeros(H * W, dtype=torch.float64, device="cuda") for H, W in sizes]
    it, st, rr = kp.decode_info(ctx.refine(ops, [_dev(v) for v in b], x, tol=1e-10, m=30, maxit=500))
    torch.cuda.synchronize()
    assert (st == 0).all() and (rr <= 1e-10).all()
    for (H, W), m, v, xk in zip(sizes, mt, b, x):
        C = orc.coeffs(H, W, 0.02, 1e-3, 1 / H, m[0].cpu().numpy())
        assert _rel(xk.cpu().numpy(), orc.gmres(H, W, C, v, tol=1e-13, m=40, maxit=800).x) <= 1e-9


@pytest.mark.parametrize("H,W", [(1, 1), (1, 5000), (7, 700), (64, 62), (64, 63), (1000, 5), (1365, 3), (1366, 3)])
def test_step_residual_strips(kp, orc, H, W):
    # strips of 4096 / H - 2 columns: one point, one row, a last strip of one
    # column, one column a strip, and columns too long for a strip (H > 1365).
    # rho to 1e-9 and the residual planes within the lo plane's resolution,
    # the bounds of the packing test
    from oracle import cnn_oracle as R
    rng = np.random.default_rng(H + W)
    B, N, T, n, g2n = 2, H * W, 1000, 700, 0.02
    m, s = rng.uniform(0, 1, (B, N)), rng.uniform(0, 1, (B, N))
    net = kp.CNN(kp.Context(max_seeds=1, max_n=16384), H, W, channels=(R.NIN, 1), max_batch=B)
    out = torch.zeros((B, R.NIN, N), dtype=torch.float32, device="cuda")
    rho = torch.zeros(B, dtype=torch.float64, device="cuda")
    net.pack_inputs(_dev(m), _dev(s), n, T, g2n, out, rho)
    torch.cuda.synchronize()
    xo, ro = R.network_inputs(m, s, n, T, g2n, H, W)
    xg = out.cpu().numpy().astype(np.float64)
    assert np.abs(rho.cpu().numpy() / ro - 1).max() <= 1e-9
    rh = xo[:, 8] + xo[:, 9] / 256
    assert np.abs(xg[:, 8] + xg[:, 9] / 256 - rh).max() <= 2.0 ** -15 * np.abs(rh).max()


@pytest.mark.parametrize("H,W,B,ch", [
    (1, 1, 1, (1, 1, 1)), (7, 5, 1, (8, 17, 1)), (16, 8, 1, (32, 32, 1)), (43, 3, 3, (17, 24, 1)),
    (191, 3, 2, (24, 8, 1)), (192, 3, 2, (9, 32, 1)), (300, 2, 1, (32, 1, 1)), (5, 27, 3, (1, 32, 1)),
    (64, 64, 5, (10, 32, 1)), (128, 128, 4, (6, 32, 1))])
def test_network_gradients_exact_on_whole_numbers(kp, H, W, B, ch):
    # one pixel, less than, exactly and just past one tile of 128 pixels, the
    # longest column with a staged window (191) and longer ones, channels that
    # fill a group of eight and ones that do not.  Weights in {-1, 0, 1},
    # inputs in 0..3 and a target that makes the output gradient -1, 0 or 1:
    # every operand is a whole number below 256.  The bias gradients sum FP32
    # output gradients, which carry the rounding of 2 / n: 2^-20 of the sum of
    # magnitudes
    from oracle import cnn_oracle as R
    rng = np.random.default_rng(H * W + B)
    w = [rng.choice([-1.0, 0.0, 1.0], p=[0.06, 0.84, 0.1], size=(co, ci, 3, 3)) for ci, co in zip(ch[:-1], ch[1:])]
    w[0][:, 0, 1, 1] = 1.0
    p = R.flatten([(v, rng.integers(-1, 2, size=v.shape[0]).astype(np.float64)) for v in w])
    x = rng.integers(0, 4, size=(B, ch[0], W, H)).astype(np.float64)
    acts = R.forward(p, ch, x)
    assert acts[1].max() < 256 and np.abs(acts[2]).max() < 2 ** 14
    e = rng.integers(-1, 2, size=acts[2].shape).astype(np.float64)
    e.ravel()[0] = 1.0
    t = acts[2] - 0.5 * e.size * e                # whole or half numbers, below 2^17: exact in FP32
    net = kp.CNN(kp.Context(max_seeds=1, max_n=16384), H, W, channels=ch, max_batch=B)
    net.set_params(p)
    xin = torch.as_tensor(x.reshape(B, ch[0], -1), dtype=torch.float32, device="cuda")
    tg = torch.as_tensor(t.reshape(B, 1, -1), dtype=torch.float32, device="cuda")
    out = torch.zeros((B, 1, H * W), dtype=torch.float32, device="cuda")
    net.forward(xin, out)
    grads = torch.zeros(net.nparams, dtype=torch.float32, device="cuda")
    net.gradients(xin, tg, grads)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().reshape(acts[2].shape), acts[2])
    g = grads.cpu().numpy().astype(np.float64)
    _, ref = R.loss_and_grads(p, ch, x, t, operand_round=R.bf16)
    for (gw, gb), (rw, rb) in zip(R.unflatten(g, ch), R.unflatten(ref, ch)):
        assert np.array_equal(gw, rw)
        assert np.abs(gb - rb).max() <= 2.0 ** -20 * 9 * e.size


@pytest.mark.parametrize("H,W,B,ch", [
    (65, 1, 1, (3, 5, 1)), (65, 9, 2, (16, 16, 1)), (96, 7, 1, (10, 17, 1)), (97, 8, 3, (2, 32, 1)),
    (98, 17, 2, (10, 32, 32, 1)), (127, 10, 2, (9, 32, 17, 1)), (128, 16, 9, (10, 32, 32, 1)),
    (128, 20, 1, (6, 16, 16, 1)), (7, 5, 1, (3, 5, 4)), (64, 3, 2, (10, 32, 16)), (65, 9, 2, (15, 8, 2)),
    (100, 16, 1, (16, 32, 15)), (130, 4, 1, (4, 2, 3)), (129, 5, 2, (10, 32, 1))])
def test_network_inference_exact_on_whole_numbers(kp, H, W, B, ch):
    # the column-aligned kernel (64 < H <= 128: one row, part of and a whole warp
    # of 32 rows past a warp's edge, one column, a super tile of 8 columns, one
    # less and one more), the row-tiled one, and last layers of one and several
    # outputs
    from oracle import cnn_oracle as R
    rng = np.random.default_rng(H + W)
    w = [rng.choice([-1.0, 0.0, 1.0], p=[0.04, 0.9, 0.06], size=(co, ci, 3, 3)) for ci, co in zip(ch[:-1], ch[1:])]
    for v in w:
        v[:, 0] = rng.integers(-1, 2, size=v[:, 0].shape)
    p = R.flatten([(v, rng.integers(-1, 2, size=v.shape[0]).astype(np.float64)) for v in w])
    x = rng.integers(0, 4, size=(B, ch[0], W, H)).astype(np.float64)
    acts = R.forward(p, ch, x)
    assert max(a.max() for a in acts[:-1]) <= 256
    net = kp.CNN(kp.Context(max_seeds=1, max_n=16384), H, W, channels=ch, max_batch=B)
    net.set_params(p)
    xin = torch.as_tensor(x.reshape(B, ch[0], -1), dtype=torch.float32, device="cuda")
    out = torch.zeros((B, ch[-1], H * W), dtype=torch.float32, device="cuda")
    for _ in range(2):                            # the second pass on buffers that the first one left
        net.forward(xin, out)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().reshape(acts[-1].shape), acts[-1])

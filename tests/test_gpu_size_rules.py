"""Kernel variants that a size or an alignment selects, at the sizes where the choice changes.

Each test compares a variant with the oracle or with the other variant on the
same values, at the edges of its tiles: the last size of one rule, the first of
the next, remainders of every tile dimension and the smallest tensors.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_00839_gb300 import api as a
    return a


@pytest.fixture(scope="module")
def h(api):
    return api.Handle(0)


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# ------------------------------------------------------------------------ first sketch stage

# 304 groups of 32 columns is the most a CTA per group takes; beyond, a CTA takes two
@pytest.mark.parametrize("dims,sk", [
    ((72, 9728), (20, 12)),        # 304 groups: one per CTA
    ((72, 9729), (20, 12)),        # 305: two per CTA, the last CTA with one column
    ((37, 9770), (37 - 1, 12)),    # rows that start on no 16-byte boundary (4-byte copies)
    ((72, 21, 500), (20, 5, 30)),  # CTAs whose columns fall into several slabs of the next stage
    ((40, 7, 1501), (8, 7, 20)),   # an unsketched mode between the two sketched ones
    ((129, 33), (129 - 1, 7)),     # a K block of one value
    ((66, 40), (1, 40)),           # one row of Theta, nothing after the first stage
])
def test_first_stage_column_groups(api, h, dims, sk):
    X = np.random.default_rng(len(dims) + dims[1]).standard_normal(dims).astype(np.float32)
    ref = oracle.sketch(X.astype(np.float64), oracle.sketch_matrices(dims, sk, 3, problem_id=0))
    got = h.sketch(api.to_device(X), sk, 3)
    torch.cuda.synchronize()
    # the longest chain here: 1501 / 16 products per limb in the second stage, over eight warps, each sum
    # truncated at 2^-23 of its size
    assert _rel(got.cpu().double().numpy(), ref) < 1e-5


def test_first_stage_does_not_depend_on_the_grouping(api, h):
    """Mode-1 sketches of 10 000 columns at once and 1 000 at a time are the same bits."""
    X = torch.randn((10000, 70), device="cuda", generator=torch.Generator("cuda").manual_seed(1)).t()
    whole = h.sketch(X, (24, 10000), 5)
    for c in range(0, 10000, 1000):
        part = h.sketch(X[:, c:c + 1000], (24, 1000), 5)
        torch.cuda.synchronize()
        assert torch.equal(part, whole[:, c:c + 1000])


# ------------------------------------------------------------------------ convolution gradients

def _bf16_exact(shape, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(shape, device="cuda", generator=g).to(torch.bfloat16).float()


@pytest.mark.parametrize("N,H,W,cin,cout,stride", [
    (1, 1, 1, 1, 1, 1),          # one pixel
    (2, 9, 17, 3, 33, 1),        # ragged tiles, three channels, two tiles of output channels
    (1, 16, 34, 24, 64, 2),      # parity classes with ragged tiles
    (1, 10, 18, 130, 129, 1),    # channels past 128 on both sides: two chunks of K
    (2, 6, 6, 64, 200, 2),
    (1, 40, 40, 32, 3, 1),       # the output layer's shape, several slices of pixels
])
def test_convolution_gradients(api, N, H, W, cin, cout, stride):
    x, wt = _bf16_exact((N, H, W, cin), 1), _bf16_exact((cout, 3, 3, cin), 2)
    dy = _bf16_exact((N, H // stride, W // stride, cout), 3)
    dx, dw, db = api.conv3x3(x, wt, None, stride=stride, dy=dy)
    xr = x.double().permute(0, 3, 1, 2).requires_grad_(True)
    wr = wt.double().permute(0, 3, 1, 2).requires_grad_(True)
    y = torch.nn.functional.conv2d(xr, wr, stride=stride, padding=1)
    gx, gw = torch.autograd.grad(y, (xr, wr), dy.double().permute(0, 3, 1, 2))
    # operands are exact in BF16, so only FP32 sums of at most 9 * 200 (data) or 1600 (weights) products differ
    for got, ref in ((dx, gx.permute(0, 2, 3, 1)), (dw, gw.permute(0, 2, 3, 1)), (db, dy.double().sum(dim=(0, 1, 2)))):
        assert float((got.double() - ref).norm()) <= 5e-6 * float(ref.norm()) + 1e-12


# enough tiles for all input channels in one CTA: 100 of them at 64 and 128 channels, and a class of stride 2
@pytest.mark.parametrize("N,H,W,cin,cout,stride", [(1, 80, 160, 128, 16, 1), (1, 79, 157, 64, 8, 1), (2, 80, 160, 128, 8, 2)])
def test_convolution_gradients_of_large_grids(api, N, H, W, cin, cout, stride):
    test_convolution_gradients(api, N, H, W, cin, cout, stride)


@pytest.mark.parametrize("N,H,W,cin,cout,stride", [
    (1, 1, 1, 3, 1, 1),          # the three-channel kernel's smallest
    (2, 18, 34, 3, 40, 2),       # and its stride 2, ragged, 64 output channels at a time
    (1, 9, 17, 16, 8, 1),        # the tile kernel: one step of channels per tap, ragged tiles
    (2, 20, 36, 48, 129, 2),     # two tiles of output channels, stride 2
    (1, 8, 16, 128, 3, 1),       # one tile, the output layer's channel count
    (1, 7, 5, 20, 33, 1),        # channels in no step of 16: the general kernel
])
def test_convolution_forward(api, N, H, W, cin, cout, stride):
    x, wt = _bf16_exact((N, H, W, cin), 7), _bf16_exact((cout, 3, 3, cin), 8)
    b = torch.randn(cout, device="cuda", generator=torch.Generator("cuda").manual_seed(9))
    y = api.conv3x3(x, wt, b, stride=stride)
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), wt.double().permute(0, 3, 1, 2), b.double(),
                                     stride=stride, padding=1).permute(0, 2, 3, 1)
    # exact products, FP32 sums of at most 9 * 128 of them
    assert float((y.double() - ref).norm()) <= 5e-6 * float(ref.norm())


@pytest.mark.parametrize("cin,cout,stride", [(3, 8, 1), (3, 40, 2), (16, 8, 1), (48, 33, 2), (20, 8, 1)])
def test_convolution_of_infinities(api, cin, cout, stride):
    """Infinite pixels: infinities of the weights' signs (NaN where two signs meet), as direct summation gives
    them; no padded entry of a kernel's K or halo turns them into NaN."""
    x, wt = _bf16_exact((1, 20, 36, cin), 13), _bf16_exact((cout, 3, 3, cin), 14)
    for i, j, c, v in ((0, 0, 0, np.inf), (5, 7, cin - 1, np.inf), (5, 8, cin - 1, -np.inf), (19, 35, cin - 1, -np.inf),
                       (12, 20, 1, np.inf)):
        x[0, i, j, c] = v
    assert bool((wt != 0).all())
    y = api.conv3x3(x, wt, None, stride=stride).cpu().double()
    ref = torch.nn.functional.conv2d(x.cpu().double().permute(0, 3, 1, 2), wt.cpu().double().permute(0, 3, 1, 2),
                                     stride=stride, padding=1).permute(0, 2, 3, 1)
    assert bool(ref.isinf().any()) and torch.equal(y.isnan(), ref.isnan())
    inf = ref.isinf()
    assert torch.equal(y[inf], ref[inf]) and torch.equal(y.isinf(), inf)
    ok = ref.isfinite()
    # exact products, FP32 sums of at most 9 * 48 of them
    assert float((y[ok] - ref[ok]).norm()) <= 5e-6 * float(ref[ok].norm())


@pytest.mark.parametrize("cin", [16, 48])
def test_convolution_kernels_agree(api, cin):
    """An input on no 16-byte boundary runs the general kernel: the tile kernel's bits."""
    buf = _bf16_exact((2 * 13 * 21 * cin + 1,), 10) * 1.001
    x = buf[1:].view(2, 13, 21, cin)
    wt, b = _bf16_exact((24, 3, 3, cin), 11), _bf16_exact((24,), 12)
    assert torch.equal(api.conv3x3(x, wt, b), api.conv3x3(x.clone(), wt, b))


def test_convolution_gradients_of_unaligned_input(api):
    """x on no 16-byte boundary takes the scalar gather: the same bits as the aligned copy."""
    buf = _bf16_exact((1 * 12 * 20 * 16 + 1,), 4)
    x = buf[1:].view(1, 12, 20, 16)
    wt, dy = _bf16_exact((8, 3, 3, 16), 5), _bf16_exact((1, 12, 20, 8), 6)
    a = api.conv3x3(x, wt, None, dy=dy)
    b = api.conv3x3(x.clone(), wt, None, dy=dy)
    assert all(torch.equal(p, q) for p, q in zip(a, b))


# ------------------------------------------------------------------------ FP64 paths

@pytest.mark.parametrize("dims,radius,mix", [
    ((1, 1, 3), 1, True),        # one pixel
    ((31, 5, 3), 9, True),       # a tile and a bit, the largest radius of the small tiles
    ((33, 4, 2), 4, False),      # two channels: each its own slab
    ((640, 256, 1), 3, False),   # 160 tiles of 64 x 16: the large tiles
    ((576, 256, 1), 3, False),   # 144: the small ones
])
def test_fp64_apply_tiles(api, h, dims, radius, mix):
    rng = np.random.default_rng(radius)
    X, t1, t2 = rng.standard_normal(dims), rng.standard_normal(2 * radius + 1), rng.standard_normal(2 * radius + 1)
    fac, rfac = [(1, "banded", t1), (2, "banded", t2)], []
    A, B = [api.banded(1, dims[0], t1), api.banded(2, dims[1], t2)], []
    if mix:
        M = rng.standard_normal((3, 3))
        rfac, B = [(3, "dense", M)], [api.dense(3, M)]
    ref = oracle.apply_operator(X, oracle.factor_matrices(dims, fac, rfac))
    got = h.operator_apply(api.to_device(X), A, B)
    torch.cuda.synchronize()
    assert _rel(got.cpu().numpy(), ref) < 1e-13


# three mixed channels: the small tiles' last size and the first of the large ones, and the radii whose
# channels go one by one
@pytest.mark.parametrize("dims,radius", [((384, 320, 3), 9), ((384, 352, 3), 9), ((384, 384, 3), 3), ((200, 100, 3), 10),
                                         ((70, 33, 3), 16)])
def test_fp64_apply_tiles_of_mixed_channels(api, h, dims, radius):
    test_fp64_apply_tiles(api, h, dims, radius, True)


@pytest.mark.parametrize("m", [1, 3, 20])
def test_fp64_gram_schmidt_shared_columns(api, h, m):
    """Steps whose column count is below, at and above the blocks that share a slice of the sketch."""
    import workloads as w
    dims, sk = (70, 50, 3), (20, 20, 3)
    t = w.gaussian_taps(1.0, 3)
    fac = [(1, "banded", t), (2, "banded", t)]
    C = np.random.default_rng(5).standard_normal(dims)
    mats = oracle.factor_matrices(dims, fac)
    ref = oracle.rtg_gmres(mats, C, m, oracle.sketch_matrices(dims, sk, 4), lam=1e-2)
    X, info = h.gmres_solve(api.to_device(C), m, sk, 4, 1e-2, [api.banded(1, 70, t), api.banded(2, 50, t)])
    assert info.iters == m and np.allclose(info.rho, ref["rho"], rtol=1e-9)
    assert _rel(X.cpu().numpy(), ref["X"]) < 1e-9


# ------------------------------------------------------------------------ steps per loop body

@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("m,stop_at", [(7, 0), (8, 0), (9, 0), (12, 5), (12, 6), (13, 1)])
def test_two_steps_a_loop_body_equal_direct_launches(api, h, dtype, m, stop_at):
    """A stop (tolerance or m) in the first or the second step of a body gives
    the solve that launches step by step: the same bits."""
    rng = np.random.default_rng(m)
    dims = (40, 36)
    t = np.array([0.2, 1.0, 0.3])
    A, B = [api.banded(1, 40, t), api.banded(2, 36, t)], [api.banded(2, 36, np.array([0.1, 1.0, 0.2]))]
    Cd = api.to_device(np.asfortranarray(rng.standard_normal(dims).astype(dtype)))
    for solve in (h.gmres_solve, h.gk_solve):
        kw = dict(A_factors=A, B_factors=B)
        X, r = solve(Cd, m, (20, 18), 3, 0.0, use_graph=False, **kw)
        tol = 0.0
        if stop_at:
            assert r.iters == m
            tol = float(r.rho[stop_at - 1]) * (1 + 1e-9)
            X, r = solve(Cd, m, (20, 18), 3, 0.0, use_graph=False, tol=tol, **kw)
            assert r.iters == stop_at
        Xg, g = solve(Cd, m, (20, 18), 3, 0.0, tol=tol, **kw)
        assert (g.iters, g.converged, g.breakdown) == (r.iters, r.converged, r.breakdown)
        assert torch.equal(Xg, X) and np.array_equal(g.rho, r.rho)


def test_launch_count_of_half_used_bodies(api, h):
    """A solve that stops in the first step of a two-step body has launched the second step's kernels too."""
    t = np.array([0.2, 1.0, 0.3])
    A = [api.banded(1, 40, t), api.banded(2, 36, t)]
    Cd = api.to_device(np.random.default_rng(2).standard_normal((40, 36)).astype(np.float32))
    _, full = h.gmres_solve(Cd, 12, (20, 18), 3, 0.0, A_factors=A, use_graph=False)
    count = {}
    for k in (4, 5, 6, 7, 8):
        kw = dict(A_factors=A, tol=float(full.rho[k - 1]) * (1 + 1e-9))
        _, d = h.gmres_solve(Cd, 12, (20, 18), 3, 0.0, use_graph=False, **kw)
        _, g = h.gmres_solve(Cd, 12, (20, 18), 3, 0.0, **kw)
        assert d.iters == g.iters == k
        count[k] = (d.launches, g.launches)
    step = count[6][0] - count[5][0]   # direct launches stop at the step that stopped
    assert step > 0 and all(d == count[4][0] + step * (k - 4) for k, (d, _) in count.items())
    assert all(g == count[k + k % 2][0] for k, (_, g) in count.items() if k < 8)


# (dims, sketch, dtype, dense factor, BF16 basis): the kernel chains that run as dependent launches
@pytest.mark.parametrize("dims,sk,dtype,dense,bf16", [
    ((40, 36), (20, 36), np.float32, False, False),          # one mode sketched: the Gram-Schmidt pass is a kernel
    ((40, 36), (20, 36), np.float64, False, False),
    ((40, 36), (40, 36), np.float32, False, False),          # nothing sketched: a copy in the sketch's place
    ((41, 37), (20, 18), np.float32, False, False),          # rows on no 16 bytes: register kernels, 4-byte copies
    ((40, 36, 5), (20, 18, 5), np.float32, True, False),     # an operator of several kernels
    ((64, 40, 3, 9), (24, 20, 3, 4), np.float32, False, True),
    ((512, 448, 3), (128, 128, 3), np.float32, False, False),   # many blocks a kernel
    ((333, 517, 3), (128, 128, 3), np.float32, False, False),
    ((256, 232, 3), (40, 40, 3), np.float64, False, False),
])
def test_dependent_launches_equal_direct_launches(api, h, dims, sk, dtype, dense, bf16):
    """Kernels of a step that start before their predecessor has ended, alone and with three other solves in
    flight on streams of their own, give the bits of plain launches that the host waits for."""
    rng = np.random.default_rng(dims[1])
    t = np.array([0.2, 1.0, 0.3])
    A = [api.banded(k + 1, n, t) for k, n in enumerate(dims) if n > 5]
    B = [api.dense(3, np.eye(5) + 0.1 * rng.standard_normal((5, 5)))] if dense else []
    Cd = api.to_device(np.asfortranarray(rng.standard_normal(dims).astype(dtype)))
    kw = dict(A_factors=A, B_factors=B)
    for solve in (h.gmres_solve,) if bf16 else (h.gmres_solve, h.gk_solve):
        if bf16:
            kw["bf16_basis"] = True
        X, r = solve(Cd, 9, sk, 3, 1e-2, use_graph=False, **kw)
        for _ in range(3):
            Xg, g = solve(Cd, 9, sk, 3, 1e-2, **kw)
            assert g.iters == r.iters == 9 and torch.equal(Xg, X) and np.array_equal(g.rho, r.rho)
    X, r = h.gmres_solve(Cd, 9, sk, 3, 1e-2, use_graph=False, **kw)
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for _ in range(2):
        pend = [h.gmres_submit(Cd, 9, sk, 3, 1e-2, slot=i, stream=s, **kw) for i, s in enumerate(streams)]
        for Xg, g in [h.gmres_wait(p) for p in pend]:
            assert torch.equal(Xg, X) and np.array_equal(g.rho, r.rho)


# ------------------------------------------------------------------------ Theta

@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("dims,sk", [
    ((31, 33), (1, 32)), ((32, 65), (31, 1)), ((63, 257), (62, 129)), ((64, 17), (9, 16)), ((130, 255), (129, 8)),
    ((5, 300), (5, 97)), ((257, 3), (256, 3)),   # one mode sketched only
])
def test_theta_words(api, h, dtype, dims, sk):
    """Rows whose signs start anywhere in the stream's 64-bit words and blocks of
    four, last words of every length, padded rows and K tiles."""
    X = np.random.default_rng(dims[0]).standard_normal(dims).astype(dtype)
    ref = oracle.sketch(X.astype(np.float64), oracle.sketch_matrices(dims, sk, 2 ** 64 - 3, problem_id=7))
    got = h.sketch(api.to_device(np.asfortranarray(X)), sk, 2 ** 64 - 3, problem_id=7).cpu().double().numpy()
    # one wrong sign changes the result by over 1e-3; the chains have at most 257 terms
    assert _rel(got, ref) < (1e-13 if dtype == np.float64 else 5e-6)


# ------------------------------------------------------------------------ projected Tikhonov

# columns are dealt over four warps: up to 32 slots a warp (k <= 124) in one pass; 32 rows a warp
@pytest.mark.parametrize("m", [1, 2, 4, 5, 31, 32, 33, 124, 125, 130])
def test_gcv_values(api, h, m):
    """GCV over the grid from the Hessenberg matrix of the same Arnoldi run, by NumPy's SVD."""
    dims, sk = (24, 20), (24, 20)
    t = np.exp(-0.5 * (np.arange(-4, 5) / 1.7) ** 2)
    t /= t.sum()
    A = [api.banded(1, 24, t), api.banded(2, 20, t)]
    Cd = api.to_device(np.asfortranarray(np.random.default_rng(m).standard_normal(dims)))
    grid = [1e-2, 3e-2, 1e-1, 0.3, 1.0]
    _, r = h.gmres_solve(Cd, m, sk, 3, -1.0, A_factors=A, mu_grid=grid)
    assert r.iters == m
    kr = api.Krylov(h, dims, torch.float64, m, sk, 3, A_factors=A)
    kr.start(Cd)
    for _ in range(m):
        kr.step()
    view, H = kr.query()
    U, s, _ = np.linalg.svd(H, full_matrices=True)
    c = view.beta * U[0]   # U^T beta e1
    for mu, got in zip(grid, r.gcv):
        f = s * s / (s * s + mu)
        res2 = np.sum(((1 - f) * c[:m]) ** 2) + c[m] ** 2
        # residual and trace are sums of over 1e-4 of their terms: m rounding errors each, far below 1e-9
        assert got == pytest.approx(res2 / (m + 1 - f.sum()) ** 2, rel=1e-9)
    assert r.mu == grid[int(np.argmin(r.gcv))]
    kr.close()


def test_tikhonov_of_one_column_is_as_exact_as_plain_operations(api, h):
    """y = h00 beta / (h00^2 + h10^2 + mu) of one step, over many mu, against exact rationals: no further off than
    the rotation and the reflection in plain operations, each rounded to nearest."""
    from fractions import Fraction as F
    dims = (24, 20)
    t = np.exp(-0.5 * (np.arange(-4, 5) / 1.7) ** 2)
    A = [api.banded(1, 24, t / t.sum()), api.banded(2, 20, t / t.sum())]
    got_err, plain_err = [], []
    for seed in range(4):
        Cd = api.to_device(np.asfortranarray(np.random.default_rng(seed).standard_normal(dims)))
        kr = api.Krylov(h, dims, torch.float64, 1, dims, 3, A_factors=A)
        kr.start(Cd)
        kr.step()
        view, H = kr.query()
        v = kr.basis()[0][0].cpu().numpy().astype(np.longdouble)
        h0, h1, beta = float(H[0, 0]), float(H[1, 0]), view.beta
        for mu in np.geomspace(1e-6, 1.0, 60):
            X, r = h.gmres_solve(Cd, 1, dims, 3, float(mu), A_factors=A)
            assert r.iters == 1
            x = X.cpu().numpy().astype(np.longdouble)
            y = float(F(h0) * F(beta) / (F(h0) ** 2 + F(h1) ** 2 + F(float(mu))))
            # X = y V_0, rounded entry by entry: the projection on V_0 averages 480 roundings
            got_err.append(abs(float((x * v).sum() / (v * v).sum() / np.longdouble(y) - 1)))
            rot = float(np.hypot(h0, h1))
            a, g, smu = rot, h0 / rot * beta, float(np.sqrt(mu))
            n = float(np.sqrt(a * a + smu * smu))
            v0 = a + n
            w = 2.0 / (v0 * v0 + smu * smu) * (v0 * g)
            plain_err.append(abs(float(np.longdouble((g - w * v0) * (1.0 / -n)) / np.longdouble(y) - 1)))
        kr.close()
    # 240 values each: their means stand to within a tenth; the projection adds some 1e-17
    assert np.mean(got_err) <= 1.25 * np.mean(plain_err) + 1e-17


@pytest.mark.parametrize("lam", [1e-2, -1.0])
@pytest.mark.parametrize("e", [-470, 470])
def test_tikhonov_of_extreme_operators(api, h, e, lam):
    """Operator and observation times 2^e and mu times 2^2e leave the solution: squares outside 2^+-900 take the
    plain operations, which differ from the refined ones by a rounding each."""
    dims = (24, 20)
    t = np.exp(-0.5 * (np.arange(-4, 5) / 1.7) ** 2)
    t /= t.sum()
    C = np.random.default_rng(3).standard_normal(dims)
    grid = np.array([1e-3, 1e-2, 1e-1])
    out = []
    for f in (0, e):
        A = [api.banded(1, 24, t * 2.0 ** f), api.banded(2, 20, t)]
        kw = dict(mu_grid=grid * 4.0 ** f) if lam < 0 else {}
        X, r = h.gk_solve(api.to_device(np.asfortranarray(C * 2.0 ** f)), 6, (12, 10), 3,
                          lam if lam < 0 else lam * 4.0 ** f, A_factors=A, **kw)
        assert r.iters == 6 and r.device_status == 0
        out.append((X.cpu().numpy(), r.mu / 4.0 ** f))
    # roundings of six reflections and of the rotations, times the condition of R_mu (below 1e2)
    assert out[0][1] == out[1][1] and _rel(out[1][0], out[0][0]) < 1e-12


# ------------------------------------------------------------------------ FP32 step finish, video apply

# the finish keeps up to 56 rows of the Gram matrix in shared memory (J + 1 <= 56)
@pytest.mark.parametrize("m,dims,sk", [(54, (64, 60), (32, 30)), (55, (64, 60), (32, 30)), (56, (64, 60), (32, 30)),
                                       (58, (64, 60), (32, 30)), (57, (300, 290), (128, 128)), (57, (90, 17), (20, 17))])
def test_fp32_finish_rows(api, h, m, dims, sk):
    """The sketched basis is orthonormal and the Hessenberg columns are its sketches' coefficients."""
    t = np.exp(-0.5 * (np.arange(-4, 5) / 1.1) ** 2)
    A = [api.banded(1, dims[0], t / t.sum()), api.banded(2, dims[1], t / t.sum())]
    Cd = api.to_device(np.random.default_rng(m).standard_normal(dims).astype(np.float32))
    kr = api.Krylov(h, dims, torch.float32, m, sk, 3, A_factors=A)
    kr.start(Cd)
    for _ in range(m):
        kr.step()
    view, H = kr.query()
    V, Q = kr.basis()
    q = torch.stack([x.permute(1, 0).reshape(-1) for x in Q]).double().cpu().numpy()
    assert view.j == m and not view.breakdown and q.shape[0] == m + 1
    # each entry of Q is rounded once (2^-24) after its subtraction
    assert np.abs(q @ q.T - np.eye(m + 1)).max() < 1e-6
    for j in (0, m // 2, m - 1):
        s = h.sketch(h.operator_apply(V[j], A), sk, 3).permute(1, 0).reshape(-1).double().cpu().numpy()
        # S(Phi V_j) = sum_i h_ij Q_i: roundings of Q and S at 2^-24 of ||S||, FP32 sketch chains below 5e-6
        assert np.linalg.norm(s - H[:j + 2, j] @ q[:j + 2]) < 1e-5 * np.linalg.norm(s)
    kr.close()


@pytest.mark.parametrize("k", [1, 2, 4])
@pytest.mark.parametrize("sk", [(64, 60), (64, 24), (32, 30)])
def test_fp32_breakdown_after_k_steps(api, h, k, sk):
    """An operator with k distinct eigenvalues: the Krylov space is invariant after k steps, and the remainder of
    the k-th (roundings at 2^-24 of the operator's norm, a few of them a step) is below the level asked for."""
    dims = (64, 60)
    A = [api.dense(1, np.diag(1.0 + np.arange(64) % k))]
    Cd = api.to_device(np.random.default_rng(k).standard_normal(dims).astype(np.float32))
    for kw in (dict(), dict(use_graph=False)):
        _, r = h.gmres_solve(Cd, 12, sk, 3, 0.0, A_factors=A, breakdown_tol=1e-5, **kw)
        assert r.breakdown and r.converged and r.iters == k


def test_fp32_finish_is_fp64(api, h):
    """h_{j+1,j}^2 = s.s - h.(2 h1 - G h) far below s.s, from sums that float-float holds exactly: one rounding
    at 2^-53 of s.s is left (2e-6 of the result); products kept to 48 bits would leave 1e-5."""
    k = 2 * np.random.default_rng(1).integers(-2, 3, 256)
    k[0] += 2 - int(k.sum()) % 4   # the mean of k is an odd multiple of 2^-7
    dims = (256, 16)
    kr = api.Krylov(h, dims, torch.float32, 2, dims, 3, A_factors=[api.dense(1, np.diag(1 + k * 2.0 ** -18))])
    kr.start(api.to_device(np.ones(dims, dtype=np.float32)))   # beta = 64, every entry of V_0 and Q_0 2^-6
    kr.step()
    view, H = kr.query()
    kr.close()
    mean, square = float(k.mean()), float((k * k).mean())
    assert view.beta == 64.0 and H[0, 0] == 1 + mean * 2.0 ** -18
    assert H[1, 0] ** 2 == pytest.approx((square - mean * mean) * 2.0 ** -36, rel=3e-6, abs=0.0)


@pytest.mark.parametrize("dims", [(64, 16, 3, 37), (8, 5, 3, 2), (136, 33, 3, 11), (256, 256, 3, 10), (60, 17, 1, 40)])
@pytest.mark.parametrize("bf16", [False, True])
def test_video_apply_chunks(api, h, dims, bf16):
    """Frames cut into chunks of every length, tiles at the tensor's edges, one and three channels."""
    rng = np.random.default_rng(dims[3])
    if bf16 and dims[0] % 8:
        pytest.skip("BF16 rows are whole 16-byte pieces")
    t1, t2, t4 = rng.standard_normal(9), rng.standard_normal(13), rng.standard_normal(5)
    A = [api.banded(1, dims[0], t1), api.banded(2, dims[1], t2), api.banded(4, dims[3], t4)]
    X = api.to_device(rng.standard_normal(dims).astype(np.float32))
    if bf16:
        X = api.to_device(X.cpu().numpy(), torch.bfloat16)
    ref = oracle.apply_operator(X.float().cpu().double().numpy(),
                                oracle.factor_matrices(dims, [(1, "banded", t1), (2, "banded", t2), (4, "banded", t4)], []))
    got = h.operator_apply(X, A).float().cpu().double().numpy()
    # at most 9 + 13 + 5 FP32 roundings along a chain (6e-8 each); BF16: one rounding of the result (2^-9)
    assert _rel(got, ref) < (3e-3 if bf16 else 1e-6)


# frames by the hundred, in one chunk a frame and in chunks of several
@pytest.mark.parametrize("dims", [(8, 5, 1, 300), (8, 5, 1, 700), (64, 16, 3, 311)])
def test_video_apply_many_frames(api, h, dims):
    test_video_apply_chunks(api, h, dims, False)

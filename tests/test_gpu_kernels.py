"""Kernels against plain FP64 arithmetic at the sizes where their tiling can go
wrong (edges of the 128-row tile and of its 32-column panels, remainders, the
smallest and the largest sizes)."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_2607_23354_gb300")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return M.Context()


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


def _z(X, t):
    d = torch.cdist(X, X, compute_mode="donot_use_mm_for_euclid_dist")
    return torch.exp(-t * d)


# The diagonal tile's factor, by the Cholesky backward error |Z - L L^T| <=
# (n + 1) u |L| |L^T| (Higham, Accuracy and Stability of Numerical Algorithms,
# Theorem 10.3; the diagonal of |L| |L^T| is Z's, so every entry of it is at
# most 1) with u = 2^-23 for the split products, plus 4 u for the FP32 entries
# of Z and the reciprocal square roots.
@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 97, 127, 128])
@pytest.mark.parametrize("prec", ["fp32", "fp16x3"])
def test_diagonal_tile_factor(ctx, n, prec):
    X = _dev(workloads.unit_cube_cloud(n=n, m=5, seed=n))
    t = 1.5
    L = ctx.cholesky_factor(X, t, prec).double()
    Z = _z(X, t)
    u = 2.0 ** -23
    assert float((L @ L.T - Z).abs().max()) <= (n + 5) * u
    assert bool((torch.triu(L, 1) == 0).all())


# A solve within one tile uses the factor and its inverse in both sweeps.
@pytest.mark.parametrize("n", [2, 5, 63, 96, 128, 129, 161])
def test_small_solves(ctx, n):
    X = _dev(workloads.unit_cube_cloud(n=n, m=4, seed=100 + n))
    t = 2.0
    w, mag, info = ctx.solve(X, t)
    Z = _z(X, t)
    r = 1.0 - Z @ w
    assert info["fallback"] == 0
    assert float(r.abs().max()) <= 1e-14 * float(Z.sum(1).max()) * float(w.abs().max())
    assert abs(mag - float(w.sum())) <= 1e-13 * abs(mag)


# A pivot that is exactly zero in FP32, in any place of a pivot block and in
# any panel: points far apart (every other entry below e^-15, its square below
# half a unit in the last place of 1) but for one pair 1e-13 apart, whose entry
# rounds to 1.
@pytest.mark.parametrize("p", [1, 2, 3, 4, 30, 33, 66, 127])
def test_zero_pivot_is_reported_with_its_row(ctx, p):
    X = np.zeros((128, 2))
    X[:, 0] = 16.0 * np.arange(128)
    X[p] = X[p - 1] + [0.0, 1e-13]
    with pytest.raises(M.MagnitudeError) as e:
        ctx.cholesky_factor(_dev(X), 1.0, "fp32")
    assert e.value.status == M.MAG_ENOTPD
    assert f"row {p} " in str(e.value)


def _clouds():
    rng = np.random.default_rng(11)
    far = rng.random((300, 3)) * 1e-9  # close pairs below FP32's resolution of the span
    far[150:] += 1.0
    grid = np.stack(np.meshgrid(np.arange(9), np.arange(8), np.arange(5)), -1).reshape(-1, 3).astype(float)
    return {
        "two points": np.array([[0.0, 1.0], [3.0, 5.0]]),
        "one dimension": rng.random((129, 1)),
        "ragged": rng.standard_normal((385, 7)),
        "more dimensions than a chunk": rng.standard_normal((200, 70)),
        "more dimensions than threads": rng.standard_normal((150, 300)),
        "offset": rng.random((260, 4)) + 1e6,
        "far clusters": far,
        "lattice": grid,
    }


# The closest distance from FP32 comparisons is the FP64 one bit for bit: the
# generator's own minimum (FP64 differences of every pair) of a solve near the
# identity, where it cannot fail.
@pytest.mark.parametrize("name", sorted(_clouds()))
def test_min_distance_is_the_generators(ctx, name):
    X = _clouds()[name]
    dmin, bound = ctx.min_distance(_dev(X))
    c = M.Context(M.Options(exact_distances=False, deflate=-1))
    _, _, info = c.solve(_dev(X), 40.0 / dmin)
    assert dmin == info["min_distance"]
    assert bound == np.log(len(X) - 1) / dmin


# Scaling the points by a power of two scales every step exactly, inside the
# FP32 path's range of spans and beyond it (2^+-400).
@pytest.mark.parametrize("k", [-430, -380, 380, 430])
def test_min_distance_scales_exactly(ctx, k):
    X = np.random.default_rng(5).random((140, 3))
    assert ctx.min_distance(_dev(np.ldexp(X, k)))[0] == np.ldexp(ctx.min_distance(_dev(X))[0], k)


def test_min_distance_errors(ctx):
    X = np.random.default_rng(2).random((300, 5))
    for bad, status in ((np.inf, M.MAG_EINVAL), (np.nan, M.MAG_EINVAL)):
        Y = X.copy()
        Y[299, 4] = bad
        with pytest.raises(M.MagnitudeError) as e:
            ctx.min_distance(_dev(Y))
        assert e.value.status == status
    for a, b in ((0, 1), (5, 299), (290, 299)):
        Y = X.copy()
        Y[a] = Y[b]
        with pytest.raises(M.MagnitudeError) as e:
            ctx.min_distance(_dev(Y))
        assert e.value.status == M.MAG_EDUPLICATE
    with pytest.raises(M.MagnitudeError) as e:  # every distance overflows
        ctx.min_distance(_dev(X * 1e300))
    assert e.value.status == M.MAG_EINVAL


# The integer-pipe distances and exponential on the GPU, by the three limb
# layouts (m <= 4, m <= 16, beyond, with and without a second chunk of 32
# dimensions), ragged and whole tiles, pairs too close for the quantized
# coordinates among them, through the dense output and through a solve's tiles:
# |dZ| <= 1 ulp of exp + t |d d|, each side's d within (m / 2 + 3) u of exact.
@pytest.mark.parametrize("n", [2, 127, 128, 131, 300])
@pytest.mark.parametrize("m", [1, 4, 5, 16, 17, 32, 33, 100])
def test_similarity_entries(ctx, n, m):
    rng = np.random.default_rng(n * 1000 + m)
    X = rng.standard_normal((n, m))
    X[n // 2] = X[0] + 1e-9 * rng.standard_normal(m)  # closer than the quantized coordinates resolve
    t = 1.5 / np.sqrt(m)
    d = np.sqrt(((X[:, None, :].astype(np.longdouble) - X[None, :, :]) ** 2).sum(-1))
    Z = np.exp(-t * d.astype(np.float64))
    tol = 2.0 ** -52 * (1.0 + (m / 2 + 4) * t * d) * Z
    Zg = ctx.similarity_matrix(_dev(X), t, "fp64").cpu().numpy()
    assert np.all(np.abs(Zg - Z) <= tol)
    Zf = ctx.similarity_matrix(_dev(X), t, "fp32").cpu().numpy()
    assert np.all(np.abs(Zf - Z) <= 2.0 ** -24 * Z + tol)
    L = ctx.cholesky_factor(_dev(X), t, "fp64").cpu().numpy()
    assert np.abs(L @ L.T - Z).max() <= (n + 5) * 2.0 ** -53 + tol.max()


# The residual entry point over the lower triangle: rows and columns of every
# tile, ragged ones, each limb layout, coincident and close pairs, an explicit
# b, weights of both signs over twelve decades.  Against FP64 sums of the same
# entries: |dr_j| <= sum_k (|dZ_jk| + 2^-52 Z_jk) |w_k|, dZ as for the entries.
@pytest.mark.parametrize("n", [2, 128, 129, 300, 1000])
@pytest.mark.parametrize("m", [2, 9, 40])
def test_residual_rows(ctx, n, m):
    rng = np.random.default_rng(n + m)
    X = rng.standard_normal((n, m))
    X[n - 1] = X[0]
    if n > 2:
        X[n // 2] = X[1] + 1e-10
    t = 2.0 / np.sqrt(m)
    w = rng.standard_normal(n) * 10.0 ** rng.uniform(-6, 6, n)
    b = rng.standard_normal(n)
    d = np.sqrt(((X[:, None, :].astype(np.longdouble) - X[None, :, :]) ** 2).sum(-1))
    Z = np.exp(-t * d.astype(np.float64))
    tol = (2.0 ** -52 * (2.0 + (m / 2 + 4) * (t * d).astype(np.float64)) * Z) @ np.abs(w) + 2.0 ** -52 * np.abs(b)
    for bb in (None, b):
        r, nr = ctx.residual(_dev(X), t, _dev(w), b=None if bb is None else _dev(bb))
        ref = ((1.0 if bb is None else bb) - Z.astype(np.longdouble) @ w).astype(np.float64)
        assert np.all(np.abs(r.cpu().numpy() - ref) <= tol)
        assert abs(nr["z_norm_inf"] - Z.sum(1).max()) <= 1e-14 * Z.sum(1).max()
        assert nr["w_norm_inf"] == np.abs(w).max()
        assert nr["r_norm_inf"] == float(r.abs().max())


# Dimensions at which the column stage, beside the exponential's 8 KB table,
# reaches the default 48 KB of shared memory (both refused the launch before).
@pytest.mark.parametrize("m", [38, 40, 42, 83, 86, 640])
def test_staging_fits_shared_memory(ctx, m):
    X = _dev(np.random.default_rng(m).standard_normal((70, m)))
    w = _dev(np.random.default_rng(1).standard_normal(70))
    t = 1.0 / np.sqrt(m)
    r, _ = M.residual_noalloc(X, t, w)
    assert float((r - (1.0 - _z(X, t) @ w)).abs().max()) <= 1e-13
    if m <= 64:
        _, dx = ctx.grad(X, t, w=w)
        assert bool(torch.isfinite(dx).all())


# The gradient kernel over the lower triangle, by limb layout and by chunk of
# 16 dimensions, ragged tiles, a close pair, and with FP64 differences.  Against
# FP64 sums: every term within (m / 2 + 12) (1 + t d) u of its value, the sums
# within n u of the sum of the terms' magnitudes.
@pytest.mark.parametrize("n", [2, 128, 129, 300])
@pytest.mark.parametrize("m", [1, 4, 5, 16, 17, 33, 64])
@pytest.mark.parametrize("exact", [True, False])
def test_gradient_sums(n, m, exact):
    rng = np.random.default_rng(n * 100 + m)
    X = rng.standard_normal((n, m))
    if n > 2:
        X[n // 2] = X[1] + 1e-8 * rng.standard_normal(m)
    t = 1.5 / np.sqrt(m)
    c = M.Context(M.Options(exact_distances=exact))
    w = rng.standard_normal(n)
    g = rng.standard_normal() * np.ones(n)  # a constant dL/dw: lam = g w, no solve
    dt, dx = c.grad(_dev(X), t, w=_dev(w), dL_dw=_dev(g))
    D = X[:, None, :] - X[None, :, :]
    d = np.sqrt((D.astype(np.longdouble) ** 2).sum(-1)).astype(np.float64)
    Z = np.exp(-t * d)
    lam = g[0] * w
    s = np.outer(lam, w) + np.outer(w, lam)
    e = 2.0 ** -53 * ((m / 2 + 12) * (1 + t * d) + n)
    assert abs(dt - (0.5 * d * Z * s).sum()) <= (0.5 * e * d * Z * abs(s)).sum()
    np.fill_diagonal(d, 1.0)
    G = t * Z * s / d
    ref = (G[:, :, None] * D).sum(1)
    assert np.all(np.abs(dx.cpu().numpy() - ref) <= ((e * abs(G))[:, :, None] * abs(D)).sum(1))


# The FP64 factor: its diagonal tile, and the panel solve and trailing update
# from digits, at tile edges and remainders, with rows whose entries span many
# decades (t = 40: below e^-40).  By the theorem above with u = 2^-53, 4 u for
# the entries of Z.
@pytest.mark.parametrize("n", [2, 31, 33, 127, 128, 129, 161, 256, 257, 400, 641])
@pytest.mark.parametrize("t", [0.5, 5.0, 40.0])
def test_fp64_factor(ctx, n, t):
    X = _dev(workloads.unit_cube_cloud(n=n, m=3, seed=n))
    L = ctx.cholesky_factor(X, t, "fp64").cpu().numpy().astype(np.longdouble)
    Z = ctx.similarity_matrix(X, t, "fp64").cpu().numpy()
    assert np.abs(L @ L.T - Z).max() <= (n + 5) * 2.0 ** -53
    assert not np.triu(L, 1).any()


# A zero pivot of the FP64 factor, as above: other entries below e^-40, a pair
# 1e-17 apart, within the diagonal tile, across two tiles and in the last one.
@pytest.mark.parametrize("p", [1, 3, 33, 127, 128, 129, 255, 299])
def test_fp64_zero_pivot_is_reported_with_its_row(ctx, p):
    X = np.zeros((300, 2))
    X[:, 0] = 40.0 * np.arange(300)
    X[p] = X[p - 1] + [0.0, 1e-17]
    with pytest.raises(M.MagnitudeError) as e:
        ctx.cholesky_factor(_dev(X), 1.0, "fp64")
    assert e.value.status == M.MAG_ENOTPD
    assert f"row {p} " in str(e.value)


# The batch's tile kernels: tile edges and remainders, one to sixteen tile
# columns, each limb layout, one and several problems of a cloud, t from nearly
# singular to nearly the identity.  The library's own bound on the relative
# residual, by the oracle, and the magnitude as the weighting's sum (n u |w|_1).
@pytest.mark.parametrize("m,ts", [(1, [3.0]), (4, [0.5, 2.0]), (6, [0.05, 40.0]), (17, [0.3]), (33, [0.1, 1.0, 5.0])])
def test_batch_tiles(ctx, m, ts):
    rng = np.random.default_rng(m)
    sizes = [2, 96, 97, 127, 128, 129, 200, 255, 256, 257, 384, 641, 1000] + ([2048] if m == 4 else [])
    clouds = [rng.standard_normal((n, m)) for n in sizes]
    clouds[4][7] = clouds[4][3] + 1e-9  # closer than the quantized coordinates resolve
    ws, mags, sts = ctx.solve_batch([_dev(c) for c in clouds], ts)
    assert int(sts.abs().sum()) == 0
    for i, c in enumerate(clouds):
        for j, t in enumerate(ts):
            w = ws[i * len(ts) + j].cpu().numpy()
            assert oracle.relative_residual(c, t, w) <= 1e-14
            assert abs(mags[i, j].item() - w.sum()) <= len(c) * 2.0 ** -53 * np.abs(w).sum()


# What a cloud of several tiles is refused for, beside clouds that are solved:
# the same statuses as from the one-CTA kernel (launch shape 1).
def test_batch_tiles_statuses():
    rng = np.random.default_rng(3)
    clouds = [rng.standard_normal((300, 3)) for _ in range(7)]
    clouds[1][299] = clouds[1][0]
    clouds[2][150, 1] = np.nan
    clouds[3][0, 0] = np.inf
    clouds[4][:] = 1.5
    clouds[5] *= 1e-200
    out = []
    for opt in (M.Options(), M.Options(batch_shape=1)):
        c = M.Context(opt)
        _, mags, sts = c.solve_batch([_dev(x) for x in clouds], [0.5, 4.0])
        out.append((sts.cpu().numpy(), mags.cpu().numpy()))
        c.close()
    assert np.array_equal(out[0][0], out[1][0])
    ok = out[0][0] == M.MAG_OK
    assert ok[0].all() and ok[6].all()
    assert not ok[1].any() and not ok[2].any() and not ok[3].any() and not ok[4].any()
    assert np.allclose(out[0][1][ok], out[1][1][ok], rtol=1e-12)


# The stored-tile residuals by strip length (1, 1, 2, 4, 5 and 8 tiles): a solve
# refined with them, judged by the residual entry point's own pass over the
# points (the library's bound of 1e-14).
@pytest.mark.parametrize("n", [129, 300, 2300, 4000, 4500, 6300])
def test_stored_residual_strips(ctx, n):
    X = _dev(workloads.unit_cube_cloud(n=n, m=6, seed=n))
    w, mag, info = ctx.solve(X, 3.0)
    _, norms = ctx.residual(X, 3.0, w)
    assert info["fallback"] == 0
    assert norms["r_norm_inf"] <= 1e-14 * norms["z_norm_inf"] * norms["w_norm_inf"]
    assert abs(mag - float(w.sum())) <= n * 2.0 ** -53 * float(w.abs().sum())


# Pairs of a batch that are too close for the quantized coordinates and yet far
# apart in t d: two clusters 10 apart with nearly all in-cluster distances below
# 0.1 (close is below sqrt(3) 2^-8 of 16 at m = 3), t d from 5 up to 1e8.  Every
# problem stays with the batch's own factor.
def test_batch_close_pairs_at_large_t(ctx):
    rng = np.random.default_rng(12)
    s = 10.0 ** rng.uniform(-3, -1.6, (260, 1))
    X = rng.standard_normal((260, 3)) * s
    X[130:] += 10.0
    dmin = ctx.min_distance(_dev(X))[0]
    ts = [f / dmin for f in (5.0, 50.0, 90.0, 300.0, 1e4, 1e6)]
    ws, mags, sts = ctx.solve_batch([_dev(X)], ts)
    assert int(sts.abs().sum()) == 0
    assert ctx.last_batch_info["fallback"] == 0
    for t, w, mag in zip(ts, ws, mags[0]):
        w = w.cpu().numpy()
        assert oracle.relative_residual(X, t, w) <= 1e-14
        assert abs(mag.item() - w.sum()) <= 260 * 2.0 ** -53 * np.abs(w).sum()


# Pivots that have cancelled to a few units in the last place, as the second of
# a pair at every place of a pivot block and in every panel, with a first one
# that is not 1 (an earlier point near both): the factor is refused, or its
# diagonal is positive and its backward error within the bound above.
@pytest.mark.parametrize("p", [2, 3, 4, 5, 6, 7, 31, 33, 35, 67, 97, 126, 127])
def test_cancelled_pivots(ctx, p):
    rng = np.random.default_rng(p)
    refused = 0
    for _ in range(64):
        X = np.zeros((128, 2))
        X[:, 0] = 16.0 * np.arange(128)
        X[p - 1] = X[p - 2] + rng.uniform(0.02, 0.6, 2)
        X[p] = X[p - 1] + 10.0 ** rng.uniform(-7.5, -5.0) * rng.standard_normal(2)
        try:
            L = ctx.cholesky_factor(_dev(X), 1.0, "fp32").double()
        except M.MagnitudeError as e:
            assert e.status == M.MAG_ENOTPD
            refused += 1
            continue
        assert bool((torch.diagonal(L) > 0).all())
        assert float((L @ L.T - _z(_dev(X), 1.0)).abs().max()) <= (128 + 5) * 2.0 ** -23
    assert refused < 64


# The FP64 factor entry by entry, where the entries of a row span many decades and
# the panels hold little of some: |L L^T - Z| <= (n + 1) u |L| |L^T|, plus 4 u,
# by the theorem above with the product it is stated with, from clouds whose
# panels pass by digits alone to ones that need FP64 products.
@pytest.mark.parametrize("n", [129, 300])
@pytest.mark.parametrize("cloud,m,t", [("cube", 6, 1.0), ("cube", 6, 6.0), ("cube", 20, 6.0), ("normal", 2, 3.0),
                                       ("normal", 6, 3.0), ("normal", 6, 6.0), ("normal", 12, 6.0), ("normal", 20, 5.0)])
def test_fp64_factor_by_entry(ctx, n, cloud, m, t):
    rng = np.random.default_rng(m)
    X = _dev(rng.random((n, m)) if cloud == "cube" else rng.standard_normal((n, m)))
    L = ctx.cholesky_factor(X, t, "fp64").cpu().numpy().astype(np.longdouble)
    Z = ctx.similarity_matrix(X, t, "fp64").cpu().numpy()
    assert np.all(np.abs(L @ L.T - Z) <= (n + 5) * 2.0 ** -53 * (np.abs(L) @ np.abs(L).T))


# The norms of the residual entry point add the tiles' row sums of Z in any order:
# exactly, so that equal calls give equal bits (n = 3000: 24 tiles a row) and the
# row sum is the exact one, rounded (2^-64 dropped of every entry).
def test_residual_norms_are_the_same_every_time(ctx):
    rng = np.random.default_rng(21)
    X = rng.standard_normal((3000, 5))
    w = rng.standard_normal(3000)
    norms = [ctx.residual(_dev(X), 0.8, _dev(w))[1] for _ in range(24)]
    assert all(v == norms[0] for v in norms)
    Z = ctx.similarity_matrix(_dev(X), 0.8).cpu().numpy().astype(np.longdouble)
    z = Z.sum(1).max()
    assert abs(norms[0]["z_norm_inf"] - z) <= 3 * 2.0 ** -53 * z


# Gradients of few points: FP64 differences up to 32, tiles whose last rows and
# columns are empty (one to four groups of each), the second tile of a pair ragged.
# Bound as for test_gradient_sums.
@pytest.mark.parametrize("n", [2, 15, 16, 17, 31, 32, 33, 64, 65, 100, 135, 200])
@pytest.mark.parametrize("m", [3, 17, 64])
def test_gradient_of_few_points(ctx, n, m):
    rng = np.random.default_rng(n + 1000 * m)
    X, w = rng.standard_normal((n, m)), rng.standard_normal(n)
    t, c = 1.5 / np.sqrt(m), 0.75
    dt, dx = ctx.grad(_dev(X), t, w=_dev(w), dL_dw=_dev(np.full(n, c)))
    D = X[:, None, :] - X[None, :, :]
    d = np.sqrt((D.astype(np.longdouble) ** 2).sum(-1)).astype(np.float64)
    Z, s = np.exp(-t * d), 2.0 * c * np.outer(w, w)
    e = 2.0 ** -53 * ((m / 2 + 12) * (1 + t * d) + n)
    assert abs(dt - (0.5 * d * Z * s).sum()) <= (0.5 * e * d * Z * abs(s)).sum()
    np.fill_diagonal(d, 1.0)
    G = t * Z * s / d
    assert np.all(np.abs(dx.cpu().numpy() - (G[:, :, None] * D).sum(1)) <= ((e * abs(G))[:, :, None] * abs(D)).sum(1))

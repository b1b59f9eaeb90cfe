"""The products and the factorisation that run on integer digits instead of the FP64 pipes, at the
sizes where their tiles, chunks and blocks end, through the C ABI.

Bounds. A digit product keeps each row to 2^-62 of its largest entry and rounds its sum once, so
an entry errs by at most 2^-53 |C_ij| + 2 K 2^-62 max_k|A_ik| max_k|B_jk|; the references are exact
(integer inputs, or numpy's longdouble with 64 bits, K 2^-63 of |A||B|^T). The solve's rows are
held to the backward error of a Cholesky solve, 4 R 2^-53 (||a|| ||H|| + ||m||) in the variables
scaled to a unit diagonal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2502_17683_gb300 import api as a
    return a


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _long(a, b):
    return a.astype(np.longdouble) @ b.astype(np.longdouble)


# 64- and 32-column tiles, K of part of a half chunk up to several chunks, K ranges in one launch
@pytest.mark.parametrize("shape", [(1, 1, 1), (127, 31, 64), (128, 64, 65), (129, 65, 128), (257, 97, 129),
                                   (40, 600, 700), (700, 300, 260), (31, 33, 8200)])
def test_emulated_product_edges(api, shape):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)
    A = rng.standard_normal((M, K)) * 10.0 ** rng.uniform(-5, 5, (M, 1)) * 10.0 ** rng.uniform(-4, 0, (1, K))
    B = rng.standard_normal((N, K)) * 10.0 ** rng.uniform(-5, 5, (N, 1))
    C = api.thc_cpd_emulated_gemm(_dev(A), _dev(B)).cpu().numpy()
    ref = _long(A, B.T)
    lim = U * np.abs(ref) + 2 * K * 2.0 ** -62 * np.max(np.abs(A), 1)[:, None] * np.max(np.abs(B), 1)[None, :]
    lim = lim + K * 2.0 ** -63 * (np.abs(A) @ np.abs(B).T)
    assert np.all(np.abs(C - ref) <= lim)


def test_emulated_product_keeps_nan_inf_and_subnormal_rows(api):
    rng = np.random.default_rng(3)
    A, B = rng.standard_normal((70, 200)), rng.standard_normal((50, 200))
    A[7, 3], B[11, 150] = np.nan, np.inf
    A[20] *= 2.0 ** -1060  # rows of subnormal numbers are numbers, too
    B[30] *= 2.0 ** 1000
    C = api.thc_cpd_emulated_gemm(_dev(A), _dev(B)).cpu().numpy()
    bad = np.zeros((70, 50), bool)
    bad[7], bad[:, 11] = True, True
    assert np.all(~np.isfinite(C[bad])) and np.all(np.isfinite(C[~bad]))
    np.testing.assert_allclose(C[20, 30], float(_long(A[20:21], B[30:31].T)[0, 0]), rtol=1e-12)


# FP64 entry points on both sides of the line between the FP64 pipes and the digits, symmetric and
# split products among them: against longdouble, no worse than an FP64 chain of the same length
@pytest.mark.parametrize("shape", [(3, 9, 17, 23), (9, 40, 130, 200), (13, 70, 257, 385), (21, 99, 389, 641)])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_fp64_mttkrp_rounds_no_worse_than_an_fma_chain(api, shape, mode):
    from thc_inputs import make_problem
    o, v, Rt, R = shape
    p = make_problem(o, v, Rt, R, seed=5 + mode)
    M = api.thc_cpd_mttkrp(_dev(p.Xo), _dev(p.Xv), _dev(p.Z), [_dev(a) for a in p.A], mode).cpu().numpy()
    X = (p.Xo, p.Xv, p.Xo, p.Xv)
    W = [_long(x.T, a) for x, a in zip(X, p.A)]
    Z = p.Z.astype(np.longdouble)
    Y = Z @ (W[2] * W[3]) if mode < 2 else Z.T @ (W[0] * W[1])
    ref = X[mode].astype(np.longdouble) @ (W[mode ^ 1] * Y)
    # every product's error in the order of its condition: the magnitudes carried through the chain
    aW = [np.abs(x.T) @ np.abs(a) for x, a in zip(X, p.A)]
    aY = np.abs(p.Z) @ (aW[2] * aW[3]) if mode < 2 else np.abs(p.Z.T) @ (aW[0] * aW[1])
    lim = (3 * v + 2 * Rt + 4) * U * (np.abs(X[mode]) @ (aW[mode ^ 1] * aY))
    assert np.all(np.abs(M - ref) <= lim)


def _normal(R, n, seed):
    rng = np.random.default_rng(seed)
    H = np.ones((R, R))
    for d in (9, max(9, R // 6), 9):
        a = rng.standard_normal((d, R))
        H *= (a / np.linalg.norm(a, axis=0)).T @ (a / np.linalg.norm(a, axis=0))
    return H, rng.standard_normal((n, R))


def _backward_ok(A, H, M):
    s = np.sqrt(np.diag(H))
    a, h, m = A * s, H / s[:, None] / s[None, :], M / s
    R = H.shape[0]
    lim = 4 * R * U * (np.linalg.norm(a, axis=1) * np.linalg.norm(h, 2) + np.linalg.norm(m, axis=1))
    return np.all(np.linalg.norm(a @ h - m, axis=1) <= lim)


# the dataflow kernel on its small grids (one to nine tiles)
@pytest.mark.parametrize("R,n", [(47, 3), (48, 1), (63, 5), (64, 8), (65, 9), (111, 16), (112, 17), (127, 2), (128, 40), (129, 3)])
@pytest.mark.parametrize("kind", ["als", "graded", "ill"])
def test_single_block_solve(api, R, n, kind):
    H, M = _normal(R, n, R + n)
    rng = np.random.default_rng(R)
    if kind == "graded":      # diagonal over twelve decades, rows of M of very different size
        s = 10.0 ** rng.uniform(-3, 3, R)
        H, M = H * s[:, None] * s[None, :], M * 10.0 ** rng.uniform(-6, 6, (n, 1))
    elif kind == "ill":       # condition ~1e8: the substitution grows far past the rows' headroom
        B = rng.standard_normal((max(1, R // 2), R))
        H = B.T @ B / R + 1e-8 * np.eye(R)
    A, used = api.thc_cpd_ldl_solve(_dev(H), _dev(M))
    assert not used and _backward_ok(A.cpu().numpy(), H, M)


def test_single_block_solve_special_rows(api):
    R = 100
    H, M = _normal(R, 6, 1)
    M[1], M[2, 50], M[4] = 0.0, np.nan, np.eye(R)[3]
    A, used = api.thc_cpd_ldl_solve(_dev(H), _dev(M))
    A = A.cpu().numpy()
    assert not used and np.all(A[1] == 0.0) and np.all(np.isnan(A[2]))
    keep = [0, 3, 4, 5]
    assert _backward_ok(A[keep], H, M[keep])


@pytest.mark.parametrize("where", ["indefinite", "singular"])
def test_single_block_solve_falls_back(api, where):
    R, n = 90, 4
    H, M = _normal(R, n, 7)
    if where == "indefinite":
        H[70, 20] = H[20, 70] = 3.0
    else:
        H[:, 60], H[60, :] = H[:, 59], H[59, :]
        H[60, 60] = H[59, 59]
    A, used = api.thc_cpd_ldl_solve(_dev(H), _dev(M))
    assert used
    if where == "singular":
        w, V = np.linalg.eigh(H)
        keep = w > R * np.finfo(float).eps * np.max(np.abs(w))
        ref = M @ ((V[:, keep] / w[keep]) @ V[:, keep].T)
        assert np.max(np.abs(A.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))


# side by side, problems of 400 columns and more factorise in fixed-point blocks (several blocks, a
# ragged last one), smaller ones do not: both against the single runs
def test_batched_fixed_point_blocks(api):
    from oracle import thc_cpd as O
    from thc_inputs import make_problem
    shapes = [(12, 57, 200, 399), (12, 57, 200, 400), (13, 61, 220, 513), (2, 9, 30, 40)]
    ps = [make_problem(*s, seed=40 + i) for i, s in enumerate(shapes)]
    batch = [dict(Xo=_dev(p.Xo), Xv=_dev(p.Xv), Z=_dev(p.Z), A=[_dev(a) for a in p.A],
                  lam=torch.ones(p.R, dtype=torch.float64, device="cuda")) for p in ps]
    res = api.thc_cpd_als_batched(batch, 3, 0.0)
    for p, r in zip(ps, res):
        ref = O.als(p.Xo, p.Xv, p.Z, p.A, 3)
        assert abs(r["fit"] - ref["fits"][-1]) <= 1e-10


# One launch splits several matrices, as given in 32 x 64 tiles and transposed in 64 x 32 ones:
# one row or column, one short of a tile, a tile, one more. Bound: a split keeps 16 bits (2^-17
# each operand, 2^-17 for the dropped lo x lo term), FP32 accumulation adds K 2^-23.
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (31, 33, 63), (32, 64, 64), (33, 65, 65), (129, 17, 191)])
def test_split_gemm_tiles(api, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M * 1000 + K)
    A = torch.randn(M, K, generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn(N, K, generator=g, device="cuda", dtype=torch.float64)
    C = api.thc_cpd_split_gemm(A, B, precision="bf16x3")
    lim = (2.0 ** -15 + K * 2.0 ** -23) * (A.abs() @ B.abs().T)
    assert ((C - A @ B.T).abs() <= lim).all()


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("o,v,Rt,R", [(1, 2, 8, 8), (3, 33, 63, 65), (31, 64, 129, 97)])
def test_split_mttkrp_operands(api, o, v, Rt, R, mode):
    g = torch.Generator(device="cuda").manual_seed(o * 100 + Rt)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    X, Z = [rnd(o, Rt), rnd(v, Rt)], rnd(Rt, Rt)
    A = [rnd(n, R) for n in (o, v, o, v)]

    def mttkrp(X, Z, A):
        W = [X[k % 2].T @ A[k] for k in range(4)]
        Y = Z @ (W[2] * W[3]) if mode < 2 else Z.T @ (W[0] * W[1])
        return X[mode % 2] @ (W[mode ^ 1] * Y)

    M = api.thc_cpd_mttkrp(X[0], X[1], Z, A, mode, precision="bf16x3")
    # three products deep, each split and accumulated as above, on absolute values
    lim = (6 * 2.0 ** -15 + (max(o, v) * 3 + 2 * Rt) * 2.0 ** -23) * mttkrp(
        [x.abs() for x in X], Z.abs(), [a.abs() for a in A])
    assert ((M - mttkrp(X, Z, A)).abs() <= lim).all()


# The digit cuts take several warps to a row up to 8 rows per SM, and up to 1024 threads to 8 columns
# up to two blocks per SM: one size on either side of both lines, for 148 to 160 SMs.
@pytest.mark.parametrize("shape", [(1150, 33, 300), (1300, 31, 257)])
def test_emulated_product_rows(api, shape):
    test_emulated_product_edges(api, shape)


# bound: FP64 sums of n, Rt and Rt terms on either side, on absolute values
@pytest.mark.parametrize("R", [2360, 2600])
@pytest.mark.parametrize("mode", [0, 3])
def test_fp64_mttkrp_many_columns(api, R, mode):
    o, v, Rt = 9, 17, 290
    g = torch.Generator(device="cuda").manual_seed(R + mode)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    X, Z = [rnd(o, Rt), rnd(v, Rt)], rnd(Rt, Rt)
    A = [rnd(n, R) for n in (o, v, o, v)]

    def mttkrp(X, Z, A):
        W = [X[k % 2].T @ A[k] for k in range(4)]
        Y = Z @ (W[2] * W[3]) if mode < 2 else Z.T @ (W[0] * W[1])
        return X[mode % 2] @ (W[mode ^ 1] * Y)

    M = api.thc_cpd_mttkrp(X[0], X[1], Z, A, mode)
    lim = 2 * (3 * v + 2 * Rt) * U * mttkrp([x.abs() for x in X], Z.abs(), [a.abs() for a in A])
    assert ((M - mttkrp(X, Z, A)).abs() <= lim).all()


# Grams and projections of several factors in one launch: rows of one product end inside a tile, T of
# 8, 16 and 32, a product that leaves the list (its tiles differ). Bound as above, in FP64.
@pytest.mark.parametrize("o,v,Rt,R", [(1, 2, 8, 8), (3, 5, 9, 65), (5, 15, 60, 80), (9, 33, 97, 161), (12, 60, 200, 300)])
def test_small_products_in_one_launch(api, o, v, Rt, R):
    g = torch.Generator(device="cuda").manual_seed(o * 100 + R)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    X, Z = [rnd(o, Rt), rnd(v, Rt)], rnd(Rt, Rt)
    A = [rnd(n, R) for n in (o, v, o, v)]
    lam = rnd(R)

    def parts(X, Z, A, lam):
        W = [X[k % 2].T @ A[k] for k in range(4)]
        G = [a.T @ a for a in A]
        return (lam * (W[0] * W[1]) * (Z @ (W[2] * W[3]))).sum(), lam @ ((G[0] * G[1] * G[2] * G[3]) @ lam)

    loss, _ = api.thc_cpd_loss(X[0], X[1], Z, A, lam=lam, normG2=1.0)
    s1, s2 = parts(X, Z, A, lam)
    a1, a2 = parts([x.abs() for x in X], Z.abs(), [a.abs() for a in A], lam.abs())
    # sums of v, v, Rt terms (s1) and v of four Grams (s2), then Rt R and R^2 terms, on either side
    lim = 2 * U * (2 * (4 * v + Rt + Rt + R) * a1 + (4 * v + 2 * R) * a2)
    assert abs(loss - float(1.0 - 2.0 * s1 + s2)) <= float(lim) + 4 * U

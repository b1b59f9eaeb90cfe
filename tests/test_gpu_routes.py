"""Calls on either side of the lines between the FP64 pipes and the digit products, against torch in
FP64 on the same device. Bounds: both sides sum K terms (a relative error of K 2^-53 each on the
absolute values) in every product of the chain."""
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


def _rnd(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)


# a Gram of 8192 terms is the longest that one digit launch sums
@pytest.mark.parametrize("o,v", [(5, 8192), (5, 8193), (8200, 7)])
def test_norm_of_long_factors(api, o, v):
    rnd, Rt = _rnd(o + v), 220
    Xo, Xv, Z = rnd(o, Rt), rnd(v, Rt), rnd(Rt, Rt)

    def norm2(Xo, Xv, Z):
        S = (Xo.T @ Xo) * (Xv.T @ Xv)
        return float((Z * (S @ Z @ S)).sum())

    lim = 2 * U * (2 * (o + v) + 2 * Rt + Rt * Rt) * norm2(Xo.abs(), Xv.abs(), Z.abs())
    assert abs(api.thc_cpd_thc_norm2(Xo, Xv, Z) - norm2(Xo, Xv, Z)) <= lim


def _pattern(x):
    return np.where(np.isnan(x), 2, np.where(np.isposinf(x), 1, np.where(np.isneginf(x), -1, 0)))


# infinities go through a digit product as through an FP64 one: infinite with the sign of the term, NaN
# against a zero or an infinity of the other sign, and nothing outside their row or column
@pytest.mark.parametrize("M,N,K", [(70, 50, 200), (129, 65, 65), (3, 2, 8200)])
def test_infinities(api, M, N, K):
    rng = np.random.default_rng(K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    A[1, 3], A[2, 0], A[2, K - 1] = np.inf, -np.inf, np.inf
    B[0, 3] = 0.0
    B[1, K // 2] = -np.inf
    if M > 100:
        A[128, 64], A[100, 5], B[64, 0] = np.inf, np.nan, np.inf
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    C = api.thc_cpd_emulated_gemm(d(A), d(B)).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = np.array([(a * B).sum(-1) for a in A])
    np.testing.assert_array_equal(_pattern(C), _pattern(ref))
    ok = np.isfinite(ref)
    lim = 2 * K * U * (np.abs(A)[:, None, :] * np.abs(B)[None, :, :]).sum(-1) if M * N * K < 1e7 else None
    assert lim is None or np.all(np.abs(C - ref)[ok] <= lim[ok])


# the same through an entry point: digits of Z, of X, of a factor and of Hadamard products, split K
@pytest.mark.parametrize("mode", [0, 3])
@pytest.mark.parametrize("zero", [False, True])
def test_infinities_in_an_mttkrp(api, mode, zero):
    o, v, Rt, R = 12, 90, 200, 300
    rng = np.random.default_rng(mode)
    X = [rng.random((n, Rt)) + 0.1 for n in (o, v)]
    Z, A = rng.random((Rt, Rt)) + 0.1, [rng.random((n, R)) + 0.1 for n in (o, v, o, v)]
    A[2][5, 7] = A[1][3, 130] = np.inf
    if zero:
        X[0][5, 3] = X[1][3, 150] = 0.0
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    M = api.thc_cpd_mttkrp(d(X[0]), d(X[1]), d(Z), [d(a) for a in A], mode).cpu().numpy()
    mul = lambda a, b: np.array([(r[:, None] * b).sum(0) for r in a])
    with np.errstate(invalid="ignore"):
        W = [mul(X[k % 2].T, A[k]) for k in range(4)]
        Y = mul(Z, W[2] * W[3]) if mode < 2 else mul(Z.T, W[0] * W[1])
        ref = mul(X[mode % 2], W[mode ^ 1] * Y)
    np.testing.assert_array_equal(_pattern(M), _pattern(ref))
    ok = np.isfinite(ref)
    assert np.all(np.abs(M - ref)[ok] <= 2 * (3 * v + 2 * Rt + 4) * U * ref[ok])


# results in and below the subnormal range: a digit product rounds to the smallest unit 2^-1074 where an
# FP64 product does (half a unit each), and gives a signed zero below
@pytest.mark.parametrize("e", [-1010, -1030, -1040, -1060, -1068, -1071, -1074, -1076, -1080])
def test_subnormal_results(api, e):
    rng = np.random.default_rng(-e)
    A, B = rng.standard_normal((70, 200)), rng.standard_normal((50, 200))
    fine = np.longdouble(2.0) ** e
    ref = (A.astype(np.longdouble) @ B.astype(np.longdouble).T) * fine
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    C = api.thc_cpd_emulated_gemm(d(A * 2.0 ** (e // 2)), d(B * 2.0 ** (e - e // 2))).cpu().numpy()
    # 2^-53 of the result, the digits' 2^-61 K max max, half a unit of the subnormal range
    top = np.max(np.abs(A), 1)[:, None] * np.max(np.abs(B), 1)[None, :]
    lim = U * np.abs(ref) + 2.0 ** -61 * 200 * top * fine + np.longdouble(2.0) ** -1075 * (1 + 2.0 ** -20)
    assert np.all(np.abs(C - ref) <= lim)
    assert e < -1074 or np.any(C != 0.0)


# more points than 1 GB of intermediates holds: two full groups and a shorter last one
@pytest.mark.parametrize("products", ["auto", "fp64"])
@pytest.mark.parametrize("na", [500, 301])
def test_exchange_in_groups(api, na, products):
    from oracle import exchange as X
    from tests._util import to_dev
    from thc_inputs import make_lt, make_problem
    o, v, Rt, R = 20, 60, 203, 261
    p = make_problem(o, v, Rt, R, seed=na)
    lam = np.random.default_rng(na).uniform(0.5, 2.0, R)
    Lam, Gam = X.lt_factors(*make_lt(o, v, na, na))
    d, dev = to_dev(p, torch), lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    e1, e2, _ = api.thc_cpd_exchange(d["Xo"], d["Xv"], d["Z"], d["A"], dev(lam), dev(Lam), dev(Gam),
                                     products=products)
    r1, r2, _ = X.exchange_robust(p.Xo, p.Xv, p.Z, p.A, lam, Lam, Gam)
    # relative to the size of the terms, as for one group
    s1 = abs(X.exchange_single(np.abs(p.Xo), np.abs(p.Xv), np.abs(p.Z), [np.abs(a) for a in p.A], lam, Lam, Gam))
    s2 = abs(X.exchange_double([np.abs(a) for a in p.A], lam, Lam, Gam))
    assert abs(e1 - r1) <= 1e-12 * s1 and abs(e2 - r2) <= 1e-12 * s2


# a left operand of more digit rows than 256 MB holds (32000 of eight chunks): two ranges of rows
def test_core_fit_in_row_ranges(api):
    o, v, Rt, na = 200, 1000, 100, 160
    rnd = _rnd(3)
    Xo, Xv, B = rnd(o, Rt), rnd(v, Rt), rnd(na, o, v)
    Z, _, used = api.thc_cpd_core_fit(Xo, Xv, B)
    E = ((B.reshape(na * o, v) @ Xv).reshape(na, o, Rt) * Xo).sum(1)
    S = (Xo.T @ Xo) * (Xv.T @ Xv)
    F = torch.linalg.solve(S, E.T).T
    ref = F.T @ F
    # sums of v, o and na terms and the solve, each against its own size: the factors' norms carry them on
    cond = float(torch.linalg.cond(S))
    lim = 4 * (v + o + na + Rt) * U * cond * float(torch.linalg.norm(F)) ** 2
    assert not used and float(torch.linalg.norm(Z - ref)) <= lim


# Z and a factor graded over 80 binary digits, the large entries of one against zeros of the other: on the
# FP64 pipes every entry is right to the rounding of its own terms (all positive), the tiny ones too
@pytest.mark.parametrize("mode", [0, 2])
def test_graded_operands_on_the_fp64_pipes(api, mode):
    o, v, Rt, R = 10, 90, 200, 300
    rng = np.random.default_rng(mode)
    X, Z = [rng.random((n, Rt)) + 0.1 for n in (o, v)], rng.random((Rt, Rt)) + 0.1
    A = [rng.random((n, R)) + 0.1 for n in (o, v, o, v)]
    Z[:, 100:], Z[100:, :] = Z[:, 100:] * 2.0 ** -80, Z[100:, :] * 2.0 ** -80
    X[1][:45, 100:], X[1][45:, :100] = 0.0, 0.0
    A[1][:45, :150], A[3][:45, :150] = 0.0, 0.0   # W2, W4: rows below 100 are zero for these columns
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    M = api.thc_cpd_mttkrp(d(X[0]), d(X[1]), d(Z), [d(a) for a in A], mode, products="fp64").cpu().numpy()
    L = lambda x: x.astype(np.longdouble)
    W = [L(X[k % 2]).T @ L(A[k]) for k in range(4)]
    Y = L(Z) @ (W[2] * W[3]) if mode < 2 else L(Z).T @ (W[0] * W[1])
    ref = L(X[mode % 2]) @ (W[mode ^ 1] * Y)
    assert np.max(ref[:, :150]) < 1e-20 * np.min(ref[:, 150:])
    assert np.all(np.abs(M - ref) <= (3 * v + 2 * Rt + 4) * U * ref)


# two K ranges (8192 terms and the rest) of which one has tiny rows only: their exponents say nothing of the
# other range's entries
@pytest.mark.parametrize("big,tiny", [(slice(0, 8192), slice(8192, 8300)), (slice(8192, 8300), slice(0, 8192))])
@pytest.mark.parametrize("scale", [1e50, 1e-120])
def test_tiny_range_beside_another(api, big, tiny, scale):
    rng = np.random.default_rng(9)
    A, B = rng.standard_normal((31, 8300)), rng.standard_normal((33, 8300))
    A[:, big], B[:, big] = A[:, big] * scale, B[:, big] * scale
    A[:, tiny], B[:, tiny] = A[:, tiny] * 1e-200, B[:, tiny] * 1e-200
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    C = api.thc_cpd_emulated_gemm(d(A), d(B)).cpu().numpy()
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble).T
    K = 8300
    top = np.max(np.abs(A), 1)[:, None] * np.max(np.abs(B), 1)[None, :]
    # one rounding per range, the digits' bound, the longdouble sum's; what underflows lies below 1e-300
    lim = 3 * U * np.abs(ref) + 2.0 ** -61 * K * top + K * 2.0 ** -63 * (np.abs(A) @ np.abs(B).T) + 1e-300
    assert np.all(np.abs(C - ref) <= lim)

"""The fixed-point LDL^T blocks (the batched driver's factorisation from R = 400 on) through the solve
that runs them alone, where they can go wrong: block and tile edges, graded and ill-conditioned
matrices whose appended rows outgrow their headroom, rows without a number, matrices that are not
positive definite.

Bound: the backward error of a Cholesky solve, ||a h - m|| <= 4 R 2^-53 (||a|| ||h|| + ||m||) for every
row, in the variables scaled to a unit diagonal."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def solve():
    import __graft_entry__ as g
    g.build()
    from paper_2502_17683_gb300 import _lib
    f = _lib.load().thc_cpd_fixed_solve
    f.argtypes, f.restype = [_lib.I, _lib.I, _lib.P, _lib.P, _lib.P, _lib.IP, _lib.OPTS], ctypes.c_int

    def run(H, M):
        h, m = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (H, M))
        a, used = torch.empty_like(m), ctypes.c_int()
        _lib.check(f(H.shape[0], M.shape[0], h.data_ptr(), m.data_ptr(), a.data_ptr(), ctypes.byref(used), None))
        return a.cpu().numpy(), bool(used.value)

    return run


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
    lim = 4 * H.shape[0] * U * (np.linalg.norm(a, axis=1) * np.linalg.norm(h, 2) + np.linalg.norm(m, axis=1))
    return np.all(np.linalg.norm(a @ h - m, axis=1) <= lim)


SIZES = [(1, 1), (16, 3), (17, 2), (100, 7), (127, 1), (128, 9), (129, 8), (257, 30), (400, 20), (513, 130)]


@pytest.mark.parametrize("R,n", SIZES)
@pytest.mark.parametrize("kind", ["als", "graded", "ill"])
def test_backward_error(solve, R, n, kind):
    H, M = _normal(R, n, R + n)
    rng = np.random.default_rng(R)
    if kind == "graded":  # diagonal over twelve decades, rows of M of very different size
        s = 10.0 ** rng.uniform(-3, 3, R)
        H, M = H * s[:, None] * s[None, :], M * 10.0 ** rng.uniform(-6, 6, (n, 1))
    elif kind == "ill":   # condition ~1e8: the substitution grows past the rows' first headroom
        B = rng.standard_normal((max(1, R // 2), R))
        H = B.T @ B / R + 1e-8 * np.eye(R)
    A, used = solve(H, M)
    assert not used and _backward_ok(A, H, M)


@pytest.mark.parametrize("R", [100, 300])
def test_rows_without_a_number(solve, R):
    H, M = _normal(R, 6, 1)
    M[1], M[2, R // 2], M[3, R - 1], M[4] = 0.0, np.nan, np.inf, np.eye(R)[3]
    A, used = solve(H, M)
    assert not used and np.all(A[1] == 0.0) and np.all(np.isnan(A[2])) and not np.any(np.isfinite(A[3]))
    keep = [0, 4, 5]
    assert _backward_ok(A[keep], H, M[keep])


@pytest.mark.parametrize("R,at", [(90, (70, 20)), (200, (70, 20)), (200, (150, 20)), (200, (150, 140))])
@pytest.mark.parametrize("where", ["indefinite", "singular"])
def test_failed_pivot_takes_the_pseudo_inverse(solve, R, at, where):
    H, M = _normal(R, 4, 7)
    i, j = at
    if where == "indefinite":
        H[i, j] = H[j, i] = 3.0
    else:
        H[:, i], H[i, :] = H[:, j], H[j, :]
        H[i, i] = H[j, j]
    A, used = solve(H, M)
    assert used
    if where == "singular":
        w, V = np.linalg.eigh(H)
        keep = w > R * np.finfo(float).eps * np.max(np.abs(w))
        ref = M @ ((V[:, keep] / w[keep]) @ V[:, keep].T)
        assert np.max(np.abs(A - ref)) <= 1e-9 * np.max(np.abs(ref))


def _growing(R):
    """2 C C^T for C = I - strictly lower ones: small integers, every pivot 2 and every step exact, but
    the substitution of a unit row doubles with each column."""
    C = np.eye(R) - np.tril(np.ones((R, R)), -1)
    return 2.0 * C @ C.T


# up to 2^49 of growth a row is done again with more headroom; beyond, the solve must not pass for one
# that succeeded
@pytest.mark.parametrize("R,fits", [(40, True), (50, True), (60, False), (128, False)])
def test_rows_that_outgrow_every_headroom(solve, R, fits):
    H, M = _growing(R), np.vstack([np.eye(R)[:1], np.ones((1, R))])
    A, used = solve(H, M)
    assert used == (not fits)
    if fits:
        assert _backward_ok(A, H, M)


# entries below the bound of their block (they pass the first check) that overdraw a diagonal entry far
# enough to wrap its 64 bits back to a positive value, inside one 16-column tile and across tiles
@pytest.mark.parametrize("R,row,cols", [(32, 5, (0, 4)), (32, 20, (0, 4)), (128, 100, (0, 4)), (128, 127, (40, 44)),
                                        (128, 127, (13, 19)), (200, 190, (130, 134))])
def test_overdrawn_diagonal_is_noticed(solve, R, row, cols):
    H = 0.25 * np.eye(R)
    H[row, cols[0]:cols[1]] = H[cols[0]:cols[1], row] = 0.475
    A, used = solve(H, np.random.default_rng(R).standard_normal((3, R)))
    assert used


# quotients below the normal range: Y = M / 4 rounded to units of 2^-1074, and A from it
@pytest.mark.parametrize("R", [20, 130])
@pytest.mark.parametrize("e", [-1020, -1040, -1068, -1073])
def test_subnormal_rows(solve, R, e):
    M = np.random.default_rng(R).standard_normal((3, R)) * 2.0 ** (e + 20) * 2.0 ** -20
    A, used = solve(4.0 * np.eye(R), M)
    assert not used and np.any(A != 0.0)
    # exact but for the reciprocal square roots (2^-52 together) and one rounding of the result
    assert np.all(np.abs(A - M / 4) <= 2.0 ** -52 * np.abs(M / 4) + 2.0 ** -1074)


# in the batch: two identical columns in every start factor make each H singular, so the sweep is rolled back
# and replayed with the pseudo-inverse, beside a problem that is not
def test_batched_problem_with_a_failed_pivot():
    import __graft_entry__ as g
    g.build()
    from oracle import thc_cpd as O
    from paper_2502_17683_gb300 import api
    from thc_inputs import make_problem
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    ps = [make_problem(12, 57, 200, 420, seed=50), make_problem(12, 57, 200, 420, seed=51)]
    As = [[a.copy() for a in p.A] for p in ps]
    for a in As[0]:
        a[:, 333] = a[:, 17]
    batch = [dict(Xo=dev(p.Xo), Xv=dev(p.Xv), Z=dev(p.Z), A=[dev(a) for a in A],
                  lam=torch.ones(420, dtype=torch.float64, device="cuda")) for p, A in zip(ps, As)]
    res = api.thc_cpd_als_batched(batch, 2, 0.0)
    for p, A, r, singular in zip(ps, As, res, (True, False)):
        ref = O.als(p.Xo, p.Xv, p.Z, tuple(A), 2)
        assert bool(r["flags"] & 1) == bool(r["flags"] & 2) == singular
        assert abs(r["loss"] - ref["losses"][-1]) <= 1e-9 * ref["normG2"]

"""The FP64 shift solve beyond the sizes of the single-tile solver (FP32 factorization refined to
FP64, with the FP64 factorization behind it): against numpy's FP64 solve, at the edges of its
tiles (32), update chunks (256), cluster sizes (batch) and odd sizes, for rows of very different
scale, for a near-singular S (left to the FP64 factorization), for S with a negative eigenvalue
(shift raised as the FP64 factorization raises it), a zero and a non-finite right-hand side."""
import numpy as np
import pytest

from gpu_helpers import Case, require_gpu, from_dev_complex, to_dev_complex, torch
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _ansatz(P):
    """A tied Jastrow on an open chain with d = 0 has P = 2 n - 1 parameters, on a ring n + n // 2."""
    import paper_2506_23928_gb300 as pkg
    for n in range(2, 201):
        for pbc in (False, True):
            q = n + n // 2 if pbc else 2 * n - 1
            if q == P:
                model = pkg.Model(pkg.lattice_couplings((n,), 1.0, 1.5), 1.0, 0.1)
                return pkg.Ansatz(model, abi.OTVMC_LJ, 0, 0, pbc)
    raise ValueError(P)


def _solve(P, S, D, eps):
    ans = _ansatz(P)
    assert ans.P == P
    T = S.shape[0]
    S_d = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    delta = torch.zeros((T, P, 2), dtype=torch.float64, device="cuda")
    shift = torch.zeros(T, dtype=torch.float64, device="cuda")
    nb = abi.otvmc_workspace_bytes(ans.handle, T, 64, abi.OTVMC_PREC_FP64)
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    check(abi.otvmc_solve_step(ans.handle, T, 64, abi.OTVMC_PREC_FP64, abi.OTVMC_REG_SHIFT, eps, 0.0, S_d, None,
                               None, to_dev_complex(D), delta, shift, work, nb))
    st = abi.otvmc_check(work)
    return st, from_dev_complex(delta).reshape(T, P), shift.cpu().numpy()


def _inputs(P, T, ns, seed, spread=0):
    g = np.random.default_rng(seed)
    A = g.normal(0, 1, (T, ns, P))
    if spread:
        A = A * 2.0 ** g.integers(-spread, spread + 1, P)
    A = A - A.mean(1, keepdims=True)
    S = np.einsum("txi,txj->tij", A, A) / ns
    return 0.5 * (S + S.transpose(0, 2, 1)), g.normal(0, 1, (T, P)) + 1j * g.normal(0, 1, (T, P))


def _want(S, D, eps):
    return np.stack([np.linalg.solve(S[t] + eps * np.eye(S.shape[1]), D[t]) for t in range(len(D))])


@pytest.mark.parametrize("P,T", [(47, 3), (48, 1), (49, 3), (63, 2), (64, 2), (65, 2), (96, 1), (97, 20), (255, 2),
                                 (256, 30), (257, 3), (287, 1), (399, 2)])
def test_refined_solve_matches_fp64(P, T):
    S, D = _inputs(P, T, 4 * P, P, spread=3 if P % 2 else 0)
    st, x, shift = _solve(P, S, D, 1e-4)
    assert st == abi.OTVMC_OK and np.all(shift == 1e-4)
    # forward error of a backward-stable FP64 solve: a few eps cond (cond below 1e4 after scaling)
    for t in range(T):
        r = D[t] - (S[t] @ x[t] + 1e-4 * x[t])
        scale = np.abs(S[t]).sum(1).max() * np.abs(x[t]).max() + np.abs(D[t]).max()
        assert np.abs(r).max() < 4 * P * 2.0 ** -53 * scale
    w = _want(S, D, 1e-4)
    for t in range(T):
        cond = np.linalg.cond(S[t] + 1e-4 * np.eye(P))
        assert np.abs(x[t] - w[t]).max() / np.abs(w[t]).max() < 4 * P * 2.0 ** -53 * cond


def test_near_singular_goes_to_fp64():
    """Rank-deficient S with a shift below FP32's resolution: the solution of the FP64 factorization."""
    P, T, eps = 99, 2, 1e-9
    S, D = _inputs(P, T, 40, 3)
    st, x, shift = _solve(P, S, D, eps)
    assert st == abi.OTVMC_OK and np.all(shift == eps)
    for t in range(T):
        r = D[t] - (S[t] @ x[t] + eps * x[t])
        scale = np.abs(S[t]).sum(1).max() * np.abs(x[t]).max() + np.abs(D[t]).max()
        assert np.abs(r).max() < 16 * P * 2.0 ** -53 * scale


def test_negative_eigenvalue_raises_the_shift():
    P, T, eps = 129, 3, 1e-3
    S, D = _inputs(P, T, 4 * P, 4)
    lam, V = np.linalg.eigh(S[1])
    S[1] -= np.outer(V[:, 0], V[:, 0]) * (lam[0] + 5e-3)  # smallest eigenvalue -5e-3: eps 1e-3 fails, 1e-1 holds
    S[1] = 0.5 * (S[1] + S[1].T)
    st, x, shift = _solve(P, S, D, eps)
    assert st == abi.OTVMC_OK
    assert shift[0] == eps and shift[2] == eps and np.isclose(shift[1], 0.1)
    w = _want(S[1:2], D[1:2], 0.1)
    assert np.abs(x[1] - w[0]).max() / np.abs(w[0]).max() < 1e-10
    S[:] = -S  # eigenvalues down to about -2.3: the shift of the third attempt, 10, holds
    st, x, shift = _solve(P, S, D, eps)
    assert st == abi.OTVMC_OK and np.allclose(shift, 10.0)
    w = _want(S, D, 10.0)
    assert np.abs(x - w).max() / np.abs(w).max() < 1e-10


def test_zero_and_non_finite_right_hand_sides():
    P, T, eps = 65, 3, 1e-4
    S, D = _inputs(P, T, 300, 5)
    D[0] = 0
    D[1, 7] = np.nan
    st, x, _ = _solve(P, S, D, eps)
    assert st == abi.OTVMC_ERR_NOT_PD  # as the FP64 factorization reports a solution that is not finite
    assert np.all(x[0] == 0) and np.all(x[1] == 0)
    w = _want(S[2:], D[2:], eps)
    assert np.abs(x[2] - w[0]).max() / np.abs(w[0]).max() < 1e-11


def test_batch_size_does_not_change_the_solution():
    """The cluster size follows the batch; the result does not."""
    P = 399
    S, D = _inputs(P, 1, 800, 6)
    _, one, _ = _solve(P, S, D, 1e-4)
    _, many, _ = _solve(P, np.repeat(S, 80, 0), np.repeat(D, 80, 0), 1e-4)
    assert np.array_equal(many, np.repeat(one, 80, 0))


@pytest.mark.parametrize("n,ns", [(5, 33), (16, 1000), (23, 131), (33, 400), (20, 100)])
def test_fp64_S_is_correctly_rounded(n, ns):
    """S of the FP64 path from exact counts (and, at 210 parameters on 100 samples, from the FP64
    products): (ns G - c c^T) / ns^2 in exact integers."""
    c = Case((n,), kappa=0.1)
    T = 2
    sig, sp = c.spins(9, T, ns)
    g = np.random.default_rng(2)
    v = to_dev_complex(g.normal(0, 1, (T, ns)) + 1j * g.normal(0, 1, (T, ns)))
    S = torch.zeros((T, c.P, c.P), dtype=torch.float64, device="cuda")
    ob = torch.zeros((T, c.P), dtype=torch.float64, device="cuda")
    D = torch.zeros((T, c.P, 2), dtype=torch.float64, device="cuda")
    work, nb = c.work(T, ns, abi.OTVMC_PREC_FP64)
    check(abi.otvmc_build_S_F(c.ans.handle, None, sp, v, T, ns, abi.OTVMC_PREC_FP64, S, None, ob, D, work, nb))
    check(abi.otvmc_check(work))
    for t in range(T):
        s = sig[t].astype(np.int64)
        j, k = np.triu_indices(n, 1)
        O = np.concatenate([s, s[:, j] * s[:, k]], 1)
        cnt = O.sum(0)
        want = (ns * (O.T @ O) - np.outer(cnt, cnt)) / float(ns * ns)
        got = S[t].cpu().numpy()
        tol = 0.0 if c.P * 4 + (ns + 15) // 16 * 16 <= 8 * ns - 64 else 4e-16 * np.sqrt(ns)
        assert np.abs(got - want).max() <= tol
        assert np.array_equal(ob[t].cpu().numpy(), cnt / ns)

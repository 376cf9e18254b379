"""Right-hand sides of the refined FP64 solve: a non-finite one is reported whatever its other entries
are, the real and the imaginary system are each solved to their own accuracy, and a solution is
correct to the rounding of FP64."""
import numpy as np
import pytest

from gpu_helpers import require_gpu
from paper_2506_23928_gb300 import abi
from test_gpu_solve_refined import _inputs, _solve, _want

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("re,im,entries", [
    (np.nan, np.nan, slice(None)), (np.nan, 0.0, slice(None)), (0.0, np.nan, slice(None)), (np.nan, 0.0, slice(7, 8)),
    (np.inf, 0.0, slice(-1, None)), (0.0, -np.inf, slice(0, 1))])
@pytest.mark.parametrize("P", [47, 65])
def test_non_finite_right_hand_side_is_reported(P, re, im, entries):
    """Beside zeros alone a NaN must not read as a right-hand side of zeros (47: the FP64 factorization)."""
    S, D = _inputs(P, 2, 300, 5)
    D[0] = 0
    D.real[0, entries] = re
    D.imag[0, entries] = im
    st, x, shift = _solve(P, S, D, 1e-4)
    assert st == abi.OTVMC_ERR_NOT_PD
    assert np.all(x[0] == 0)
    w = _want(S[1:], D[1:], 1e-4)
    assert np.abs(x[1] - w[0]).max() / np.abs(w[0]).max() < 1e-11


def test_solution_beyond_the_range_is_reported():
    """A finite right-hand side whose solution is not: S = 1e-20, shift 0."""
    P = 65
    S = np.stack([np.eye(P) * 1e-20, np.eye(P)])
    D = np.ones((2, P), dtype=np.complex128)
    D[0, 3] = 1e289
    st, x, _ = _solve(P, S, D, 0.0)
    assert st == abi.OTVMC_ERR_NOT_PD
    assert np.all(x[0] == 0) and np.all(x[1] == 1)


@pytest.mark.parametrize("P,ratio", [(199, 1e-8), (199, 1e8), (65, 1e-30), (287, 1e-14), (48, 0.0)])
def test_parts_are_solved_separately(P, ratio):
    """The bound of the FP64 solve, 4 P 2^-53 cond of the largest entry, for each part by itself."""
    S, D = _inputs(P, 2, 4 * P, 11)
    D = D.real * ratio + 1j * D.imag
    st, x, shift = _solve(P, S, D, 1e-4)
    assert st == abi.OTVMC_OK and np.all(shift == 1e-4)
    for t in range(2):
        A = S[t] + 1e-4 * np.eye(P)
        tol = 4 * P * 2.0 ** -53 * np.linalg.cond(A)
        for got, rhs in ((x[t].real, D[t].real), (x[t].imag, D[t].imag)):
            w = np.linalg.solve(A, rhs)
            assert np.abs(got - w).max() <= tol * np.abs(w).max()


@pytest.mark.parametrize("P,ns,eps", [(99, 110, 1e-4), (199, 230, 1e-4), (399, 440, 1e-3), (399, 420, 1e-4)])
def test_solution_is_correct_to_its_rounding(P, ns, eps):
    """Against the solution in extended precision, at conditions of 1e3 to 5e3 where a plain FP64 solve
    is off by 5e-15 to 6e-14.  Bound: the rounding of x and what is left after the last correction, 2^-53
    each, and the residual's error, entries of the scaled S below 2^-8 cut at 2^-60, through the inverse."""
    S, D = _inputs(P, 2, ns, 21)
    st, x, shift = _solve(P, S, D, eps)
    assert st == abi.OTVMC_OK and np.all(shift == eps)
    L = np.longdouble
    for t in range(2):
        A = S[t].astype(L) + L(eps) * np.eye(P).astype(L)
        inv = np.linalg.inv(A.astype(np.float64))
        d = 2.0 ** -((np.floor(np.log2(np.diag(S[t]) + eps)).astype(int) + 1) >> 1)
        tol = 2.0 ** -52 + 2.0 ** -60 * np.linalg.norm(inv / np.outer(d, d), 2)
        for got, rhs in ((x[t].real, D[t].real), (x[t].imag, D[t].imag)):
            w = np.zeros(P, L)
            for _ in range(10):
                w = w + inv @ (rhs.astype(L) - A @ w).astype(np.float64)
            assert np.abs(got - w).max() <= tol * np.abs(w).max()

"""Right-hand sides of the refined FP64 solve: a non-finite one is reported whatever its other entries
are."""
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

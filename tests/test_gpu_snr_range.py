"""The SNR filter beyond P = 96 at the ends of its range: more trajectories than the second dimension of
a grid holds."""
import numpy as np
import pytest

from gpu_helpers import require_gpu, from_dev_complex, to_dev_complex, torch
import synth
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _snr(ans, S, obar, sp, v, D, thr, eps_svd):
    T, P, ns = S.shape[0], ans.P, sp.shape[1]
    delta = torch.zeros((T, P, 2), dtype=torch.float64, device="cuda")
    nb = abi.otvmc_snr_workspace_bytes(ans.handle, T)
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    check(abi.otvmc_solve_snr(ans.handle, T, ns, S, obar, sp, v, D, thr, eps_svd, delta, None, work, nb))
    check(abi.otvmc_check(work))
    return delta


def _ansatz(kind, n, d, pbc):
    import paper_2506_23928_gb300 as pkg
    return pkg.Ansatz(pkg.Model(pkg.lattice_couplings((n,), 1.0, 1.5, False, pbc), 1.0, 0.1), kind, 0, d, pbc)


def _pack(sig):
    return torch.from_numpy(synth.pack_spins(sig).view(np.int64)).cuda()


def test_more_trajectories_than_a_grid_dimension():
    """65537 trajectories of the smallest system beyond the shared-memory solver, all alike but the last."""
    T, n, ns = 65537, 49, 8
    ans = _ansatz(abi.OTVMC_LJ, n, 0, False)
    P = ans.P
    assert P == 97
    g = np.random.default_rng(6)
    sig = synth.random_spins(7, 2, ns, n)
    s = sig.astype(np.float64)
    p, q = np.triu_indices(n, 1)
    pair = s[:, :, p] * s[:, :, q]
    O = np.concatenate([s] + [pair[:, :, q - p == x].sum(2, keepdims=True) for x in range(1, n)], 2)
    obar = O.mean(1)
    v = g.normal(0, 1, (2, ns)) + 1j * g.normal(0, 1, (2, ns))
    D = np.einsum("txi,tx->ti", O - obar[:, None], v - v.mean(1, keepdims=True)) / ns
    B = g.normal(0, 1, (2, P, 4 * P))
    S = B @ B.transpose(0, 2, 1) / (4 * P)
    pick = torch.zeros(T, dtype=torch.int64, device="cuda")
    pick[-1] = 1
    two = [torch.from_numpy(S).cuda(), torch.from_numpy(obar).cuda(), _pack(sig), to_dev_complex(v), to_dev_complex(D)]
    small = _snr(ans, *two, 4.0, 1e-12)
    many = _snr(ans, *[a.reshape(2, -1)[pick].reshape(T, *a.shape[1:]) for a in two], 4.0, 1e-12)
    assert bool((small.abs().amax((1, 2)) > 0).all())
    assert torch.equal(many[-1], small[1])
    assert bool((many[:-1] == small[0]).all())

"""The SNR filter beyond P = 96 (tridiagonalisation, weighted Gram matrix in exact integers, QL)
against numpy's eigendecomposition: full and tied Jastrow, chain and ring, tile edges of 64, ragged
and single-chunk sample counts, polarised samples, several spin words, and a batch."""
import numpy as np
import pytest

from gpu_helpers import require_gpu, from_dev_complex, to_dev_complex, torch
import synth
from oracle import tvmc
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _O(kind, n, d, pbc, sig):
    s = sig.astype(np.float64)
    j, k = np.triu_indices(n, 1)
    pair = s[:, j] * s[:, k]
    if kind == abi.OTVMC_JASTROW:
        return np.concatenate([s, pair], 1)
    D = np.minimum(k - j, n - (k - j)) if pbc else k - j
    groups = [[p] for p in np.nonzero(D <= d)[0]] + [np.nonzero(D == x)[0] for x in range(d + 1, n) if np.any(D == x)]
    return np.concatenate([s] + [pair[:, g].sum(1, keepdims=True) for g in groups], 1)


@pytest.mark.parametrize("kind,n,d,pbc,ns,T,down", [
    (abi.OTVMC_JASTROW, 14, 0, False, 700, 2, False), (abi.OTVMC_JASTROW, 16, 0, False, 1000, 1, True),
    (abi.OTVMC_LJ, 65, 0, True, 400, 2, False), (abi.OTVMC_LJ, 64, 1, True, 800, 1, False),
    (abi.OTVMC_LJ, 65, 0, False, 517, 1, False), (abi.OTVMC_LJ, 100, 1, True, 2051, 1, False),
    (abi.OTVMC_LJ, 130, 0, True, 900, 1, True), (abi.OTVMC_LJ, 193, 0, True, 1500, 1, False)])
def test_snr_beyond_shared_memory(kind, n, d, pbc, ns, T, down):
    import paper_2506_23928_gb300 as pkg
    model = pkg.Model(pkg.lattice_couplings((n,), 1.0, 1.5, False, pbc), 1.0, 0.1)
    ans = pkg.Ansatz(model, kind, 0, d, pbc)
    P, thr = ans.P, 4.0
    assert P > 96
    sig = synth.random_spins(3 * n, T, ns, n)
    if down:
        sig[:, :, :] = np.where(synth.rng(4).random(sig.shape) < 0.8, -1, sig)
    w = np.full(ns, 1.0 / ns)
    S, D, ob, want, v = [], [], [], [], []
    for t in range(T):
        O = _O(kind, n, d, pbc, sig[t])
        assert O.shape[1] == P
        g = synth.rng(50 + t)
        c = (g.normal(0, 0.02, P) + 1j * g.normal(0, 0.02, P)) / np.maximum(1.0, O.std(0))
        vt = O @ c + 0.1 * (g.normal(0, 1, ns) + 1j * g.normal(0, 1, ns)) + (0.3 - 0.2j)
        cnt = O.sum(0)
        St = (ns * (O.T @ O) - np.outer(cnt, cnt)) / float(ns * ns)
        Dt = O.T @ (vt - vt.mean()) / ns
        S.append(St), D.append(Dt), ob.append(cnt / ns), v.append(vt)
        want.append(tvmc.solve_snr(St, Dt, O, vt, w, snr_thresh=thr, eps_svd=1e-12))
    S_d, ob_d = torch.from_numpy(np.stack(S)).cuda(), torch.from_numpy(np.stack(ob)).cuda()
    sp = torch.from_numpy(synth.pack_spins(sig).view(np.int64)).cuda()
    delta = torch.zeros((T, P, 2), dtype=torch.float64, device="cuda")
    lam = torch.zeros((T, P), dtype=torch.float64, device="cuda")
    nb = abi.otvmc_snr_workspace_bytes(ans.handle, T)
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    check(abi.otvmc_solve_snr(ans.handle, T, ns, S_d, ob_d, sp, to_dev_complex(np.stack(v)), to_dev_complex(np.stack(D)),
                              thr, 1e-12, delta, lam, work, nb))
    check(abi.otvmc_check(work))
    got = from_dev_complex(delta).reshape(T, P)
    for t in range(T):
        l0 = np.linalg.eigvalsh(S[t])
        assert np.abs(np.sort(lam[t].cpu().numpy()) - l0).max() < 1e-12 * l0[-1]
        assert np.abs(got[t] - want[t]).max() < 1e-8 * np.abs(want[t]).max()


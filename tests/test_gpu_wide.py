"""The mixed path's estimators beyond 128 sites and pair moments beyond 64 (k_wide.cu), at the edges
of their groups, chunks of 16 rows, spin words and sample blocks, against the oracle.  The bounds
are those of the mixed path: FP32 sums of n terms."""
import numpy as np
import pytest

import synth
from gpu_helpers import Case, from_dev_complex, rel_err, require_gpu, torch
from oracle import tvmc
from oracle.observables import moments_from_samples
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check

pytestmark = pytest.mark.gpu
MIXED = abi.OTVMC_PREC_MIXED
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("n,ns", [(129, 300), (129, 9), (144, 289), (160, 400), (161, 325), (192, 385), (193, 387), (200, 401)])
def test_estimators_beyond_128_sites(n, ns):
    """Rows past a chunk, sample blocks past a CTA; 9 samples are too few for the records' place."""
    c = Case((n,), h=0.7, kappa=0.1, gamma=0.05)
    T, dt = 2, 0.01
    th, th_d = c.theta(11, T, 0.05)
    sig, sp = c.spins(12, T, ns)
    dW = synth.random_normals(13, (T, c.nops), np.sqrt(dt))
    E = torch.zeros((T, ns, 2), dtype=torch.float64, device="cuda")
    v, lpl = torch.zeros_like(E), torch.zeros((T, c.nops), dtype=torch.float64, device="cuda")
    work, nb = c.work(T, ns, MIXED)
    check(abi.otvmc_local_estimators(c.ans.handle, th_d, sp, T, ns, torch.from_numpy(dW).cuda(), dt, MIXED, E, v, lpl,
                                     work, nb))
    check(abi.otvmc_check(work))
    for t in range(T):
        ev = tvmc.evaluate(c.omodel, c.oans, th[t], sig[t], tvmc.mc_weights(ns), dW[t], dt, with_S=False)
        assert rel_err(from_dev_complex(E)[t, :, 0], ev["E"]) < TOL
        assert rel_err(from_dev_complex(v)[t, :, 0], tvmc.local_v(ev, dW[t], dt)) < TOL
        assert rel_err(lpl.cpu().numpy()[t], ev["lpl"]) < TOL


@pytest.mark.parametrize("n,ns", [(65, 129), (80, 64), (96, 1), (97, 200), (100, 131), (128, 65), (129, 33), (200, 70)])
def test_observables_beyond_64_sites(n, ns):
    """One and two groups a block, a block without samples, chunks with a remainder."""
    c = Case((n,), kappa=0.1)
    T = 2
    th, th_d = c.theta(61, T, 0.05)
    sig, sp = c.spins(62, T, ns)
    mom = torch.zeros((T, 9), dtype=torch.float64, device="cuda")
    work, nb = c.work(T, ns, MIXED)
    check(abi.otvmc_observables(c.ans.handle, th_d, sp, T, ns, MIXED, mom, work, nb))
    check(abi.otvmc_check(work))
    for t in range(T):
        m, q = moments_from_samples(c.oans, th[t], sig[t], tvmc.mc_weights(ns))
        want = np.concatenate([m, q[[0, 1, 2, 0, 0, 1], [0, 1, 2, 1, 2, 2]]])
        assert rel_err(mom.cpu().numpy()[t], want) < TOL

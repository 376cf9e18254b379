"""The FP32 RBM sampler's forms: hidden units at the edges of its lanes (1, 2, 4 and 8 a lane, the table
in shared memory or not), weights small enough for the product form and large enough to need the sum
form and FP64.  Chains are compared bit for bit with the oracle's FP64 decisions."""
import numpy as np
import pytest

from gpu_helpers import require_gpu, torch, unpack
from oracle import tvmc
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check
from test_gpu_rbm import RbmCase

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("scale", [0.01, 0.08, 0.6])
@pytest.mark.parametrize("n,m,ns", [(5, 1, 9), (6, 31, 33), (33, 32, 25), (9, 33, 130), (40, 64, 24), (7, 65, 50),
                                    (73, 97, 26), (65, 128, 12), (10, 129, 40), (66, 200, 9)])
def test_sampler_forms(n, m, ns, scale):
    c = RbmCase(n, m)
    T, traj0, seed, ev, sweeps = 2, 1, 91, 3, 2
    th, th_d = c.theta(4, T, scale)
    sig, sp = c.spins(5, T, ns)
    acc = torch.zeros(T, dtype=torch.int64, device="cuda")
    nb = T * m * ns * 24 + T * n * (40 * m + 8) + 65536
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    check(abi.otvmc_sample(c.ans.handle, th_d, T, traj0, ns, sweeps, seed, ev, sp, acc, work, nb))
    got = unpack(sp, n)
    for t in range(T):
        want, a = tvmc.metropolis(c.oans, th[t], sig[t], seed, traj0 + t, ev, sweeps)
        assert np.array_equal(got[t], want)
        assert int(acc[t]) == int(a.sum())

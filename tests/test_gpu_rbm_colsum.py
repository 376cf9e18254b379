"""Column sums of the RBM's log-derivatives with the samples split over a cluster: sample counts at the
edges of the chunks (32) and of the split, one and two spin words.  The sums are whole numbers, so that
a step of one trajectory and of it in a batch give the same bits whatever the split."""
import numpy as np
import pytest

from gpu_helpers import require_gpu, torch
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check
from test_gpu_rbm import RbmCase

pytestmark = pytest.mark.gpu
MIXED = abi.OTVMC_PREC_MIXED


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _step(c, th_d, sp, T, ns):
    desc = abi.RunDesc(ntraj=T, traj0=0, ns=ns, n_steps=1, step0=0, n_sweep=1, dt=0.01, scheme=abi.OTVMC_HEUN,
                       precision=MIXED, reg=abi.OTVMC_REG_SHIFT, eps=1e-3, snr_thresh=4.0, seed=3, measure_every=0,
                       measure_final=0, use_graph=0)
    nb = abi.otvmc_run_workspace_bytes(c.ans.handle, desc)
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    th, s = th_d.clone(), sp.clone()
    check(abi.otvmc_run_trajectories(c.ans.handle, desc, th, s, None, work, nb))
    check(abi.otvmc_check(work))
    return th.cpu().numpy()


@pytest.mark.parametrize("n,m,ns", [(8, 16, 64), (8, 31, 128), (20, 32, 136), (66, 9, 264), (12, 40, 512)])
def test_split_does_not_change_a_bit(n, m, ns):
    c = RbmCase(n, m)
    T = 40  # a batch that fills the GPU by itself is split less than one trajectory
    th, th_d = c.theta(7, T, 0.02)
    sig, sp = c.spins(8, T, ns)
    many = _step(c, th_d, sp, T, ns)
    one = _step(c, th_d[:1].clone(), sp[:1].clone(), 1, ns)
    assert np.isfinite(many).all()
    assert np.array_equal(many[0], one[0])

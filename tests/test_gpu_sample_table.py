"""The Jastrow sampler's lookup tables: chains equal to the FP64 oracle's, bit for bit, at the
edges of the table widths (N = 102 | 103, 133 | 134, 168 | 169, 200), of the groups per register
and of the spin words, for zero, small and large parameters (wide guard band: the FP64 decision
inside it), polarised chains and ragged sample counts."""
import numpy as np
import pytest

from gpu_helpers import Case, require_gpu, to_dev_complex, unpack, torch
import synth
from oracle import tvmc
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _check(n, ns, scale, polarised=False, sweeps=2):
    c = Case((n,), kappa=0.1)
    T, traj0, seed, ev = 2, 3, 77, 6
    th = synth.random_theta(5 + n, T, c.P, scale)
    th_d = to_dev_complex(th)
    sig = synth.random_spins(6 + n, T, ns, n)
    if polarised:
        sig[:] = -1
    sp = torch.from_numpy(synth.pack_spins(sig).view(np.int64)).cuda()
    acc = torch.zeros(T, dtype=torch.int64, device="cuda")
    work, nb = c.work(T, ns, abi.OTVMC_PREC_MIXED)
    check(abi.otvmc_sample(c.ans.handle, th_d, T, traj0, ns, sweeps, seed, ev, sp, acc, work, nb))
    check(abi.otvmc_check(work))
    got = unpack(sp, n)
    for t in range(T):
        want, na = tvmc.metropolis(c.oans, th[t], sig[t], seed, traj0 + t, ev, sweeps)
        assert np.array_equal(got[t], want)
        assert int(acc[t]) == int(np.sum(na))


@pytest.mark.parametrize("n", [2, 6, 7, 30, 31, 60, 61, 64, 65, 90, 91, 102, 103, 120, 121, 133, 134, 160, 161,
                               168, 169, 180, 181, 200])
def test_sampler_tables_bit_exact(n):
    _check(n, 67, 0.05)


@pytest.mark.parametrize("n,scale,polarised", [(33, 0.0, False), (64, 1.0, False), (100, 0.5, True), (9, 30.0, False),
                                               (140, 1e-6, True)])
def test_sampler_tables_parameter_sizes(n, scale, polarised):
    _check(n, 130, scale, polarised)


def test_sampler_full_blocks():
    _check(24, 1500, 0.1)

"""The SNR filter beyond P = 96 at the ends of its range: directions whose variance is many orders below
that of the others, sample counts and tied sums at which whole-number sums grow large, and more
trajectories than the second dimension of a grid holds."""
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


@pytest.mark.parametrize("ns,a,eps_svd", [(65536, 1e-2, 1e-12), (65536, 1e-2, 0.0), (4096, 0.1, 0.0)])
def test_direction_of_small_variance(ns, a, eps_svd):
    """Two sites that differ in one sample only, whose v lies a times as far from the mean as the others:
    the variance along s_j - s_k is about ns^2 below that of a single spin.  S (any symmetric matrix)
    has that direction as an isolated eigenvector.  Eigenvectors to 8 P 2^-53 move the amplitude there, at
    least sqrt(2) / ns, by a part of 8 P 2^-53 ns of either sign over the samples; the filter is the
    variance's third power."""
    n, j, k, xs, thr = 14, 3, 9, 17, 4.0
    ans = _ansatz(abi.OTVMC_JASTROW, n, 0, False)
    P = ans.P
    sig = synth.random_spins(5, 1, ns, n)
    sig[0, :, k] = sig[0, :, j]
    sig[0, xs, k] = -sig[0, xs, j]
    s = sig[0].astype(np.float64)
    p, q = np.triu_indices(n, 1)
    O = np.concatenate([s, s[:, p] * s[:, q]], 1)
    g = np.random.default_rng(8)
    v = g.normal(0, 1, ns) + 1j * g.normal(0, 1, ns)
    v[xs] = 0
    v -= v.sum() / (ns - 1)
    v[xs] = a * (1 + 0.5j)
    vc = v - v.mean()
    u = np.zeros(P)
    u[j], u[k] = np.sqrt(0.5), -np.sqrt(0.5)
    Q = np.linalg.qr(np.concatenate([u[:, None], g.normal(0, 1, (P, P - 1))], 1))[0]
    S = (Q * np.concatenate([[1e-3], np.linspace(1.0, 3.0, P - 1)])) @ Q.T
    S = 0.5 * (S + S.T)
    obar = O.mean(0)
    y = (O[:, j] - O[:, k]) * np.sqrt(0.5)
    y -= y.mean()
    Qx = y * vc
    rho = Qx.mean()
    var = (np.abs(Qx - rho) ** 2).mean()
    D = u * rho
    got = _snr(ans, torch.from_numpy(S[None]).cuda(), torch.from_numpy(obar[None]).cuda(), _pack(sig),
               to_dev_complex(v[None]), to_dev_complex(D[None]), thr, eps_svd)
    got = u @ from_dev_complex(got).reshape(P)
    snr = np.abs(rho) / np.sqrt(var / ns)
    want = rho / (1 + (thr / snr) ** 6) / (u @ S @ u)
    tol = 3 * (2 * 8 * P * 2.0 ** -53 * ns / np.sqrt(ns) + 2.0 ** -40)
    assert np.abs(got - want) <= tol * np.abs(want)


def test_large_sums():
    """Half the samples polarised, half Neel-ordered on a ring of 200 sites (tied sums of 200 and -200) and
    half a million of them, |v - mean| of one size: centred sums of w O O' of 2^46 200^2 ns^3."""
    n, ns, thr = 200, 500000, 4.0
    ans = _ansatz(abi.OTVMC_LJ, n, 0, True)
    P = ans.P
    conf = np.stack([np.ones(n, np.int8), np.where(np.arange(n) % 2, -1, 1).astype(np.int8)])
    s = conf.astype(np.int64)
    p, q = np.triu_indices(n, 1)
    Dd = np.minimum(q - p, n - (q - p))
    pair = s[:, p] * s[:, q]
    O = np.concatenate([s] + [pair[:, Dd == x].sum(1, keepdims=True) for x in range(1, n // 2 + 1)], 1).astype(np.float64)
    assert O.shape[1] == P and np.abs(O).max() == n
    g = np.random.default_rng(3)
    kind = g.integers(0, 2, ns)
    v = 0.99 * np.exp(2j * np.pi * g.random(ns))
    vc = v - v.mean()
    cnt = np.array([(kind == c).sum() for c in (0, 1)], dtype=np.float64)
    obar = (cnt @ O) / ns
    Oc = O - obar
    vs = np.array([vc[kind == c].sum() for c in (0, 1)])
    w = np.array([(np.abs(vc[kind == c]) ** 2).sum() for c in (0, 1)])
    D = (Oc.T @ vs) / ns
    Q = np.linalg.qr(g.normal(0, 1, (P, P)))[0]
    S = (Q * np.linspace(1.0, 2.0, P)) @ Q.T
    S = 0.5 * (S + S.T)
    sp = torch.from_numpy(synth.pack_spins(conf[None]).view(np.int64)).cuda()[0][torch.from_numpy(kind).cuda()][None]
    got = _snr(ans, torch.from_numpy(S[None]).cuda(), torch.from_numpy(obar[None]).cuda(), sp.contiguous(),
               to_dev_complex(v[None]), to_dev_complex(D[None]), thr, 1e-12)
    got = from_dev_complex(got).reshape(P)
    lam, V = np.linalg.eigh(S)
    y = Oc @ V
    rho = V.T @ D
    var = (w @ y ** 2) / ns - np.abs((vs @ y) / ns) ** 2
    f = 1 / (1 + (thr / (np.abs(rho) / np.sqrt(var / ns))) ** 6)
    want = V @ (f / lam * rho)
    assert np.abs(got - want).max() < 1e-8 * np.abs(want).max()


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


@pytest.mark.parametrize("wild", [False, True])
def test_obar_that_is_no_column_mean(wild):
    """The centring takes obar as it is given: not c / ns, and with an entry far beyond any |O|."""
    n, ns, thr = 14, 700, 1.0
    ans = _ansatz(abi.OTVMC_JASTROW, n, 0, False)
    P = ans.P
    sig = synth.random_spins(5, 1, ns, n)
    s = sig[0].astype(np.float64)
    p, q = np.triu_indices(n, 1)
    O = np.concatenate([s, s[:, p] * s[:, q]], 1)
    g = np.random.default_rng(9)
    obar = O.mean(0) + g.normal(0, 0.1, P)
    if wild:
        obar[40] = 1000.25
    v = g.normal(0, 1, ns) + 1j * g.normal(0, 1, ns)
    Q = np.linalg.qr(g.normal(0, 1, (P, P)))[0]
    S = (Q * np.linspace(1.0, 2.0, P)) @ Q.T
    S = 0.5 * (S + S.T)
    D = g.normal(0, 1, P) + 1j * g.normal(0, 1, P)
    got = _snr(ans, torch.from_numpy(S[None]).cuda(), torch.from_numpy(obar[None]).cuda(), _pack(sig),
               to_dev_complex(v[None]), to_dev_complex(D[None]), thr, 1e-12)
    lam, V = np.linalg.eigh(S)
    Qx = ((O - obar) @ V) * (v - v.mean())[:, None]
    var = (np.abs(Qx) ** 2).mean(0) - np.abs(Qx.mean(0)) ** 2
    rho = V.T @ D
    want = V @ (rho / lam / (1 + (thr / (np.abs(rho) / np.sqrt(var / ns))) ** 6))
    assert np.abs(from_dev_complex(got).reshape(P) - want).max() < 1e-10 * np.abs(want).max()

"""Whole-number sums of the FP8 Gram pass at the ends of the ranges in which they are taken as exact, just
below 2^24: tied rows h of 13 over 99200 samples, and +-1 rows over 2^24 - 1 samples (a multiple of 8 on the mixed path)."""
import numpy as np
import pytest

from gpu_helpers import Case, require_gpu, to_dev_complex, torch
import synth
from paper_2506_23928_gb300 import abi
from paper_2506_23928_gb300.abi import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("order", ["random_last", "random_first", "mixed"])
def test_tied_rows_at_the_most_samples(order):
    """A ring of 200 sites, polarised (tied sums of 200 = 16 * 13 - 8) but for 300 random samples, whose
    products of any size are added to sums near 13 * 13 * 99200 = 2^24 - 12416."""
    import paper_2506_23928_gb300 as pkg
    n, ns, few = 200, 99200, 300
    ans = pkg.Ansatz(pkg.Model(pkg.lattice_couplings((n,), 1.0, 1.5, False, True), 1.0, 0.1), abi.OTVMC_LJ, 0, 0, True)
    g = np.random.default_rng(11)
    sig = np.ones((1, ns, n), np.int8)
    at = {"random_last": np.arange(ns - few, ns), "random_first": np.arange(few),
          "mixed": g.choice(ns, few, replace=False)}[order]
    sig[0, at] = synth.random_spins(12, 1, few, n)[0]
    v = synth.random_normals(13, (1, ns)) + 1j * synth.random_normals(14, (1, ns))
    P = ans.P
    S = torch.zeros((1, P, P), dtype=torch.float64, device="cuda")
    ob = torch.zeros((1, P), dtype=torch.float64, device="cuda")
    D = torch.zeros((1, P, 2), dtype=torch.float64, device="cuda")
    nb = abi.otvmc_workspace_bytes(ans.handle, 1, ns, abi.OTVMC_PREC_FP64)
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    sp = torch.from_numpy(synth.pack_spins(sig).view(np.int64)).cuda()
    check(abi.otvmc_build_S_F(ans.handle, None, sp, to_dev_complex(v), 1, ns, abi.OTVMC_PREC_FP64, S, None, ob, D,
                              work, nb))
    check(abi.otvmc_check(work))
    s = sig[0].astype(np.float32)
    tied = [sum(s[:, j] * s[:, (j + x) % n] for j in range(n if 2 * x < n else x)) for x in range(1, n // 2 + 1)]
    O = np.concatenate([s, np.stack(tied, 1)], 1).astype(np.float64)  # whole numbers, exact in FP32
    assert O.shape[1] == P
    cnt = O.sum(0)
    # below 2^49: exact in FP64
    want = (ns * (O.T @ O) - np.outer(cnt, cnt)) / float(ns) ** 2
    assert np.array_equal(S[0].cpu().numpy(), want)
    assert np.array_equal(ob[0].cpu().numpy(), cnt / ns)


@pytest.mark.parametrize("precision,ns", [(abi.OTVMC_PREC_FP64, (1 << 24) - 1), (abi.OTVMC_PREC_MIXED, (1 << 24) - 8)])
def test_pairs_at_the_most_samples(precision, ns):
    """Three sites: one always up, one up but for 5 samples, one random."""
    n = 3
    c = Case((n,))
    g = np.random.default_rng(21)
    bits = np.full(ns, 1, np.uint64)
    bits |= np.uint64(2)
    bits[g.choice(ns, 5, replace=False)] ^= np.uint64(2)
    bits |= g.integers(0, 2, ns, dtype=np.uint64) << np.uint64(2)
    v = g.normal(0, 1, ns) + 1j * g.normal(0, 1, ns)
    P = c.P
    G = torch.zeros((1, P, P), dtype=torch.float32, device="cuda")
    S = torch.zeros((1, P, P), dtype=torch.float64, device="cuda")
    ob = torch.zeros((1, P), dtype=torch.float64, device="cuda")
    D = torch.zeros((1, P, 2), dtype=torch.float64, device="cuda")
    work, nb = c.work(1, ns, precision)
    sp = torch.from_numpy(bits.view(np.int64).reshape(1, ns, 1)).cuda()
    fp64 = precision == abi.OTVMC_PREC_FP64
    check(abi.otvmc_build_S_F(c.ans.handle, None, sp, to_dev_complex(v[None]), 1, ns, precision, S if fp64 else None,
                              None if fp64 else G, ob, D, work, nb))
    check(abi.otvmc_check(work))
    s = [2.0 * ((bits >> np.uint64(j)) & np.uint64(1)).astype(np.float64) - 1.0 for j in range(n)]
    O = np.stack(s + [s[0] * s[1], s[0] * s[2], s[1] * s[2]], 1)
    cnt, gram = O.sum(0), O.T @ O
    assert np.array_equal(ob[0].cpu().numpy(), cnt / ns)
    if fp64:
        # below 2^48: exact in FP64
        assert np.array_equal(S[0].cpu().numpy(), (ns * gram - np.outer(cnt, cnt)) / float(ns) ** 2)
    else:
        iu = np.triu_indices(P)
        assert np.array_equal(G[0].cpu().numpy().astype(np.float64)[iu], gram[iu])

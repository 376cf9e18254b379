"""S, D and obar of the tied Jastrow from the tensor-core pass (tied rows as 16 h + l) against whole-
number arithmetic on the host: chain and ring, tie distances up to the full Jastrow, spin words and
operand tiles at their edges, ragged and single samples, polarised chains (|O| = N), and one
sample count beyond the tensor-core build's, which takes the integer sums of the CUDA cores."""
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


def _groups(n, d, pbc):
    j, k = np.triu_indices(n, 1)
    D = np.minimum(k - j, n - (k - j)) if pbc else k - j
    free = [[p] for p in np.nonzero(D <= d)[0]]
    return free + [np.nonzero(D == x)[0] for x in range(d + 1, n) if np.any(D == x)]


@pytest.mark.parametrize("n,d,pbc,ns,T,down", [
    (2, 0, True, 16, 2, False), (3, 0, False, 33, 1, False), (10, 1, True, 256, 3, False), (7, 6, False, 20, 1, False),
    (63, 0, True, 100, 2, False), (64, 2, False, 300, 1, False), (65, 1, True, 511, 2, False),
    (100, 1, True, 257, 2, True), (127, 0, True, 1, 1, False), (128, 0, True, 64, 1, False),
    (129, 0, False, 64, 1, True), (200, 0, False, 40, 1, True), (200, 3, True, 48, 1, False),
    (193, 0, True, 1000, 1, False), (4, 0, True, 99208, 1, False)])
def test_tied_build_is_exact(n, d, pbc, ns, T, down):
    import paper_2506_23928_gb300 as pkg
    model = pkg.Model(pkg.lattice_couplings((n,), 1.0, 1.5, False, pbc), 1.0, 0.1)
    ans = pkg.Ansatz(model, abi.OTVMC_LJ, 0, d, pbc)
    sig = synth.random_spins(n + ns, T, ns, n)
    if down:
        sig[0, : max(1, ns - 3)] = -1
    v = synth.random_normals(7, (T, ns)) + 1j * synth.random_normals(8, (T, ns), 0.1)
    P = ans.P
    S = torch.zeros((T, P, P), dtype=torch.float64, device="cuda")
    ob = torch.zeros((T, P), dtype=torch.float64, device="cuda")
    D = torch.zeros((T, P, 2), dtype=torch.float64, device="cuda")
    nb = abi.otvmc_workspace_bytes(ans.handle, T, ns, abi.OTVMC_PREC_FP64)
    work = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    sp = torch.from_numpy(synth.pack_spins(sig).view(np.int64)).cuda()
    check(abi.otvmc_build_S_F(ans.handle, None, sp, to_dev_complex(v), T, ns, abi.OTVMC_PREC_MIXED, S, None, ob, D,
                              work, nb))
    check(abi.otvmc_check(work))
    gotD = from_dev_complex(D).reshape(T, P)
    groups = _groups(n, d, pbc)
    j, k = np.triu_indices(n, 1)
    for t in range(T):
        s = sig[t].astype(np.int64)
        pair = s[:, j] * s[:, k]
        O = np.concatenate([s] + [pair[:, g].sum(1, keepdims=True) for g in groups], 1)
        assert O.shape[1] == P
        cnt = O.sum(0)
        want = (ns * (O.T @ O) - np.outer(cnt, cnt)) / float(ns * ns)
        got = S[t].cpu().numpy()
        if ns <= 99200:
            assert np.array_equal(got, want)
            assert np.array_equal(ob[t].cpu().numpy(), cnt / ns)
        else:
            assert np.abs(got - want).max() < 1e-15 * n * n
            assert np.abs(ob[t].cpu().numpy() - cnt / ns).max() < 1e-15 * n
        vc = v[t] - v[t].mean()
        wantD = (O.T @ vc) / ns
        # quantisation of v to 2^-(60 - log2 ns) of its largest value, and the reference's own FP64 sums
        assert np.abs(gotD[t] - wantD).max() <= np.abs(O).max() * np.abs(v[t]).max() * (ns * 2.0 ** -58 + 2.0 ** -48)

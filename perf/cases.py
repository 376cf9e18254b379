"""Workloads of the library's public entry points, for timing and for comparing two builds.

A case is a dict of plain values; `family` names the entry point (or the short sequence of them)
that one pass calls:

  run          otvmc_run_trajectories: one trajectory step of a batch (whole call; measured, but for
               the learned ansatz, whose users measure on few steps)
  sample       otvmc_sample: Metropolis sweeps of every chain
  estimators   otvmc_local_estimators
  observables  otvmc_observables
  build        otvmc_build_S_F (the tied Jastrow's S and D)
  solve        otvmc_solve_step on a given S (the tied Jastrow's solve)
  snr          otvmc_solve_snr
  linear       otvmc_build_S_F, then otvmc_solve_step on its result

The sizes are those of `synth.WORKLOADS` and `synth.PAPER_WORKLOADS` (lattice, rates, ansatz,
samples per trajectory), with fewer trajectories where a stage is timed alone; `draw` spreads
sizes over the same ranges.  Inputs are made with torch on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

import paper_2506_23928_gb300 as pkg
from paper_2506_23928_gb300 import abi

MIXED, FP64 = "mixed", "fp64"
_PREC = {MIXED: abi.OTVMC_PREC_MIXED, FP64: abi.OTVMC_PREC_FP64}
_CHAIN64 = dict(lx=64, ly=1, J=1.0, alpha=1.5, h=1.0, kappa=0.1, gamma=0.05, pbc=False, kac=False)
_SQUARE10 = dict(lx=10, ly=10, J=1.0, alpha=3.0, h=0.5, kappa=0.05, gamma=0.0, pbc=False, kac=False)
_RING100 = dict(lx=100, ly=1, J=-1.0, alpha=1.0, h=-1.07, kappa=0.27, gamma=0.0, pbc=True, kac=True)
_RING160 = dict(lx=160, ly=1, J=-1.0, alpha=1.0, h=0.0, kappa=0.1, gamma=0.0, pbc=True, kac=True)
_JASTROW = dict(ansatz="jastrow", m=0, d=0)
_LJPH1 = dict(ansatz="lj", m=0, d=1)


def listed():
    return [
        # the smallest run in use: the 8-spin validation quench, where launches are all that counts
        dict(name="run_chain8", family="run", lx=8, ly=1, J=1.0, alpha=1.5, h=1.0, kappa=0.1, gamma=0.0, pbc=False,
             kac=False, **_JASTROW, T=16, ns=1024, dt=0.01, scheme="heun", precision=MIXED, eps=1e-4),
        # the benchmark workload: a step of 256 trajectories of the 64-spin chain
        dict(name="run_chain64", family="run", **_CHAIN64, **_JASTROW, T=256, ns=4096, dt=0.005, scheme="midpoint",
             precision=MIXED, eps=1e-4),
        # the learned ansatz: the chain64_rbm workload at the smallest sample count of its mix
        dict(name="run_chain64_rbm", family="run", **dict(_CHAIN64, gamma=0.0), ansatz="rbm", m=128, d=0, T=16,
             ns=2048, dt=0.005, scheme="midpoint", precision=MIXED, eps=1e-4),
        # sampling a lattice of more than one spin word (square10_jastrow)
        dict(name="sample_square10", family="sample", **_SQUARE10, **_JASTROW, T=128, ns=8192, n_sweep=2),
        # sampling the learned ansatz alone (chain64_rbm)
        dict(name="sample_chain64_rbm", family="sample", **dict(_CHAIN64, gamma=0.0), ansatz="rbm", m=128, d=0, T=8,
             ns=4096, n_sweep=2),
        # local energies of the paper's largest ring (Fig. 2 setup, tied Jastrow)
        dict(name="estimators_ring160", family="estimators", **_RING160, **_LJPH1, T=100, ns=4096, dt=0.005,
             precision=MIXED),
        # magnetisation and covariance at a measurement of the square lattice
        dict(name="observables_square10", family="observables", **_SQUARE10, **_JASTROW, T=64, ns=8192,
             precision=MIXED),
        # the tied Jastrow's geometric tensor (Fig. 3 setup, P = 249)
        dict(name="build_ring100", family="build", **_RING100, **_LJPH1, T=100, ns=4096),
        # its shifted solve at the Fig. 2 setup's P = 399
        dict(name="solve_ring160", family="solve", **_RING160, **_LJPH1, T=100, ns=4096, eps=1e-4),
        # the paper's own regulariser on the Fig. 3 setup
        dict(name="snr_ring100", family="snr", **_RING100, **_LJPH1, T=100, ns=4096, thr=4.0),
        # geometric tensor and solve of the square lattice, the largest full Jastrow (P = 5050)
        dict(name="linear_square10", family="linear", **_SQUARE10, **_JASTROW, T=16, ns=8192, precision=MIXED,
             eps=1e-4),
        # the same two calls in plain FP64 at a size where a user checks against it, a ragged sample count
        dict(name="linear_chain32_fp64", family="linear", **dict(_CHAIN64, lx=32), **_JASTROW, T=8, ns=1001,
             precision=FP64, eps=1e-4),
    ]


# ------------------------------------------------------------------------------- drawn cases

def _params(c):
    n = c["lx"] * c["ly"]
    if c["ansatz"] == "rbm":
        return n + c["m"] + n * c["m"]
    if c["ansatz"] == "jastrow":
        return n * (n + 1) // 2
    return n + len(_groups(n, c["d"], c["pbc"]))


def _size(c):
    """A rough operation count of one pass, used to keep drawn cases below the listed ones."""
    n, T, ns, P, f = c["lx"] * c["ly"], c["T"], c["ns"], _params(c), c["family"]
    m = max(1, c["m"])
    est = ns * n * (n if c["ansatz"] != "rbm" else n * m / 4 + m)
    if f == "sample":
        return T * ns * n * (n + 60) if c["ansatz"] != "rbm" else T * ns * n * (m + 60)
    if f in ("estimators", "observables"):
        return T * est * (6 if c["precision"] == FP64 else 1)
    if f == "build":
        return T * ns * (P * P + n * n)
    if f == "solve":
        return T * (P ** 3 / 3.0 + 1e5)
    if f == "snr":
        return 152 * math.ceil(T / 152) * (8.0 * P ** 3 + ns * P * P)
    if f == "linear":
        return T * (ns * P * P + P ** 3 / 3.0) * (40 if c["precision"] == FP64 else 1)
    # run
    q = min(P, ns) if c["ansatz"] == "rbm" else P
    lin = (ns * P * P if c["ansatz"] != "rbm" else ns * ns * (n + m)) + 3.0 * q ** 3
    return 2 * T * (lin * (40 if c["precision"] == FP64 else 1) + 100 * est)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    base = dict(rng.choice(listed()))
    cap = _size(base) if base["family"] != "run" else _size(listed()[1 if base["ansatz"] != "rbm" else 2])
    name = base.pop("name")
    c = base
    while True:
        # a chain or a ring of any length in the range, or a rectangle
        lo, hi = {"run_chain8": (4, 24), "run_chain64": (24, 64), "run_chain64_rbm": (6, 64),
                  "sample_square10": (6, 160), "sample_chain64_rbm": (6, 64),
                  "estimators_ring160": (8, 160), "observables_square10": (8, 128), "build_ring100": (10, 160), "solve_ring160": (10, 160), "snr_ring100": (8, 100),
                  "linear_square10": (24, 100), "linear_chain32_fp64": (5, 36)}[name]
        c["lx"], c["ly"] = _log_int(rng, lo, hi), 1
        if not c["pbc"] and rng.random() < 0.3:
            c["ly"] = rng.randint(2, 4)
            c["lx"] = max(2, c["lx"] // c["ly"])
        if c["ansatz"] == "lj":
            c["d"] = rng.randint(0, 2)
        if c["ansatz"] == "rbm":
            c["m"] = _log_int(rng, 6, base["m"])
        c["kappa"] = round(rng.uniform(0.05, 0.5), 3)
        if rng.random() < 0.5:
            c["gamma"] = round(rng.uniform(0.01, 0.1), 3)
        if c["family"] == "run":
            c["scheme"] = rng.choice(["heun", "midpoint"])
        if c["family"] in ("estimators", "observables"):
            c["precision"] = rng.choice([MIXED, MIXED, FP64])
        top = {"run_chain8": 2048, "run_chain64_rbm": 2048, "linear_chain32_fp64": 1500}.get(name, max(4096, c["ns"]))
        low = 128
        if c["family"] in ("linear", "solve", "snr") or (c["family"] == "run" and c["ansatz"] != "rbm"):
            low = max(low, _params(c) + 1)  # samples outnumber the parameters
        if low >= top:
            continue
        c["ns"] = _log_int(rng, low, top)
        if c["family"] in ("run", "linear") and c["precision"] == MIXED:
            c["ns"] = -(-c["ns"] // 8) * 8  # the mixed build takes multiples of eight samples
        c["T"] = 1
        most = int(min(512, cap / _size(c)))
        if c["ansatz"] == "rbm":
            most = min(most, int(4.5e10 / (80.0 * max(_params(c), c["ns"]) ** 2)))  # bytes of workspace
        if most >= 1:
            c["T"] = _log_int(rng, 1, most)
            if _size(c) <= cap:
                return c


# ----------------------------------------------------------------------------------- inputs

def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + what) & 0x7FFFFFFFFFFFFFFF)
    return g


def _normal(g, shape, scale=1.0):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g) * scale


def _theta(c, seed):
    """Parameters some way into a quench: phases of the couplings' size, small real parts."""
    P, n = _params(c), c["lx"] * c["ly"]
    g = _gen(seed, 1)
    th = torch.empty((c["T"], P, 2), dtype=torch.float64, device="cuda")
    if c["ansatz"] == "rbm":
        th.copy_(_normal(g, (c["T"], P, 2), 0.01))
        th[:, :n + c["m"]] = 0.0  # the workloads start from small hidden weights alone
    else:
        th[..., 0] = _normal(g, (c["T"], P), 0.02)
        th[..., 1] = _normal(g, (c["T"], P), 0.1)
        th[:, :n, 1] *= 0.2
    return th


def _signs(c, seed):
    """[T][ns][N] configurations, +-1 in int8: neighbouring sites correlated, on average a little down
    (independent and even for the learned ansatz, whose weights are small)."""
    n = c["lx"] * c["ly"]
    g = _gen(seed, 2)
    j = torch.arange(n, device="cuda", dtype=torch.float32)
    rho, edge = (0.0, 0.0) if c["ansatz"] == "rbm" else (0.4, 0.1)
    mix = torch.triu(rho ** (j[None, :] - j[:, None]).clamp(min=0)) * math.sqrt(1 - rho * rho)
    out = torch.empty((c["T"], c["ns"], n), dtype=torch.int8, device="cuda")
    for t in range(c["T"]):
        x = torch.randn((c["ns"], n), device="cuda", generator=g) @ mix
        out[t] = (x > edge).to(torch.int8) * 2 - 1
    return out


def _pack(sig):
    T, ns, n = sig.shape
    W = (n + 63) // 64
    words = torch.zeros((T, ns, W), dtype=torch.int64, device="cuda")
    for j in range(n):
        words[..., j // 64] |= (sig[..., j] > 0).to(torch.int64) << (j % 64)
    return words


def _nops(c):
    n = c["lx"] * c["ly"]
    return (n if c["kappa"] > 0 else 0) + (n if c["gamma"] > 0 else 0)


def _dW(c, seed):
    return _normal(_gen(seed, 3), (c["T"], _nops(c)), math.sqrt(c["dt"]))


def _pairs(n):
    j, k = np.triu_indices(n, 1)
    return j, k


def _groups(n, d, pbc):
    """Pairs that share a parameter of the tied Jastrow, as lists of indices into _pairs(n)."""
    j, k = _pairs(n)
    D = k - j
    if pbc:
        D = np.minimum(D, n - D)
    free = [[int(p)] for p in np.nonzero(D <= d)[0]]
    return free + [[int(p) for p in np.nonzero(D == x)[0]] for x in range(d + 1, n) if np.any(D == x)]


def _group_matrix(c):
    n = c["lx"] * c["ly"]
    groups = _groups(n, c["d"], c["pbc"])
    A = np.zeros((n * (n - 1) // 2, len(groups)), dtype=np.float32)
    for g, grp in enumerate(groups):
        A[grp, g] = 1.0
    return torch.from_numpy(A).cuda()


def _O(c, sig, A):
    """Log-derivatives of one trajectory's samples, [ns][P] in FP64 (small whole numbers)."""
    s = sig.to(torch.float32)
    j, k = (torch.from_numpy(x).cuda() for x in _pairs(s.shape[1]))
    pair = s[:, j] * s[:, k]
    return torch.cat([s, pair if A is None else pair @ A], 1).double()


def _v(c, seed, sig):
    """Local terms v(x) with parts that follow the spins and parts that do not, [T][ns] complex."""
    g = _gen(seed, 4)
    n, T, ns = sig.shape[2], c["T"], c["ns"]
    w = torch.complex(_normal(g, (T, n), 0.01), _normal(g, (T, n), 0.01))
    u = torch.complex(_normal(g, (T, n), 0.01), _normal(g, (T, n), 0.01))
    v = torch.complex(_normal(g, (T, ns), 0.03), _normal(g, (T, ns), 0.03))
    s = sig.double()
    ss = s * torch.roll(s, 1, 2)
    return v + torch.einsum("txn,tn->tx", s + 0j, w) + torch.einsum("txn,tn->tx", ss + 0j, u)


def _S_D(c, sig, v, A, t):
    """S, mean of O, D and centred O of trajectory t in FP64."""
    O = _O(c, sig[t], A)
    ob = O.mean(0)
    Oc = O - ob
    S = Oc.T @ Oc / c["ns"]
    vc = v[t] - v[t].mean()
    D = torch.complex(Oc.T @ vc.real, Oc.T @ vc.imag) / c["ns"]
    return S, ob, D, Oc, vc


def _model(c):
    extent = (c["lx"],) if c["ly"] == 1 else (c["lx"], c["ly"])
    J = pkg.lattice_couplings(extent, c["J"], c["alpha"], c["kac"], c["pbc"])
    model = pkg.Model(J, c["h"], c["kappa"], c["gamma"])
    kind = {"jastrow": abi.OTVMC_JASTROW, "rbm": abi.OTVMC_RBM, "lj": abi.OTVMC_LJ}[c["ansatz"]]
    return J, pkg.Ansatz(model, kind, c["m"], c["d"], c["pbc"])


def _bytes(nb):
    return torch.zeros(nb, dtype=torch.uint8, device="cuda"), nb


def _f64(*shape):
    return torch.zeros(shape, dtype=torch.float64, device="cuda")


def _ri(z):
    return torch.view_as_real(z).contiguous()


def prepare(case, seed):
    c = dict(case)
    _, ans = _model(c)
    T, ns, n, P, f = c["T"], c["ns"], c["lx"] * c["ly"], ans.P, c["family"]
    st = dict(c=c, ans=ans, prec=_PREC[c.get("precision", MIXED)], seed=int(seed))
    if f == "run":
        st["desc"] = abi.RunDesc(
            ntraj=T, traj0=0, ns=ns, n_steps=1, step0=0, n_sweep=2, dt=c["dt"],
            scheme=abi.OTVMC_HEUN if c["scheme"] == "heun" else abi.OTVMC_MIDPOINT, precision=st["prec"],
            reg=abi.OTVMC_REG_SHIFT, eps=c["eps"], snr_thresh=4.0, seed=int(seed),
            measure_every=0 if c["ansatz"] == "rbm" else 1, measure_final=0, use_graph=0)
        st["theta0"], st["spins0"] = _theta(c, seed), _pack(_signs(c, seed))
        st["theta"], st["spins"] = torch.empty_like(st["theta0"]), torch.empty_like(st["spins0"])
        st["mom"] = _f64(1, T, abi.OTVMC_MOMENTS) if c["ansatz"] != "rbm" else None
        st["work"], st["nb"] = _bytes(abi.otvmc_run_workspace_bytes(ans.handle, st["desc"]))
        return st
    if f == "sample":
        st["theta"], st["spins0"] = _theta(c, seed), _pack(_signs(c, seed))
        st["spins"] = torch.empty_like(st["spins0"])
        st["work"], st["nb"] = _bytes(abi.otvmc_workspace_bytes(ans.handle, T, ns, abi.OTVMC_PREC_MIXED))
        return st
    if f == "snr":
        st["work"], st["nb"] = _bytes(abi.otvmc_snr_workspace_bytes(ans.handle, T))
    else:
        st["work"], st["nb"] = _bytes(abi.otvmc_workspace_bytes(ans.handle, T, ns, st["prec"]))
    if f in ("estimators", "observables"):
        st["theta"], st["spins"] = _theta(c, seed), _pack(_signs(c, seed))
        if f == "estimators":
            st["dW"] = _dW(c, seed)
            st["E"], st["v"], st["lpl"] = _f64(T, ns, 2), _f64(T, ns, 2), _f64(T, max(1, _nops(c)))
        else:
            st["mom"] = _f64(T, abi.OTVMC_MOMENTS)
        return st
    sig = _signs(c, seed)
    v = _v(c, seed, sig)
    st["spins"], st["v"] = _pack(sig), _ri(v)
    st["delta"] = _f64(T, P, 2)
    if f in ("solve", "snr"):
        A = _group_matrix(c) if c["ansatz"] == "lj" else None
        st["S"], st["obar"], st["D"] = _f64(T, P, P), _f64(T, P), _f64(T, P, 2)
        for t in range(T):
            S, ob, D, _, _ = _S_D(c, sig, v, A, t)
            st["S"][t], st["obar"][t], st["D"][t] = S, ob, _ri(D)
        st["shift"] = _f64(T)
        return st
    mixed = st["prec"] == abi.OTVMC_PREC_MIXED and c["ansatz"] == "jastrow"
    st["S"] = None if mixed else _f64(T, P, P)  # the mixed Jastrow solve takes the Gram counts
    st["G"] = torch.zeros((T, P, P), dtype=torch.float32, device="cuda") if mixed else None
    st["obar"], st["D"], st["shift"] = _f64(T, P), _f64(T, P, 2), _f64(T)
    return st


def run(st):
    c, h, prec = st["c"], st["ans"].handle, st["prec"]
    T, ns, f = c["T"], c["ns"], c["family"]
    if f == "run":
        # a step from the given state, which stays as it is
        st["theta"].copy_(st["theta0"])
        st["spins"].copy_(st["spins0"])
        abi.check(abi.otvmc_run_trajectories(h, st["desc"], st["theta"], st["spins"], st["mom"], st["work"], st["nb"]))
        return [st["theta"], st["spins"], st["mom"]]
    if f == "sample":
        st["spins"].copy_(st["spins0"])
        abi.check(abi.otvmc_sample(h, st["theta"], T, 0, ns, c["n_sweep"], st["seed"], 2, st["spins"], None,
                                   st["work"], st["nb"]))
        return [st["spins"]]
    if f == "estimators":
        abi.check(abi.otvmc_local_estimators(h, st["theta"], st["spins"], T, ns, st["dW"], c["dt"], prec, st["E"],
                                             st["v"], st["lpl"], st["work"], st["nb"]))
        return [st["E"], st["v"], st["lpl"]]
    if f == "observables":
        abi.check(abi.otvmc_observables(h, st["theta"], st["spins"], T, ns, prec, st["mom"], st["work"], st["nb"]))
        return [st["mom"]]
    if f == "snr":
        abi.check(abi.otvmc_solve_snr(h, T, ns, st["S"], st["obar"], st["spins"], st["v"], st["D"], c["thr"], 1e-12,
                                      st["delta"], None, st["work"], st["nb"]))
        return [st["delta"]]
    if f in ("build", "linear"):
        abi.check(abi.otvmc_build_S_F(h, None, st["spins"], st["v"], T, ns, prec, st["S"], st["G"], st["obar"],
                                      st["D"], st["work"], st["nb"]))
        if f == "build":
            return [st["S"], st["obar"], st["D"]]
    abi.check(abi.otvmc_solve_step(h, T, ns, prec, abi.OTVMC_REG_SHIFT, c["eps"], 0.0, st["S"], st.get("G"), st["obar"],
                                   st["D"], st["delta"], st["shift"], st["work"], st["nb"]))
    if f == "solve":
        return [st["delta"], st["shift"]]
    return [st["obar"], st["D"], st["delta"], st["shift"]] + ([st["S"]] if st["S"] is not None else [])


# ----------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Inputs read once, outputs written once, and the method's multiply-adds (complex ones as four)."""
    c = case
    n, T, ns, P, f = c["lx"] * c["ly"], c["T"], c["ns"], _params(c), c["family"]
    W = (n + 63) // 64
    spins, theta, m = 8.0 * T * ns * W, 16.0 * T * P, max(1, c["m"])
    # one proposal reads a field, one in about two updates them all
    sample = 2.0 * n * ns * T * (n if c["ansatz"] != "rbm" else 8 * m)
    fields = ns * T * n * (6.0 * n if c["ansatz"] != "rbm" else 8.0 * m + 8)
    pairs = 8.0 * ns * T * n * n * (1 if c["ansatz"] != "rbm" else m)
    if f == "sample":
        return {"bytes": theta + 2 * spins, "flops": sample}
    if f == "estimators":
        return {"bytes": theta + spins + 8.0 * T * _nops(c) * 2 + 32.0 * T * ns, "flops": fields}
    if f == "observables":
        return {"bytes": theta + spins + 72.0 * T, "flops": fields + pairs}
    gram, chol = 1.0 * ns * T * P * (P + 1) + 4.0 * ns * T * P, T * (P ** 3 / 3.0 + 4.0 * P * P)
    mats, vecs = 8.0 * T * P * P, 24.0 * T * P
    if f == "build":
        return {"bytes": spins + 16.0 * T * ns + mats + vecs, "flops": gram}
    if f == "solve":
        return {"bytes": mats + 2 * 16.0 * T * P, "flops": chol}
    if f == "snr":
        # tridiagonalisation, eigenvectors, projections of every sample
        return {"bytes": mats + spins + 16.0 * T * ns + 40.0 * T * P,
                "flops": T * (4.0 / 3 + 2.0 + 3.0) * P ** 3 + 2.0 * T * ns * P * P}
    if f == "linear":
        return {"bytes": spins + 16.0 * T * ns + vecs + 16.0 * T * P + (mats if c["precision"] == FP64 else 0),
                "flops": gram + chol}
    if c["ansatz"] == "rbm" and P > ns:
        lin = T * (8.0 * ns * ns * m / 2 + (2 * ns) ** 3 / 3.0)
    elif c["ansatz"] == "rbm":
        lin = T * (4.0 * ns * P * P + (2.0 * P) ** 3 / 3.0)
    else:
        lin = gram + chol
    return {"bytes": 2 * theta + 2 * spins + 72.0 * T, "flops": 2 * (sample + fields + lin) + pairs}


# ------------------------------------------------------------------------------ the same in 64 bits

def _fields(c, J, theta, sig):
    """Flip ratios r_j(x) [ns][N] of one trajectory and the coupling matrix eta."""
    n = sig.shape[1]
    th = torch.view_as_complex(theta)
    pj, pk = (torch.from_numpy(x).cuda() for x in _pairs(n))
    eta = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    pair = th[n:]
    if c["ansatz"] == "lj":
        idx = np.empty(n * (n - 1) // 2, dtype=np.int64)
        for g, grp in enumerate(_groups(n, c["d"], c["pbc"])):
            idx[grp] = g
        pair = pair[torch.from_numpy(idx).cuda()]
    eta[pj, pk] = pair
    eta = eta + eta.T
    s = sig.double()
    f = th[:n] + torch.complex(s @ eta.real, s @ eta.imag)
    return torch.exp(-2.0 * s * f), eta, s


def _exact_estimators(c, J, seed):
    theta, sig, dW = _theta(c, seed), _signs(c, seed), _dW(c, seed)
    T, ns, n = sig.shape
    Jt = torch.from_numpy(np.ascontiguousarray(J)).cuda()
    E, v = _f64(T, ns, 2), _f64(T, ns, 2)
    lpl = _f64(T, max(1, _nops(c)))
    nd = n if c["kappa"] > 0 else 0
    for t in range(T):
        r, _, s = _fields(c, Jt, theta[t], sig[t])
        EH = 0.5 * ((s @ Jt) * s).sum(1) + c["h"] * r.sum(1)
        down = 0.5 * (1.0 - s)  # where sigma^- leads to
        bracket = torch.zeros(ns, dtype=torch.complex128, device="cuda")
        vt = torch.zeros(ns, dtype=torch.complex128, device="cuda")
        if c["kappa"] > 0:
            B = math.sqrt(c["kappa"]) * down * r
            l = (math.sqrt(c["kappa"]) * r).mean(0).real
            lpl[t, :n] = l
            bracket = bracket + (c["kappa"] * 0.5 * (1.0 + s) - 2.0 * l * B).sum(1)
            vt = vt + (B * dW[t, :n]).sum(1)
        if c["gamma"] > 0:
            B = math.sqrt(c["gamma"]) * s
            l = 2.0 * B.mean(0)
            lpl[t, nd:nd + n] = l
            bracket = bracket + (2.0 * c["gamma"] - 2.0 * l * B).sum(1)
            vt = vt + (B * dW[t, nd:nd + n]).sum(1)
        Ee = EH - 0.5j * bracket
        E[t], v[t] = _ri(Ee), _ri(vt - 1j * c["dt"] * Ee)
    return [E, v, lpl]


def _exact_observables(c, J, seed):
    theta, sig = _theta(c, seed), _signs(c, seed)
    T, ns, n = sig.shape
    mom = _f64(T, abi.OTVMC_MOMENTS)
    off = 1.0 - torch.eye(n, dtype=torch.float64, device="cuda")
    for t in range(T):
        r, eta, s = _fields(c, None, theta[t], sig[t])
        Ep, Em = torch.exp(4.0 * eta) * off, torch.exp(-4.0 * eta) * off
        u, d = r * (s > 0), r * (s < 0)  # the ratio of two flips is r_j r_k exp(+-4 eta_jk)
        uu, dd = ((u @ Ep) * u).sum(1), ((d @ Ep) * d).sum(1)
        ud = ((u @ Em) * d).sum(1)
        tot, srt, sr = s.sum(1), (s * r).sum(1), r.sum(1)
        q = [uu + dd + 2 * ud, -(uu + dd - 2 * ud), tot * tot - n, -1j * (uu - dd), tot * sr - srt,
             -1j * (srt * tot - sr)]
        q = [x.mean() for x in q]
        m = [sr.mean(), (-1j * srt).mean(), tot.mean()]
        row = [float(x.real) / n for x in m] + [(float(x.real) + (n if i < 3 else 0)) / n ** 2 for i, x in enumerate(q)]
        mom[t] = torch.tensor(row, dtype=torch.float64)
    return [mom]


def _exact_linear(c, seed):
    f = c["family"]
    sig = _signs(c, seed)
    v = _v(c, seed, sig)
    A = _group_matrix(c) if c["ansatz"] == "lj" else None
    T, P = c["T"], _params(c)
    keep_S = f == "build" or (f == "linear" and c["precision"] == FP64)
    Ss = _f64(T, P, P) if keep_S else None
    obar, Ds, delta, shift = _f64(T, P), _f64(T, P, 2), _f64(T, P, 2), _f64(T) + c.get("eps", 0.0)
    for t in range(T):
        S, ob, D, Oc, vc = _S_D(c, sig, v, A, t)
        obar[t], Ds[t] = ob, _ri(D)
        if keep_S:
            Ss[t] = S
        if f == "build":
            continue
        if f == "snr":
            lam, V = (x.cuda() for x in torch.linalg.eigh(S.cpu()))
            rho = torch.complex(V.T @ D.real, V.T @ D.imag)
            proj = Oc @ V
            q2 = (proj ** 2 * (vc.real ** 2 + vc.imag ** 2)[:, None]).mean(0)
            var = q2 - rho.real ** 2 - rho.imag ** 2
            snr = rho.abs() / torch.sqrt(var / c["ns"] + 1e-300)
            filt = 1.0 / (1.0 + (c["thr"] / snr) ** 6) / (1.0 + (1e-12 * lam.max() / lam.clamp(min=1e-300)) ** 6)
            w = torch.where(lam > 0, filt / lam.clamp(min=1e-300), torch.zeros_like(lam)) * rho
            x = torch.complex(V @ w.real, V @ w.imag)
        else:
            S.diagonal().add_(c["eps"])
            L = torch.linalg.cholesky(S)
            x = torch.cholesky_solve(torch.stack([D.real, D.imag], 1), L)
            x = torch.complex(x[:, 0].contiguous(), x[:, 1].contiguous())
        delta[t] = _ri(x)
    if f == "build":
        return [Ss, obar, Ds]
    if f == "solve":
        return [delta, shift]
    if f == "snr":
        return [delta]
    return [obar, Ds, delta, shift] + ([Ss] if keep_S else [])


def exact(case, seed):
    c, f = dict(case), case["family"]
    if f in ("run", "sample"):
        return None  # whole steps, whose samples decide the rest; bits
    if f in ("estimators", "observables"):
        extent = np.array([[i, j] for i in range(c["lx"]) for j in range(c["ly"])], dtype=np.float64)
        dist = np.abs(extent[:, None] - extent[None])
        if c["pbc"]:
            dist = np.minimum(dist, np.array([c["lx"], c["ly"]], dtype=np.float64) - dist)
        r = np.sqrt((dist ** 2).sum(-1))
        J = np.where(r > 0, c["J"] * np.where(r > 0, r, 1.0) ** -c["alpha"], 0.0)
        if c["kac"]:
            J = J / (np.sum(r[np.triu_indices(len(r), 1)] ** -c["alpha"]) / (len(r) - 1))
        return _exact_estimators(c, J, seed) if f == "estimators" else _exact_observables(c, J, seed)
    return _exact_linear(c, seed)

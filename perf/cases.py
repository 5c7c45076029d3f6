"""Performance cases of the library: what its users have it compute.

A case is a dict of plain values.  listed() names the workloads themselves,
draw(rng) gives further ones of the same ranges, prepare(case, seed) builds
what a program holds before the call (operators, a resident system or batch,
device arrays), run(state) is one pass through the public entry points,
work(case) counts what a pass cannot do without, and exact(case, seed) is the
same result from plain torch in 64 bits: matrix exponentials and Taylor
series of the Liouvillian in place of an adaptive integrator, and the
Monte-Carlo trajectories from exact propagators with jump times to 2^-50 of
an output interval.

The mixed-precision mode (QT_MIXED) propagates complex64 states, so its
results are kept as complex64; FP64 results stay complex128.
"""
import math

import numpy as np
import torch

from paper_1110_0573_gb300 import qt
from paper_1110_0573_gb300 import systems as S

DEV = "cuda"
# rtol, atol of each precision, as in the benchmark's workloads
TOL = {"fp64": (1e-8, 1e-10), "mixed": (1e-7, 1e-9)}


def listed():
    return [
        # the smallest call: the paper's single-photon cavity decay (section
        # 3.2.1) as one host-memory qt_mesolve, operators and all, as a script
        # or a notebook calls it
        dict(name="decay_host", kind="decay", N=5, n_t=100, precision="fp64"),
        # one small master equation with its density matrices at every output:
        # the Jaynes-Cummings model of section 4.2, dim 20, on a resident system
        dict(name="jc_me", kind="jc_me", N=10, t_end=50.0, n_t=201, precision="fp64"),
        # its Monte-Carlo counterpart through host memory, with jump records
        dict(name="jc_mc_host", kind="jc_mc", N=10, t_end=50.0, n_t=201, ntraj=500),
        # many trajectories of one mid-size system: the driven Kerr cavity,
        # dim 64 (the benchmark's headline workload)
        dict(name="kerr_mc", kind="kerr_mc", N=64, n_t=401, ntraj=16384, precision="mixed"),
        # the same with a drive that is ramped on: a time-dependent Hamiltonian
        dict(name="kerr_ramp_mc", kind="kerr_ramp_mc", N=64, n_t=401, ntraj=16384,
             precision="mixed"),
        # trajectories of a large sparse system: the dissipative XXZ chain, dim 1024
        dict(name="xxz_mc", kind="xxz_mc", L=10, n_t=101, ntraj=4096, precision="mixed"),
        # the master equation of the same chain on a dense 1024 x 1024 matrix
        dict(name="xxz_me", kind="xxz_me", L=10, n_t=101, precision="mixed"),
        # a dense Hamiltonian, where the products belong on the tensor cores;
        # returns the density matrices
        dict(name="dense_me", kind="dense_me", d=1024, t_end=0.5, n_t=6),
        # a parameter sweep: many uneven small systems, half master equation
        # and half Monte Carlo, in one batched launch
        dict(name="sweep", kind="sweep", n=512, ntraj=256, n_t=121),
        # gradients of a pulse-optimisation loss, forward and backward, through
        # the autograd function: transmon and cavity, dim 60, 256 drive vectors
        dict(name="transmon_grad", kind="grad", N=20, batch=256, n_seg=16),
        # two-time correlation functions of the Jaynes-Cummings model
        dict(name="jc_corr", kind="corr", N=10, n_t=304, n_tau=151, precision="fp64"),
        # the steady state of the Kerr cavity through host memory
        dict(name="kerr_ss_host", kind="ss", N=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above; long times shrink as systems grow,
    so that no drawn case costs more than the largest listed one."""
    kind = rng.choice(["decay", "jc_me", "jc_mc", "kerr_mc", "kerr_ramp_mc", "xxz_mc", "xxz_me",
                       "dense_me", "sweep", "grad", "corr", "ss"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "decay":
        return dict(kind=kind, N=_log_int(rng, 3, 24), n_t=_log_int(rng, 20, 300), precision=prec)
    if kind == "jc_me":
        N = rng.randint(3, 30)
        return dict(kind=kind, N=N, t_end=round(50.0 * min(1.0, (8.0 / N) ** 3.5), 3),
                    n_t=rng.randint(11, 201), precision=prec)
    if kind == "jc_mc":
        N = rng.randint(3, 30)
        return dict(kind=kind, N=N, t_end=round(50.0 * min(1.0, (10.0 / N) ** 2), 3),
                    n_t=rng.randint(51, 301), ntraj=_log_int(rng, 20, 1000))
    if kind == "kerr_mc":
        top = 512 if prec == "fp64" else 16384
        return dict(kind=kind, N=_log_int(rng, 8, 128), n_t=rng.randint(101, 401),
                    ntraj=_log_int(rng, 64, top), precision=prec)
    if kind == "kerr_ramp_mc":
        top = 512 if prec == "fp64" else 8192
        return dict(kind=kind, N=_log_int(rng, 8, 80), n_t=rng.randint(101, 401),
                    ntraj=_log_int(rng, 64, top), precision=prec)
    if kind == "xxz_mc":
        top = 128 if prec == "fp64" else 4096
        return dict(kind=kind, L=rng.randint(4, 10), n_t=rng.randint(21, 101),
                    ntraj=_log_int(rng, 32, top), precision=prec)
    if kind == "xxz_me":
        return dict(kind=kind, L=rng.randint(4, 10), n_t=rng.randint(11, 101), precision=prec)
    if kind == "dense_me":
        return dict(kind=kind, d=_log_int(rng, 96, 1024), t_end=round(rng.uniform(0.2, 0.6), 3),
                    n_t=rng.randint(2, 6))
    if kind == "sweep":
        return dict(kind=kind, n=_log_int(rng, 64, 512), ntraj=_log_int(rng, 24, 256),
                    n_t=rng.randint(31, 121))
    if kind == "grad":
        return dict(kind=kind, N=rng.randint(4, 20), batch=_log_int(rng, 16, 256),
                    n_seg=rng.randint(4, 16))
    if kind == "corr":
        return dict(kind=kind, N=rng.randint(3, 12), n_t=_log_int(rng, 16, 304),
                    n_tau=rng.randint(21, 151), precision=prec)
    return dict(kind=kind, N=rng.randint(8, 72))


# ------------------------------------------------------------------ inputs


def _vary(seed):
    """A factor near one per call, from the seed alone."""
    g = np.random.Generator(np.random.Philox(seed))
    return lambda: float(g.uniform(0.95, 1.05))


def _system(case, seed):
    """The system of a case: the operator library's model with its parameters
    moved by up to 5 % by the seed."""
    v, kind = _vary(seed), case["kind"]
    if kind == "decay":
        return S.cavity_thermal_decay(N=case["N"], kappa=v() / 0.129, nth=0.063 * v(),
                                      nt=case["n_t"])
    if kind in ("jc_me", "jc_mc", "corr"):
        t = dict(t_end=case["t_end"], nt=case["n_t"]) if kind != "corr" else {}
        return S.jaynes_cummings(N=case["N"], g=2 * np.pi * 0.05 * v(), kappa=0.005 * v(),
                                 gamma=0.05 * v(), n0=case["N"] // 2, **t)
    if kind in ("kerr_mc", "kerr_ramp_mc", "ss"):
        drive = v()
        s = S.kerr_cavity(N=case["N"], Delta=0.5 * v(), K=0.1 * v(),
                          E=0.0 if kind == "kerr_ramp_mc" else drive, kappa=0.5 * v(),
                          nth=0.1 * v(), nt=case.get("n_t", 2))
        if kind == "kerr_ramp_mc":  # f(t) (a + a^dag), f rising from 0 on [0, 5]
            a = S.destroy(case["N"])
            s["td"] = [((a + a.T.conj()).tocsr(), np.array([0.0, 5.0]), np.array([0.0, drive]))]
        return s
    if kind in ("xxz_mc", "xxz_me"):
        return S.xxz_chain(L=case["L"], Delta=0.5 * v(), h=0.3 * v(), gamma_deph=0.05 * v(),
                           gamma_damp=0.02 * v(), nt=case["n_t"])
    if kind == "dense_me":
        return S.dense_random_hamiltonian(d=case["d"], seed=seed, gamma=0.1 * v(),
                                          t_end=case["t_end"], nt=case["n_t"])
    raise ValueError(kind)


def _opts(case):
    prec = case.get("precision", "mixed" if case["kind"] in ("dense_me", "sweep") else "fp64")
    rtol, atol = (1e-6, 1e-8) if case["kind"] in ("dense_me", "sweep", "xxz_me") else TOL[prec]
    if prec == "fp64":
        rtol, atol = TOL["fp64"]
    return dict(rtol=rtol, atol=atol,
                precision=qt.QT_MIXED if prec == "mixed" else qt.QT_FP64,
                me_method=qt.QT_ME_DENSE_TC if case["kind"] == "dense_me" else qt.QT_ME_AUTO)


def _dev(a, dtype=torch.complex128):
    return torch.tensor(np.asarray(a), dtype=dtype, device=DEV)


def _grad_inputs(case, seed):
    v = _vary(seed)
    s = S.transmon_cavity(N=case["N"], T1=20.0 * v(), T2=15.0 * v(), kappa=0.001 * v(),
                          n_seg=case["n_seg"])
    return s, S.drive_vectors(case["batch"], case["n_seg"], seed=seed), \
        np.tile(s["gamma"], (case["batch"], 1))


def _sweep_inputs(case, seed):
    return S.cavity_qubit_sweep(n_instances=case["n"], seed=seed, ntraj=case["ntraj"],
                                nt=case["n_t"])


def prepare(case, seed):
    kind = case["kind"]
    o = qt.qt_opts_default(**_opts(case))
    st = dict(case=case, seed=seed, opts=o, mixed=o.precision == qt.QT_MIXED)
    if kind == "grad":
        s, omega, gamma = _grad_inputs(case, seed)
        st["adjoint"] = qt.Adjoint(s["H0"], s["Hd"], s["A"], s["P1"], s["P2"], s["psi0"],
                                   s["n_seg"], s["t_seg"], case["batch"], max_per_seg=64)
        st["omega"] = _dev(omega, torch.float64).requires_grad_(True)
        st["gamma"] = _dev(gamma, torch.float64).requires_grad_(True)
        return st
    if kind == "sweep":
        problems, tlist = _sweep_inputs(case, seed)
        st["batch"] = qt.Batch(problems)
        st["tlist"] = _dev(tlist, torch.float64)
        st["expect"] = torch.zeros(case["n"] * case["n_t"] * 2, dtype=torch.complex128, device=DEV)
        return st
    s = _system(case, seed)
    st["sys"] = s
    if kind in ("decay", "jc_mc", "ss"):  # host-memory calls take the operators themselves
        return st
    d, n_t = s["H"].shape[0], len(s["tlist"])
    st["tlist"] = _dev(s["tlist"], torch.float64)
    st["psi0"] = _dev(s["psi0"])
    if kind == "corr":
        a = S.tensor(S.destroy(case["N"]), S.qeye(2))
        st["system"] = qt.System(s["H"], s["c_ops"], [S.dag(a), a])
        st["tlist"] = _dev(np.linspace(0.0, 30.0, case["n_t"]), torch.float64)
        st["taulist"] = _dev(np.linspace(0.0, 30.0, case["n_tau"]), torch.float64)
        st["corr"] = torch.zeros((case["n_t"], case["n_tau"], 2), dtype=torch.complex128, device=DEV)
        return st
    st["system"] = qt.System(s["H"], s["c_ops"], s["e_ops"], td=s.get("td"))
    st["expect"] = torch.zeros((n_t, len(s["e_ops"])), dtype=torch.complex128, device=DEV)
    if kind in ("jc_me", "dense_me"):
        st["states"] = torch.zeros((n_t, d, d), dtype=torch.complex128, device=DEV)
    return st


def _jump_table(case, traj, k, channel, tau):
    """The jump records as arrays with a row per trajectory (channel -1, time
    0 past its last jump): no more jumps than quanta in the initial state."""
    ch = np.full((case["ntraj"], case["N"] // 2 + 2), -1, dtype=np.int64)
    at = np.zeros(ch.shape)
    ch[traj, k], at[traj, k] = channel, tau
    return ch, at


def run(st):
    kind, o = st["case"]["kind"], st["opts"]
    if kind == "decay":
        s = st["sys"]
        out = [qt.qt_mesolve(s["H"], s["c_ops"], s["e_ops"], s["psi0"], s["tlist"], opts=o)[0]]
        return [x.astype(np.complex64) for x in out] if st["mixed"] else out
    if kind == "jc_mc":
        s = st["sys"]
        mean, _, jumps, _ = qt.qt_mcsolve(s["H"], s["c_ops"], s["e_ops"], s["psi0"], s["tlist"],
                                          st["case"]["ntraj"], seed=st["seed"], opts=o)
        return [mean, *_jump_table(st["case"], jumps["traj"], jumps["k"], jumps["channel"],
                                   jumps["tau"])]
    if kind == "ss":
        return [qt.qt_steadystate(st["sys"]["H"], st["sys"]["c_ops"])[0]]
    if kind == "grad":
        loss = qt.master_equation_loss(st["adjoint"], st["omega"], st["gamma"], o)
        return [loss.detach(), *torch.autograd.grad(loss.sum(), (st["omega"], st["gamma"]))]
    if kind == "sweep":
        st["batch"].qt_batch_solve_dev(st["tlist"], o, st["expect"])
        per_problem = st["expect"].view(st["case"]["n"], st["case"]["n_t"], 2)
        out = [per_problem[0::2], per_problem[1::2]]  # master equation, Monte Carlo
    elif kind == "corr":
        st["system"].qt_correlation_2op_2t_dev(st["psi0"], st["tlist"], st["taulist"], 1, o,
                                               st["corr"])
        out = [st["corr"]]
    elif kind in ("kerr_mc", "kerr_ramp_mc", "xxz_mc"):
        st["system"].qt_mcsolve_dev(st["psi0"], st["tlist"], st["case"]["ntraj"], st["seed"], o,
                                    st["expect"])
        out = [st["expect"]]
    else:
        st["system"].qt_mesolve_dev(st["psi0"], st["tlist"], o, st["expect"], st.get("states"))
        out = [st["expect"]] + ([st["states"]] if "states" in st else [])
    return [x.to(torch.complex64) for x in out] if st["mixed"] else out


# -------------------------------------------------------------------- work

# The largest frequency that the solution of each model carries (its
# eigenvalue spread where the explicit method's stability sets the step), from
# which the number of right-hand sides of a Dormand-Prince solve follows: six
# per step of length 6 rtol^(1/5) / frequency.
_FREQ = {"decay": lambda c: 9.0 * c["N"], "jc_me": lambda c: 3.1 * c["N"],
         "jc_mc": lambda c: 3.1 * c["N"], "corr": lambda c: 3.1 * c["N"],
         "kerr_mc": lambda c: max(8.0, 24.0 * (c["N"] / 64) ** 2),
         "kerr_ramp_mc": lambda c: max(8.0, 24.0 * (c["N"] / 64) ** 2),
         "xxz_mc": lambda c: 0.85 * c["L"], "xxz_me": lambda c: 0.85 * c["L"],
         "dense_me": lambda c: 0.1 * c["d"], "sweep": lambda c: 9.0, "grad": lambda c: 0.75}
_TEND = {"decay": 0.6, "kerr_mc": 20.0, "kerr_ramp_mc": 20.0, "xxz_mc": 10.0, "xxz_me": 10.0,
         "sweep": 30.0, "corr": 30.0}


def work(case):
    """Bytes of the inputs and outputs, and flops: right-hand sides times 8
    per stored entry of H_eff (twice for a density matrix, both sides) and per
    collapse term, plus the Dormand-Prince combinations (11 multiply-adds per
    real component and right-hand side)."""
    kind = case["kind"]
    if kind == "ss":  # one product with the Liouvillian per Krylov vector, d^2 entries each
        n = case["N"] ** 2
        steps = 7.0 * case["N"]
        return {"bytes": 16 * n, "flops": steps * n * (8 * 7 + 16 * steps)}
    n_rhs = 6 * _FREQ[kind](case) * case.get("t_end", _TEND.get(kind, case.get("n_seg", 0.0))) \
        / (6.0 * _opts(case)["rtol"] ** 0.2)
    if kind == "sweep":  # cutoffs 4..32: mean d 36, mean d^2 1560
        per = 0.5 * case["n"] * (1560 * (8 * 9 + 44) + case["ntraj"] * 36 * (8 * 4 + 44))
        return {"bytes": 32 * case["n"] * case["n_t"], "flops": n_rhs * per}
    if kind == "grad":  # a step forward, its stages again, and their adjoints
        d = 3 * case["N"]
        per = case["batch"] * d * d * (8 * 9 + 44) * 3
        return {"bytes": 16 * case["batch"] * (case["n_seg"] + 4), "flops": n_rhs * per}
    if kind == "dense_me":
        d, w, wc = case["d"], case["d"], 2
    elif kind in ("xxz_mc", "xxz_me"):
        d, w, wc = 2 ** case["L"], 1.5 * case["L"], 2 * case["L"]
    else:
        d = case["N"] * (2 if kind in ("jc_me", "jc_mc", "corr") else 1)
        w, wc = (1 if kind == "decay" else 2 if d == 2 * case["N"] else 3), 2
    n_e = {"decay": 1, "xxz_mc": case.get("L"), "xxz_me": case.get("L")}.get(kind, 2)
    if kind in ("jc_mc", "kerr_mc", "kerr_ramp_mc", "xxz_mc"):
        return {"bytes": 16 * (d * (w + wc + 1) + case["n_t"] * n_e),
                "flops": n_rhs * case["ntraj"] * d * (8 * w + 44)}
    # a Hermitian state needs one side of the product and one triangle
    flops = n_rhs * d * d * (8 * w + 4 * wc + 22)
    out = 16 * case["n_t"] * (n_e + (d * d if kind in ("jc_me", "dense_me") else 0))
    if kind == "corr":
        flops = case["n_t"] * n_rhs * d * d * (16 * w + 8 * wc + 44)
        out = 32 * case["n_t"] * case["n_tau"]
    return {"bytes": 16 * d * (w + wc + 1) + out, "flops": flops}


# ------------------------------------------- the same results in 64 bits


def _dense(m):
    return torch.tensor(m.toarray(), dtype=torch.complex128, device=DEV)


class _Liouvillian:
    """L(X) = -i (H_eff X - X H_eff^dag) + sum_n C_n X C_n^dag on [..., d, d]."""

    def __init__(self, H, c_ops):
        heff = H.astype(np.complex128)
        self.jumps, diag = [], 0.0
        for c in c_ops:
            heff = heff - 0.5j * (c.conj().T @ c)
            c = c.tocsr()
            if np.diff(c.indptr).max(initial=0) > 1:
                self.jumps.append(_dense(c))
                continue
            idx, val = np.arange(c.shape[0]), np.zeros(c.shape[0], dtype=np.complex128)
            rows = np.flatnonzero(np.diff(c.indptr))
            idx[rows], val[rows] = c.indices, c.data
            if np.array_equal(idx[rows], rows):
                diag = diag + np.outer(val, val.conj())
            else:
                self.jumps.append((torch.tensor(idx, device=DEV), _dev(np.outer(val, val.conj()))))
        self.diag = None if np.ndim(diag) == 0 else _dev(diag)
        self.K = -1j * _dense(heff)
        self.Kd = self.K.conj().T.contiguous()
        self.bound = 2.0 * float(abs(heff).sum(axis=1).max()) + sum(
            float(abs(c).sum(axis=1).max()) * float(abs(c).sum(axis=0).max()) for c in c_ops)

    def __call__(self, X):
        out = self.K @ X + X @ self.Kd
        if self.diag is not None:
            out += self.diag * X
        for j in self.jumps:
            if torch.is_tensor(j):
                out += j @ X @ j.conj().T
            else:
                idx, w = j
                out += w * X[..., idx, :][..., :, idx]
        return out

    def matrix(self):
        d = self.K.shape[0]
        E = torch.eye(d * d, dtype=torch.complex128, device=DEV).reshape(d * d, d, d)
        return self(E).reshape(d * d, d * d).T.contiguous()


def _taylor(apply, X, dt, bound):
    """exp(dt L) X by Taylor steps of norm at most 3."""
    n = max(1, math.ceil(bound * dt / 3.0))
    h = dt / n
    for _ in range(n):
        term = X
        for k in range(1, 29):
            term = apply(term) * (h / k)
            X = X + term
    return X


def _evolve(L, X, times):
    """X at each of the equally spaced times (X given at the first)."""
    out, dt = [X], float(times[1] - times[0])
    if X.shape[-1] <= 24:
        P = torch.linalg.matrix_exp(L.matrix() * dt).T.contiguous()
        for _ in times[1:]:
            out.append((out[-1].reshape(-1, P.shape[0]) @ P).reshape(X.shape))
        return out
    for _ in times[1:]:
        out.append(_taylor(L, out[-1], dt, L.bound))
    return out


def _trace(O, X):
    return torch.einsum("ij,...ji->...", O, X)


def _uniform(seed, traj, k, stream):
    """The library's uniforms: Philox4x32-10 (Salmon et al. 2011), counter
    (trajectory, jump, stream, 0), key = seed, 52 bits."""
    u32, mask = np.uint64(32), np.uint64(0xFFFFFFFF)
    c = [np.asarray(traj, np.uint64), np.asarray(k, np.uint64),
         np.full(len(traj), stream, np.uint64), np.zeros(len(traj), np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> u32) ^ c[1] ^ np.uint64(k0), b & mask, (a >> u32) ^ c[3] ^ np.uint64(k1),
             a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    m = (c[0] >> np.uint64(6)).astype(np.float64) * 67108864.0 + (c[1] >> np.uint64(6))
    return (m + 0.5) * 2.0 ** -52


def _trajectories(s, ntraj, seed):
    """Sums of the normalised expectations over the trajectories, and their
    jumps (trajectory, index, channel, time): exact propagators over 2^-k of
    an output interval, applied in binary descent to the last instant with
    <psi|psi> > r."""
    bits, tl = 50, s["tlist"]
    dt, d = float(tl[1] - tl[0]), len(s["psi0"])
    heff = s["H"] - 0.5j * sum(c.conj().T @ c for c in s["c_ops"])
    scale = torch.tensor([dt * 2.0 ** -k for k in range(bits + 1)], dtype=torch.float64, device=DEV)
    U = torch.linalg.matrix_exp(-1j * _dense(heff).T * scale[:, None, None])
    C, O = [_dense(c).T for c in s["c_ops"]], [_dense(e).T for e in s["e_ops"]]
    psi = (_dev(s["psi0"]) / np.linalg.norm(s["psi0"])).expand(ntraj, d).clone()
    nk = np.zeros(ntraj, dtype=np.int64)
    r = _dev(_uniform(seed, np.arange(ntraj), nk, 0), torch.float64)
    norm2 = lambda x: x.real.square().sum(1) + x.imag.square().sum(1)  # noqa: E731
    record = []

    def sums():
        return torch.stack([((psi.conj() * (psi @ o)).sum(1) / norm2(psi)).sum() for o in O])

    out = [sums()]
    for m in range(1, len(tl)):
        whole = psi @ U[0]
        ends = norm2(whole) > r
        idx = torch.nonzero(~ends).reshape(-1)
        psi = torch.where(ends[:, None], whole, psi)
        left = torch.full_like(idx, 1 << bits)
        while len(idx):
            x, rr = psi[idx], r[idx]
            for k in range(1, bits + 1):
                y = x @ U[k]
                take = (left >= 1 << (bits - k)) & (norm2(y) > rr)
                x = torch.where(take[:, None], y, x)
                left = left - take * (1 << (bits - k))
            psi[idx] = x
            idx, x, left = idx[left > 0], x[left > 0], left[left > 0]
            if not len(idx):
                break
            left = left - 1  # the jump, at the first instant past the crossing
            who = idx.cpu().numpy()
            y = torch.stack([x @ c for c in C], 1)
            p = y.real.square().sum(2) + y.imag.square().sum(2)
            cum = p.cumsum(1)
            target = _dev(_uniform(seed, who, nk[who], 1), torch.float64) * cum[:, -1]
            n = (cum < target[:, None]).sum(1).clamp(max=len(C) - 1)
            row = torch.arange(len(idx), device=DEV)
            psi[idx] = y[row, n] / p[row, n].sqrt()[:, None]
            tau = tl[m] - left.cpu().numpy() * (dt * 2.0 ** -bits)
            record += list(zip(who, nk[who], n.cpu().numpy(), tau))
            nk[who] += 1
            r[idx] = _dev(_uniform(seed, who, nk[who], 0), torch.float64)
            idx, left = idx[left > 0], left[left > 0]
        out.append(sums())
    return torch.stack(out), record


def _exact_sweep(case, seed):
    """The master-equation problems, padded to one size and evolved together."""
    problems, tlist = _sweep_inputs(case, seed)
    me = problems[0::2]
    d = max(p["dim"] for p in me)

    def pad(ops):
        out = np.zeros((len(ops), d, d), dtype=np.complex128)
        for q, m in enumerate(ops):
            out[q, :m.shape[0], :m.shape[0]] = m.toarray()
        return _dev(out)

    C = pad([p["c_ops"][0] for p in me])
    heff = [p["H"] - 0.5j * (p["c_ops"][0].conj().T @ p["c_ops"][0]) for p in me]
    K = -1j * pad(heff)
    O = [pad([p["e_ops"][e] for p in me]) for e in range(2)]
    Kd, Cd = K.conj().transpose(1, 2).contiguous(), C.conj().transpose(1, 2).contiguous()
    apply = lambda X: K @ X + X @ Kd + C @ (X @ Cd)  # noqa: E731
    bound = max(2.0 * abs(h).sum(axis=1).max() + (abs(p["c_ops"][0]).max()) ** 2
                for h, p in zip(heff, me))
    X = torch.zeros((len(me), d, d), dtype=torch.complex128, device=DEV)
    X[:, 0, 0] = 1.0
    out = []
    for m in range(len(tlist)):
        if m:
            X = _taylor(apply, X, float(tlist[m] - tlist[m - 1]), float(bound))
        out.append(torch.stack([torch.einsum("bij,bji->b", o, X) for o in O], 1))
    return [torch.stack(out, 1), None]


def _exact_grad(case, seed):
    """Loss and gradients of the continuous problem: forward states and the
    adjoint of each segment by Taylor steps, the time integrals of the loss
    and of the gradients by Gauss-Legendre quadrature."""
    s, omega, gamma = _grad_inputs(case, seed)
    om = _dev(omega, torch.float64)
    g = gamma[0]
    H0, Hd, P1, P2 = (_dense(s[k]) for k in ("H0", "Hd", "P1", "P2"))
    A = [_dense(a) for a in s["A"]]
    N = [a.conj().T @ a for a in A]
    K0 = -1j * H0 - 0.5 * sum(gk * n for gk, n in zip(g, N))
    bound = 2.0 * float(abs(s["H0"]).sum(axis=1).max() + np.abs(omega).max() *
                        abs(s["Hd"]).sum(axis=1).max()) + \
        2.0 * sum(float(gk) * abs(a).max() ** 2 for gk, a in zip(g, s["A"]))
    x, wq = np.polynomial.legendre.leggauss(10)
    nodes = np.concatenate([[0.0], (x + 1) / 2, [1.0]]) * s["t_seg"]
    wq = wq / 2 * s["t_seg"]

    def gen(seg, adjoint):
        K = K0 - 1j * om[:, seg, None, None] * Hd
        B = A
        if adjoint:
            K, B = K.conj().transpose(1, 2), [a.conj().T for a in A]
        K = K.contiguous()

        def f(X):
            Y = K @ X
            out = Y + Y.conj().transpose(1, 2)  # X is Hermitian throughout
            for gk, b in zip(g, B):
                out += gk * (b @ X @ b.conj().T)
            return out
        return f

    psi = _dev(s["psi0"]) / np.linalg.norm(s["psi0"])
    rho = torch.outer(psi, psi.conj()).expand(case["batch"], -1, -1).contiguous()
    loss, seg_nodes = torch.zeros(case["batch"], dtype=torch.float64, device=DEV), []
    for seg in range(case["n_seg"]):
        f, at = gen(seg, False), []
        for q in range(1, len(nodes)):
            rho = _taylor(f, rho, nodes[q] - nodes[q - 1], bound)
            if q <= 10:
                loss = loss + wq[q - 1] * _trace(P2, rho).real
                at.append(rho.cpu())
        seg_nodes.append(at)
    loss = loss + _trace(P1, rho).real
    # d lambda / dt = -L^dag(lambda) - P2 backwards; the stationary source goes
    # into an extra term of the Taylor series
    lam = P1.expand(case["batch"], -1, -1).contiguous()
    go = torch.zeros_like(om)
    gg = torch.zeros((case["batch"], len(A)), dtype=torch.float64, device=DEV)
    for seg in reversed(range(case["n_seg"])):
        f = gen(seg, True)
        for q in reversed(range(1, len(nodes))):
            h = nodes[q] - nodes[q - 1]
            n = max(1, math.ceil(bound * h / 3.0))
            for _ in range(n):
                term = (f(lam) + P2) * (h / n)
                new = lam + term
                for k in range(2, 29):
                    term = f(term) * (h / n / k)
                    new = new + term
                lam = new
            if q >= 2:
                X = seg_nodes[seg][q - 2].to(DEV)
                D = Hd @ X - X @ Hd
                go[:, seg] += wq[q - 2] * torch.einsum("bij,bij->b", lam.conj(), -1j * D).real
                for k, (a, nk) in enumerate(zip(A, N)):
                    D = a @ X @ a.conj().T - 0.5 * (nk @ X + X @ nk)
                    gg[:, k] += wq[q - 2] * torch.einsum("bij,bij->b", lam.conj(), D).real
    return [loss, go, gg]


def exact(case, seed):
    kind = case["kind"]
    if kind == "kerr_ramp_mc":
        return None  # no propagator serves two intervals of a ramp: minutes
    if kind == "sweep":
        return _exact_sweep(case, seed)  # its Monte-Carlo half would take minutes
    if kind == "grad":
        return _exact_grad(case, seed)
    s = _system(case, seed)
    if kind in ("jc_mc", "kerr_mc", "xxz_mc"):
        if kind == "xxz_mc" and case["L"] > 7:
            return None  # 51 dense propagators of the whole space per jump: over a minute
        sums, record = _trajectories(s, case["ntraj"], seed)
        if kind != "jc_mc":
            return [sums]
        rec = np.array(record, dtype=np.float64).reshape(-1, 4)
        return [sums / case["ntraj"], *_jump_table(case, *rec[:, :3].astype(np.int64).T, rec[:, 3])]
    L = _Liouvillian(s["H"], s["c_ops"])
    d = s["H"].shape[0]
    if kind == "ss":
        M = L.matrix()
        one = torch.eye(d, dtype=torch.complex128, device=DEV).reshape(-1)
        rho = torch.linalg.solve(M + torch.outer(one, one), one).reshape(d, d)
        rho = 0.5 * (rho + rho.conj().T)
        return [rho / rho.trace()]
    psi = _dev(s["psi0"]) / np.linalg.norm(s["psi0"])
    rho = torch.outer(psi, psi.conj())
    if kind == "corr":
        a = S.tensor(S.destroy(case["N"]), S.qeye(2))
        A, B = _dense(S.dag(a)), _dense(a)
        at = torch.stack(_evolve(L, rho, np.linspace(0.0, 30.0, case["n_t"])))
        X = _evolve(L, B @ at, np.linspace(0.0, 30.0, case["n_tau"]))
        return [torch.stack([torch.stack([_trace(A, x), _trace(B, x)], -1) for x in X], 1)]
    states = _evolve(L, rho, s["tlist"])
    expect = torch.stack([torch.stack([_trace(_dense(e), x) for e in s["e_ops"]]) for x in states])
    return [expect] + ([torch.stack(states)] if kind in ("jc_me", "dense_me") else [])

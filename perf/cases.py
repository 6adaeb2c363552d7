"""The calls that a user of this framework spends its time in, as timed cases.

Every case goes through the public classes of ``paper_2110_10310_gb300.system``
on seeded inputs of ``workloads``.  ``listed`` names the fixed cases, ``draw``
gives more of the same ranges, ``prepare`` builds what a program holds before
the call, ``run`` is one pass and ``exact`` is the same result from plain torch
in 64 bits.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_2110_10310_gb300 import _lib as L
from paper_2110_10310_gb300.system import LindbladBatch, LindbladSystem


def listed():
    return [
        # smallest gradient: one qubit, X gate, the whole 1000-step horizon (launch and latency)
        {"name": "qubit_x", "call": "gradient", "system": "gate", "levels": "2", "steps": 1000},
        # the two-transmon CNOT gradient over its whole horizon, the inner call of an optimisation
        {"name": "cnot_2x3", "call": "gradient", "system": "gate", "levels": "3x3", "steps": 10000},
        # the same gate with a Jaynes-Cummings coupling and the running penalty
        {"name": "cnot_jc_penalty", "call": "gradient", "system": "gate", "levels": "3x3", "steps": 4000,
         "coupling": True, "penalty": True},
        # three unequal qudits (vec 576, an odd number of states): state preparation
        {"name": "qudits_3x4x2", "call": "gradient", "system": "chain", "levels": "3x4x2", "states": 9, "steps": 500},
        # 256 independent problems of uneven size in one launch from a captured graph
        {"name": "batch256", "call": "batch", "system": "random", "problems": 256, "steps": 1000},
        # two qubits and a 20-level cavity, ground-state reset from the ensemble state (one state, ragged levels)
        {"name": "reset_2x2x20", "call": "gradient", "system": "reset", "levels": "2x2x20", "steps": 1000},
        # four 4-level qudits (vec 65536), three states, several checkpoint segments
        {"name": "qudits_4x4", "call": "gradient", "system": "chain", "levels": "4x4x4x4", "states": 3, "steps": 400},
        # largest: six qutrits (vec 531441), one checkpoint segment of forward, recompute and adjoint
        {"name": "qutrits_6x3", "call": "gradient", "system": "ring", "levels": "3x3x3x3x3x3", "states": 32,
         "steps": 100},
        # the opt-in paired-single arithmetic, forward only, final states returned
        {"name": "qutrits_6x3_f32x2", "call": "forward", "system": "ring", "levels": "3x3x3x3x3x3", "states": 8,
         "steps": 60, "precision": "f32x2"},
        # step-level call: adjoint steps on given (non-Hermitian) vectors
        {"name": "propagate_4x3", "call": "propagate", "system": "chain", "levels": "3x3x3x3", "states": 8,
         "steps": 100, "adjoint": True},
        # step-level call: y = M x, the operator alone
        {"name": "apply_6x3", "call": "apply", "system": "ring", "levels": "3x3x3x3x3x3", "states": 16, "steps": 100,
         "adjoint": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gate", "chain", "batch", "reset", "ring", "propagate", "apply"])
    if kind == "gate":
        lev = rng.choice(["2", "3", "4", "5", "2x2", "2x3", "3x2", "3x3"])
        c = {"call": "gradient", "system": "gate", "levels": lev, "steps": _log(rng, 200, 10000 if "x" in lev else 999)}
        if "x" in lev:
            c["coupling"] = rng.random() < 0.3
        c["penalty"] = rng.random() < 0.3
        return c
    if kind == "batch":
        return {"call": "batch", "system": "random", "problems": _log(rng, 4, 256), "steps": _log(rng, 100, 1000)}
    if kind == "reset":
        return {"call": "gradient", "system": "reset", "levels": "2x2x%d" % rng.randint(5, 24),
                "steps": _log(rng, 100, 1200)}
    if kind == "ring":
        q = rng.choice([4, 5, 6])
        return {"call": rng.choice(["gradient", "forward"]), "system": "ring", "levels": "x".join(["3"] * q),
                "states": _log(rng, 1, 24), "steps": _log(rng, 10, 100),
                "precision": rng.choice(["f64", "f64", "f32x2"])}
    levels = [rng.randint(2, 4) for _ in range(rng.choice([3, 4]))]
    lev = "x".join(str(n) for n in levels)
    if kind == "chain":
        return {"call": rng.choice(["gradient", "gradient", "forward"]), "system": "chain", "levels": lev,
                "states": _log(rng, 1, 12), "steps": _log(rng, 50, 400)}
    if kind == "propagate":
        return {"call": "propagate", "system": "chain", "levels": lev, "states": _log(rng, 1, 16),
                "steps": _log(rng, 20, 200), "adjoint": rng.random() < 0.5}
    q = rng.choice([3, 4, 5, 6])
    return {"call": "apply", "system": "ring", "levels": "x".join(["3"] * q), "states": _log(rng, 1, 24),
            "steps": 100, "adjoint": rng.random() < 0.5}


def _levels(case):
    return tuple(int(n) for n in case["levels"].split("x"))


def _problem(case, seed):
    """The seeded inputs of a case: a ``workloads`` problem at that workload's own step size."""
    kind, steps = case["system"], int(case["steps"])
    if kind == "gate":
        lev = _levels(case)
        if len(lev) == 1:
            p = W.config1(seed=seed)
            if lev[0] > 2:
                p.system.levels, p.system.essential = lev, (2,)
                p.system.selfkerr_ghz = np.array([0.2])
                p.rho0 = np.stack([W.basis_outer(lev, (2,), i, j) for i in range(2) for j in range(2)])
        else:
            p = W.config2(seed=seed, levels=lev)
        if case.get("coupling"):
            p.system.jc_ghz = np.array([[0.0, 0.005], [0.0, 0.0]])
            p.system.rot_ghz = np.array([4.80, 4.86])
        if case.get("penalty"):
            p.gamma1, p.penalty_a = 0.1, 20.0
    elif kind == "reset":
        p = W.reset_ensemble(levels=_levels(case), seed=seed)
    elif kind == "chain":
        p = W.config4(seed=seed, levels=_levels(case), n_states=int(case["states"]))
    else:
        p = W.config5(seed=seed, levels=_levels(case), n_states=int(case["states"]))
    if steps < p.system.n_steps:
        W.prefix(p, steps)
    return p


def _vectors(case, seed):
    """(n, N, N) complex matrices psi phi^+ of random pure states, seeded."""
    N, n = math.prod(_levels(case)), int(case["states"])
    rng = np.random.Generator(np.random.PCG64(seed + 104729))
    a = rng.standard_normal((2, n, N)) + 1j * rng.standard_normal((2, n, N))
    a /= np.linalg.norm(a, axis=2, keepdims=True)
    return torch.from_numpy(a[0]), torch.from_numpy(a[1])


def _outer(case, seed, device):
    a, b = (t.to(device) for t in _vectors(case, seed))
    return a[:, :, None] * b[:, None, :].conj()


def prepare(case, seed):
    if case["call"] == "batch":
        # the batch's systems are fixed (their sizes decide the outputs' sizes), the inputs seeded
        ps = W.config3(n_problems=int(case["problems"]))
        rng = np.random.Generator(np.random.PCG64(seed + 104729))
        for p in ps:
            N = p.system.N
            p.controls.alpha = rng.uniform(-0.01, 0.01, size=p.controls.n_params)
            p.rho0 = np.stack([W.synthetic.pure_density(W.random_pure_state(rng, N)) for _ in range(p.M)])
            p.targets = np.stack([W.synthetic.pure_density(W.random_pure_state(rng, N))] * p.M)
        systems = [LindbladSystem(W.prefix(p, int(case["steps"])), sweep=L.LB_SWEEP_RESIDENT) for p in ps]
        batch = LindbladBatch(systems)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            batch.capture(1, stream=stream)
        return {"batch": batch, "stream": stream}
    p = _problem(case, seed)
    if case["call"] in ("propagate", "apply"):
        # the operator's own states are not used by these calls beyond their number
        x = _outer(case, seed, "cuda")
        return {"system": LindbladSystem(p), "x": x, "call": case["call"], "adjoint": bool(case["adjoint"]),
                "steps": p.system.n_steps}
    prec = L.LB_PREC_F32X2 if case.get("precision") == "f32x2" else L.LB_PREC_F64
    return {"system": LindbladSystem(p, precision=prec), "alpha": np.array(p.controls.alpha), "call": case["call"]}


def run(state):
    if "batch" in state:
        G, grad = state["batch"].gradient(stream=state["stream"])
        return {"G": G, "grad": grad}
    s = state["system"]
    if state["call"] == "apply":
        return s.apply(state["x"], state["steps"] // 2, adjoint=state["adjoint"])
    if state["call"] == "propagate":
        return s.propagate(state["x"], 0, state["steps"], adjoint=state["adjoint"])
    s.set_alpha(state["alpha"])
    if state["call"] == "forward":
        G, rho = s.forward(want_states=True)
        return {"G": np.float64(G), "rho": rho}
    G, grad = s.gradient()
    return {"G": np.float64(G), "grad": grad}


def work(case):
    """Bytes: states and targets in, results out.  Flops: one operator product per step and direction
    (8 + 36 Q per element), the step update (10) and for gradients the pieces of every control (28 Q)."""
    if case["call"] == "batch":
        ps = W.config3(n_problems=int(case["problems"]), n_steps=8)
        fl = by = 0.0
        for p in ps:
            N, Q = p.system.N, p.system.Q
            el = p.M * N * (N + 1) / 2
            fl += el * int(case["steps"]) * (2 * (18 + 36 * Q) + 28 * Q)
            by += 2 * 16.0 * p.M * N * N + 8 * p.controls.n_params
        return {"bytes": by, "flops": fl}
    lev = _levels(case)
    N, Q, steps = math.prod(lev), len(lev), int(case["steps"])
    states = int(case.get("states", 1 if case["system"] == "reset" else 16 if len(lev) > 1 else 4))
    full = states * N * N
    if case["call"] == "apply":
        return {"bytes": 32.0 * full, "flops": full * (8.0 + 36 * Q)}
    if case["call"] == "propagate":
        return {"bytes": 32.0 * full, "flops": full * steps * (18.0 + 36 * Q)}
    # Hermitian states need their elements k <= l only; |i><j| of a gate needs one of each conjugate pair
    el = full * (0.5 * (N + 1) / N)
    if case["system"] == "gate":
        ne = math.isqrt(states)
        el = N * N * (ne * (ne + 1) / 2 - ne / 2)
    per = 18.0 + 36 * Q
    if case["call"] == "forward":
        return {"bytes": 3 * 16.0 * full, "flops": el * steps * per}
    return {"bytes": 2 * 16.0 * full, "flops": el * steps * (2 * per + 28 * Q)}


# ---------------------------------------------------------------------------
# the same results from plain torch in complex128: the matrix form of the
# master equation on tensors X[i, k_1..k_Q, l_1..l_Q]


def _shift(X, axis, up, n):
    """Along `axis`: up: Y[m] = sqrt(m + 1) X[m + 1]; else Y[m] = sqrt(m) X[m - 1]."""
    w = torch.sqrt(torch.arange(1, n, dtype=torch.float64, device=X.device))
    shape = [1] * X.dim()
    shape[axis] = n - 1
    Y = torch.zeros_like(X)
    Y.narrow(axis, 0 if up else 1, n - 1).copy_(X.narrow(axis, 1 if up else 0, n - 1) * w.view(shape))
    return Y


class _Model:
    def __init__(self, p, device):
        s, c = p.system, p.controls
        self.lev, self.Q, self.N, self.NT = s.levels, len(s.levels), math.prod(s.levels), s.n_steps
        self.h, self.dev = s.T_ns / s.n_steps, device
        tau = 2.0 * math.pi
        dig = np.stack(np.unravel_index(np.arange(self.N), s.levels)).astype(np.float64)
        E = np.zeros(self.N)
        gam = np.zeros((self.N, self.N))
        self.g1 = []
        for q in range(self.Q):
            n = dig[q]
            E += tau * (s.detuning_ghz[q] * n - 0.5 * s.selfkerr_ghz[q] * n * (n - 1.0))
            t1, t2 = s.t1_us[q], s.t2_us[q]
            r1 = 1.0 / (1000.0 * t1) if np.isfinite(t1) and t1 > 0 else 0.0
            r2 = 1.0 / (1000.0 * t2) if np.isfinite(t2) and t2 > 0 else 0.0
            gam += 0.5 * r2 * (n[:, None] - n[None, :]) ** 2 + 0.5 * r1 * (n[:, None] + n[None, :])
            self.g1.append(r1)
            for r in range(q):
                E -= tau * s.crosskerr_ghz[r, q] * dig[r] * n
        D = torch.from_numpy(-gam - 1j * (E[:, None] - E[None, :])).to(device)
        self.D = D.reshape((1,) + tuple(self.lev) * 2)
        # controls: d_q(t_{j+1/2}) and the factors S_s(t) e^{i Omega t} it is linear in
        t = (np.arange(self.NT) + 0.5) * self.h
        dt = (c.horizon_ns or s.T_ns) / (c.n_splines - 2)
        x = np.abs(t[:, None] / dt - (np.arange(c.n_splines)[None, :] - 0.5))
        self.S = np.where(x < 0.5, 0.75 - x * x, np.where(x < 1.5, 0.5 * (x - 1.5) ** 2, 0.0))
        self.ph = [np.exp(1j * tau * np.asarray(car)[None, :] * t[:, None]) for car in c.carriers_ghz]
        self.d, off, al = [], 0, np.asarray(c.alpha)
        for q in range(self.Q):
            nf = len(c.carriers_ghz[q])
            a = al[off:off + 2 * nf * c.n_splines].reshape(nf, c.n_splines, 2)
            off += 2 * nf * c.n_splines
            self.d.append(tau * np.einsum("js,jf,fs->j", self.S, self.ph[q], a[..., 0] + 1j * a[..., 1]))
        self.jc = []
        if s.jc_ghz is not None:
            for a in range(self.Q):
                for b in range(a + 1, self.Q):
                    if s.jc_ghz[a, b]:
                        eta = tau * (s.rot_ghz[a] - s.rot_ghz[b])
                        self.jc.append((a, b, tau * s.jc_ghz[a, b] * np.exp(1j * eta * t)))

    def comm(self, X, q):
        """[a_q, X] and [a_q^+, X]"""
        n, r, c = self.lev[q], 1 + q, 1 + self.Q + q
        return (_shift(X, r, True, n) - _shift(X, c, False, n), _shift(X, r, False, n) - _shift(X, c, True, n))

    def off(self, X, j, adj):
        sg = 1j if adj else -1j
        Y = torch.zeros_like(X)
        for q in range(self.Q):
            d = complex(self.d[q][j])
            P, R = self.comm(X, q)
            Y += sg * d * P + sg * d.conjugate() * R
            if self.g1[q]:
                n, r, c = self.lev[q], 1 + q, 1 + self.Q + q
                Y += self.g1[q] * _shift(_shift(X, r, not adj, n), c, not adj, n)
        for a, b, g in self.jc:
            na, nb, ra, rb, ca, cb = (self.lev[a], self.lev[b], 1 + a, 1 + b, 1 + self.Q + a, 1 + self.Q + b)
            gj = complex(g[j])
            U = _shift(_shift(X, rb, True, nb), ra, False, na) - _shift(_shift(X, ca, True, na), cb, False, nb)
            V = _shift(_shift(X, ra, True, na), rb, False, nb) - _shift(_shift(X, cb, True, nb), ca, False, na)
            Y += sg * gj * U + sg * gj.conjugate() * V
        return Y

    def diag(self, adj):
        return self.D.conj() if adj else self.D

    def stage(self, q, j, adj, guess):
        """z of (I - h/2 M) z = q by the Jacobi iteration, to rounding."""
        hh = 0.5 * self.h
        inv = 1.0 / (1.0 - hh * self.diag(adj))
        z = inv * q if guess is None else guess
        top, done = float(q.abs().max()), False
        for _ in range(60):
            zn = inv * (q + hh * self.off(z, j, adj))
            ch = float((zn - z).abs().max())
            z = zn
            if done or ch == 0.0:
                break
            done = ch <= 4e-16 * top
        return z


def _sweep(m, q, adj, keep=True):
    """Stage vectors and final state of a sweep over all steps from q; the adjoint runs them in reverse."""
    zs, prev = [], None
    for j in (range(m.NT - 1, -1, -1) if adj else range(m.NT)):
        z = m.stage(q, j, adj, prev)
        q, prev = 2 * z - q, z
        if keep:
            zs.append(z)
    return zs, q


def _dense_steps(m):
    """The step propagators (I - h/2 M_j)^-1 (I + h/2 M_j) of a small system, from M applied to every unit matrix."""
    V = m.N * m.N
    eye = torch.eye(V, dtype=torch.complex128).reshape((V,) + tuple(m.lev) * 2)
    col = lambda X: X.reshape(V, V).T.contiguous()  # noqa: E731
    A, B = [], []
    for q in range(m.Q):
        P, R = m.comm(eye, q)
        A.append(col(-1j * (P + R)))
        B.append(col(P - R))
    d, jc = m.d, m.jc
    m.d, m.jc = [np.zeros(1)] * m.Q, []
    base = col(m.off(eye, 0, False) + m.D * eye)
    terms, coef = A + B, [x.real for x in d] + [x.imag for x in d]
    for a, b, g in jc:
        for f in (1.0, 1j):
            m.jc = [(a, b, np.array([f]))]
            terms.append(col(m.off(eye, 0, False) + m.D * eye) - base)
        coef += [g.real, g.imag]
    m.d, m.jc = d, jc
    T, C = torch.stack(terms).reshape(len(terms), -1), torch.from_numpy(np.stack(coef, 1)).to(torch.complex128)
    I = torch.eye(V, dtype=torch.complex128)
    P = torch.empty(m.NT, V, V, dtype=torch.complex128)
    for j in range(0, m.NT, 500):
        Mj = base + (C[j:j + 500] @ T).reshape(-1, V, V)
        P[j:j + 500] = torch.linalg.solve(I - 0.5 * m.h * Mj, I + 0.5 * m.h * Mj)
    return P, A, B


def _targets(p):
    if p.objective == "nm":
        d = np.abs(np.arange(p.system.N) - p.meta["m"]).astype(np.complex128)
        return np.broadcast_to(np.diag(d), p.rho0.shape)
    if p.targets is not None:
        return p.targets
    idx = [W.synthetic.essential_to_full(i, p.system.levels, p.system.essential) for i in range(len(p.gate))]
    V = np.zeros((p.system.N, p.system.N), dtype=np.complex128)
    V[np.ix_(idx, idx)] = p.gate
    return V @ p.rho0 @ V.conj().T


def _exact_gradient(p, device, forward_only):
    N = p.system.N
    dense = N * N <= 100
    m = _Model(p, "cpu" if dense else device)
    lead = tuple(m.lev) * 2
    q0 = torch.from_numpy(p.rho0).to(m.dev).reshape((-1,) + lead)
    tar = torch.from_numpy(np.array(_targets(p))).to(m.dev).reshape((-1,) + lead)
    w = np.ones(p.M) if p.weights is None else np.asarray(p.weights)
    w = torch.from_numpy(w / p.M).to(m.dev).reshape((-1,) + (1,) * (2 * m.Q))
    pen = np.zeros(m.NT)
    if p.gamma1:
        pen = p.gamma1 * m.h * np.exp(-((np.arange(m.NT) * m.h - p.system.T_ns) / p.penalty_a) ** 2) / p.penalty_a

    def merit(q):
        if p.objective == "nm":
            return float((w * (tar.conj() * q).real).sum())
        return float((w * 0.5 * (q - tar).abs() ** 2).sum())

    if not dense:
        zs, q = _sweep(m, q0, False, not forward_only)
        G = merit(q)
        if forward_only:
            return {"G": np.float64(G), "rho": q.reshape(-1, N, N)}
        zh, _ = _sweep(m, w * tar if p.objective == "nm" else w * (q - tar), True)
        zh = zh[::-1]
        ga = np.zeros((2, m.Q, m.NT))
        for j in range(m.NT):
            for k in range(m.Q):
                P, R = m.comm(zs[j], k)
                ga[0, k, j] = float((zh[j].conj() * (-1j * (P + R))).real.sum())
                ga[1, k, j] = float((zh[j].conj() * (P - R)).real.sum())
    else:
        P, A, B = _dense_steps(m)
        V = N * N
        qs = torch.empty(m.NT + 1, V, p.M, dtype=torch.complex128)
        qs[0] = q0.reshape(p.M, V).T
        for j in range(m.NT):
            qs[j + 1] = P[j] @ qs[j]
        back = lambda x: x.T.reshape((-1,) + lead)  # noqa: E731
        G = merit(back(qs[m.NT])) + sum(pen[j] * merit(back(qs[j])) for j in range(m.NT) if pen[j])
        wv, tv = w.reshape(1, -1), tar.reshape(p.M, V).T
        lam = wv * (qs[m.NT] - tv)
        zh = torch.empty(m.NT, V, p.M, dtype=torch.complex128)
        for j in range(m.NT - 1, -1, -1):
            nxt = P[j].conj().T @ lam
            zh[j] = 0.5 * (nxt + lam)
            lam = nxt + (pen[j] * wv * (qs[j] - tv) if pen[j] else 0.0)
        z = 0.5 * (qs[:-1] + qs[1:])
        ga = np.array([[(zh.conj() * (T @ z)).real.sum((1, 2)).numpy() for T in ops] for ops in (A, B)])
    grad = []
    for k in range(m.Q):
        ph = m.ph[k]
        re = np.einsum("js,jf,j->fs", m.S, ph.real, ga[0, k]) + np.einsum("js,jf,j->fs", m.S, ph.imag, ga[1, k])
        im = np.einsum("js,jf,j->fs", m.S, ph.real, ga[1, k]) - np.einsum("js,jf,j->fs", m.S, ph.imag, ga[0, k])
        grad.append((2.0 * math.pi * m.h * np.stack([re, im], -1)).reshape(-1))
    return {"G": np.float64(G), "grad": np.concatenate(grad)}


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] == "batch":
        return None  # hundreds of problems: minutes in plain torch
    N, steps = math.prod(_levels(case)), int(case["steps"])
    if case["call"] == "gradient" and int(case.get("states", 1)) * N * N * steps > 2e8:
        return None  # over 20 s
    p = _problem(case, seed)
    if case["call"] in ("propagate", "apply"):
        m = _Model(p, device)
        x = _outer(case, seed, device).reshape((-1,) + tuple(m.lev) * 2)
        adj = bool(case["adjoint"])
        if case["call"] == "apply":
            y = m.off(x, m.NT // 2, adj) + m.diag(adj) * x
        else:
            _, y = _sweep(m, x, adj, False)
        return y.reshape(-1, N, N)
    return _exact_gradient(p, device, case["call"] == "forward")

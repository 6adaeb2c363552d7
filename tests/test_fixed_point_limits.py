"""The fixed-point sweeps at the limits of their arithmetic: states that grow,
cancel, vanish or decay between two rescalings, peaked states, tables that do
not fit, and the calls that share their buffers.

Tolerances: the method's accuracy targets against the oracle (states and
objective 1e-10, gradient 1e-9 of the largest entry) unless a test derives its
own."""

import importlib
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from oracle import imr, model

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

torch = pytest.importorskip("torch")
gpu = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10310_gb300 import _lib

    _lib.load(build_if_missing=True)
    return _lib


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / np.max(np.abs(b)))


def _sys(p, **kw):
    from paper_2110_10310_gb300.system import LindbladSystem

    return LindbladSystem(p, **kw)


def _fixed(s):
    assert s.stats()["arithmetic"] == "fixed"
    return s


def _basis(levels, k, l):
    N = int(np.prod(levels))
    r = np.zeros((N, N), dtype=np.complex128)
    r[k, l] = 1.0
    return r


def _constant_drive(levels, n_steps, h, theta, t1_us=100.0, t2_us=50.0):
    """Resonant subsystems under constant drives of theta rad per step."""
    p = W.random_problem(811, levels=levels, n_states=1, n_steps=n_steps, T_ns=h * n_steps, amp=0.01, ckpt_every=0)
    Q = len(levels)
    p.system.detuning_ghz[:] = 0.0
    p.system.selfkerr_ghz[:] = 0.0
    p.system.crosskerr_ghz[:] = 0.0
    p.system.t1_us, p.system.t2_us = np.full(Q, t1_us), np.full(Q, t2_us)
    p.controls.carriers_ghz = [np.zeros(1) for _ in range(Q)]
    a = np.zeros((Q, 1, p.controls.n_splines, 2))
    a[..., 0] = theta / (2.0 * np.pi * h)
    p.controls.alpha = a.reshape(-1)
    p.weights = None
    p.rho0 = np.stack([_basis(levels, 0, 0)])
    return p


@gpu
def test_an_adjoint_state_that_gathers_within_a_chunk(L):
    """The target is what |00> has spread into over the last chunk's 22 steps,
    so that the adjoint state gathers into one entry 8.4 times its largest
    there: 2^63.06 in the scale of the chunk's end."""
    p = _constant_drive((3, 3), 748, 0.1, 0.0476)
    m = model.Model(p.system, p.controls)
    q = model.vec(p.rho0).T.copy()
    for j in range(726, 748):
        q, _ = imr.imr_step(m, j, q)
    p.targets = model.unvec(q[:, 0], 9)[None]
    p.objective, p.weights = "trace", np.array([1.04])
    s = _sys(p)
    G, g = s.gradient()
    assert _fixed(s).stats()["sweep"] == "cluster"
    Go, go, _ = imr.gradient(p)
    assert abs(G - Go) <= 1e-10 * abs(Go)
    assert _rel(g, go) < 1e-9


@gpu
@pytest.mark.parametrize("n_steps,theta,weight,sweep", [(23, 0.7796, 1.0, "resident"), (64, np.pi / 4.5, 1.06, "cluster")])
def test_a_penalty_source_that_cancels_the_adjoint_state(L, n_steps, theta, weight, sweep):
    """A free coherence whose adjoint turns by theta per step while a constant
    running penalty adds the same source each step: the sum falls to some
    hundredths of both addends -- after seven sources in the sequential sweep,
    and where the response of a chunk's eight sources meets the adjoint state."""
    h = 0.1
    p = _constant_drive((2,), n_steps, h, 1e-4, t1_us=np.inf, t2_us=np.inf)
    # the implicit midpoint step turns a phase by 2 atan(h delta / 2)
    p.system.detuning_ghz[:] = 2.0 * np.tan(0.5 * theta) / h / (2.0 * np.pi)
    p.rho0 = np.full((1, 2, 2), 0.5, dtype=np.complex128)
    p.targets = np.array([[[0.0, 0.5], [0.5, 0.0]]], dtype=np.complex128)
    p.objective, p.penalty_a = "trace", 1e6
    p.gamma1 = weight * p.penalty_a / h
    s = _sys(p)
    G, g = s.gradient()
    assert _fixed(s).stats()["sweep"] == "cluster" and (s.stats()["kernel_launches"] > 8) == (sweep == "cluster")
    Go, go, _ = imr.gradient(p)
    assert abs(G - Go) <= 1e-10 * abs(Go)
    assert _rel(g, go) < 1e-9


def _vanishing(levels, n_steps, zero):
    """Two states, one of which has a zero weight or is zero itself."""
    p = W.random_problem(813, levels=levels, n_states=2, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.02, ckpt_every=0)
    p.weights = np.array([1.0, 1.0])
    if zero == "weight":
        p.weights[1] = 0.0
    else:
        p.rho0[1] = 0.0
    return p


@gpu
@pytest.mark.parametrize("levels,n_steps,sweep", [((2, 2), 24, 1), ((2, 2), 24, 0), ((2, 2), 80, 0), ((3, 2, 3), 10, 1), ((3, 3), 20, 2)])
@pytest.mark.parametrize("zero", ["weight", "state"])
def test_states_of_zeros(L, levels, n_steps, sweep, zero):
    """The one-CTA sweeps (register and table path), the chunks and the grid."""
    p = _vanishing(levels, n_steps, zero)
    s = _sys(p, sweep=sweep)
    G, g = s.gradient()
    _fixed(s)
    Go, go, _ = imr.gradient(p)
    assert abs(G - Go) <= 1e-10 * abs(Go)
    assert _rel(g, go) < 1e-9
    x = torch.from_numpy(p.rho0).cuda()
    x[0] = 0.0
    for adj in (False, True):
        assert not s.propagate(x[:1], 0, n_steps, adjoint=adj).any()


@gpu
@pytest.mark.parametrize("levels,n_steps,sweep", [((2, 2), 24, 1), ((2, 2), 80, 0), ((3, 2, 3), 10, 1), ((3, 3), 20, 2)])
def test_a_tolerance_below_the_resolution(L, levels, n_steps, sweep):
    p = W.random_problem(814, levels=levels, n_states=2, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.02, ckpt_every=0)
    s = _sys(p, sweep=sweep, rtol=1e-30)
    G, g = s.gradient()
    _fixed(s)
    Go, go, _ = imr.gradient(p)
    assert abs(G - Go) <= 1e-10 * abs(Go)
    assert _rel(g, go) < 1e-9


HARNESS = r"""
#include <cstdio>
#include "lb_fixed.cuh"
int main() {
  long long a, x, b, y;
  while (std::scanf("%lld %lld %lld %lld", &a, &x, &b, &y) == 4) {
    lbk::FxSum s{0, 0u};
    lbk::fx_sum_mac(s, lbk::fx_split(a), lbk::fx_split(x));
    lbk::fx_sum_mac(s, lbk::fx_split(b), lbk::fx_split(y));
    std::printf("%lld %u\n", s.hi, s.lo);
  }
  return 0;
}
"""


def test_sums_of_products_keep_32_bits_below_the_cut(tmp_path):
    """Each product is whole but for its last 32 bits (rounded down)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    B = importlib.import_module("paper_2110_10310_gb300.build")
    src, exe = tmp_path / "h.cu", str(tmp_path / "h")
    src.write_text(HARNESS)
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-I", B.CSRC, "-o", exe, str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    rng = random.Random(6)
    top = 1 << 61
    cases = [(top, -top, top, top - 1), (-1, 1, 0, 5), (-top, -top, -top, -top), (2**31, 2**31, -2**31, 2**31 - 1)]
    for _ in range(2000):
        cases.append(tuple(rng.randrange(-top, top) >> rng.randrange(0, 60) for _ in range(4)))
    inp = "\n".join(" ".join(str(v) for v in c) for c in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, timeout=60).stdout.split("\n")
    for (a, x, b, y), line in zip(cases, out):
        hi, lo = (int(v) for v in line.split())
        assert 0 <= a * x + b * y - ((hi << 32) + lo) * 2**32 < 2 * 2**32


SHIFTS = r"""
#include <cstdio>
#include "lb_fixed.cuh"
int main() {
  long long x;
  int s;
  unsigned h;
  while (std::scanf("%lld %d %u", &x, &s, &h) == 3)
    std::printf("%lld %d %d\n", lbk::fx_shift(x, s), lbk::fx_rescale_shift(h), lbk::fx_quarter_shift(h));
  return 0;
}
"""


def test_shifts_of_states_of_any_size(tmp_path):
    """fx_shift rounds to nearest at every size, and the shifts that keep a
    state's scale bring its largest high word to [2^27, 2^28) or leave it there."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    B = importlib.import_module("paper_2110_10310_gb300.build")
    src, exe = tmp_path / "h.cu", str(tmp_path / "h")
    src.write_text(SHIFTS)
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-I", B.CSRC, "-o", exe, str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    rng = random.Random(7)
    cases = [(0, 0, 0), (1, 0, 1), ((1 << 61) - 1, 61, (1 << 31) - 1), (-(1 << 61), 61, 1 << 28)]
    for _ in range(3000):
        s = rng.randrange(-20, 62)
        x = rng.randrange(-(1 << 61), 1 << 61) >> (max(0, -s) + rng.randrange(0, 3))
        cases.append((x, s, rng.randrange(0, 1 << 31) >> rng.randrange(0, 31)))
    inp = "\n".join(" ".join(str(v) for v in c) for c in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, timeout=60).stdout.split("\n")
    for (x, s, h), line in zip(cases, out):
        y, rs, qs = (int(v) for v in line.split())
        assert y == ((x + ((1 << s) >> 1)) >> s if s >= 0 else x << -s)
        kept = h == 0 or 94906266 <= h < 1 << 28
        assert rs == (0 if kept else h.bit_length() - 28)
        quarter = h == 0 or 94906266 // 4 <= h < 1 << 26
        assert qs == (-2 if quarter else h.bit_length() - 28)


def _long_gradient(p):
    """G's pieces and the gradient of one state in extended precision (numpy's
    longdouble): the matrix form, each stage by the Jacobi iteration."""
    ld, cld = np.longdouble, np.clongdouble
    m = model.Model(p.system, p.controls)
    lev, Q, N = p.system.levels, len(p.system.levels), m.N
    NT, h = p.system.n_steps, ld(p.system.T_ns / p.system.n_steps)
    dig = np.stack(np.unravel_index(np.arange(N), lev))
    num = [d.astype(ld) for d in dig]
    st = [int(np.prod(lev[q + 1:])) for q in range(Q)]
    # row k of a X is sqrt(n_q + 1) times row k + st of X; of a^+ X sqrt(n_q) times row k - st
    up = [np.where(dig[q] + 1 < lev[q], np.sqrt(num[q] + 1), ld(0)) for q in range(Q)]
    dn = [np.sqrt(num[q]) for q in range(Q)]

    def left(X, q, dag):
        return dn[q][:, None] * np.roll(X, st[q], 0) if dag else up[q][:, None] * np.roll(X, -st[q], 0)

    def right(X, q, dag):
        return np.roll(X, -st[q], 1) * up[q] if dag else np.roll(X, st[q], 1) * dn[q]

    def comm(X, q):
        return left(X, q, False) - right(X, q, False), left(X, q, True) - right(X, q, True)

    one = np.ones((N, N), dtype=ld)
    E = sum(ld(2 * np.pi * p.system.detuning_ghz[q]) * num[q]
            - ld(np.pi * p.system.selfkerr_ghz[q]) * num[q] * (num[q] - 1) for q in range(Q))
    for q in range(Q):
        for r in range(q):
            E = E - ld(2 * np.pi * p.system.crosskerr_ghz[r, q]) * num[r] * num[q]
    g1 = [ld(1.0 / (1000.0 * t)) for t in p.system.t1_us]
    g2 = [ld(1.0 / (1000.0 * t)) for t in p.system.t2_us]
    D = (-1j * (E[:, None] - E[None, :])).astype(cld)
    for q in range(Q):
        d = num[q][:, None] - num[q][None, :]
        D = D - (g2[q] * d * d + g1[q] * (num[q][:, None] + num[q][None, :])) / 2 * one
    t = [m.t_half(j) for j in range(NT)]
    amp = np.array([model.control_amplitudes(p.controls, x, p.system.T_ns) for x in t])

    def off(X, j, adj):
        Y = np.zeros_like(X)
        for q in range(Q):
            P, R = comm(X, q)
            Y = Y + (1j if adj else -1j) * (cld(amp[j][q]) * P + cld(np.conj(amp[j][q])) * R)
            Y = Y + g1[q] * right(left(X, q, adj), q, not adj)
        return Y

    def stage(x, j, adj):
        d = D.conj() if adj else D
        inv = 1 / (1 - h / 2 * d)
        z = inv * x
        for _ in range(60):
            z, old = inv * (x + h / 2 * off(z, j, adj)), z
            if np.abs(z - old).max() <= ld(1e-22) * np.abs(x).max():
                break
        return z

    rho, zs = p.rho0[0].astype(cld), []
    for j in range(NT):
        zs.append(stage(rho, j, False))
        rho = 2 * zs[-1] - rho
    lam = rho - p.targets[0].astype(cld)
    lmax = float(np.abs(lam).max())
    grad = np.zeros(p.controls.n_params, dtype=ld)
    for j in range(NT - 1, -1, -1):
        zh = stage(lam, j, True)
        lam = 2 * zh - lam
        for q in range(Q):
            P, R = comm(zs[j], q)
            pr = np.real((zh.conj() * (-1j * (P + R))).sum()), np.real((zh.conj() * (P - R)).sum())
            for f, om in enumerate(p.controls.carriers_ghz[q]):
                ph = ld(2 * np.pi * om * t[j])
                for s in range(p.controls.n_splines):
                    S = ld(model.bspline_basis(s, t[j], p.controls.n_splines, p.system.T_ns)) * 2 * ld(np.pi) * h
                    k = model.alpha_index(p.controls, q, f, s)
                    grad[k] += S * (np.cos(ph) * pr[0] + np.sin(ph) * pr[1])
                    grad[k + 1] += S * (np.cos(ph) * pr[1] - np.sin(ph) * pr[0])
    return grad, lmax


@gpu
@pytest.mark.parametrize("levels,sweep,symmetry", [
    ((4, 4), 1, 0), ((4, 4), 1, 1), ((4, 4, 4), 1, 0), ((4, 4, 4), 1, 1), ((3, 3, 3), 2, 0), ((4, 4, 4), 2, 0),
    ((4, 4, 4), 2, 1)])
def test_gradient_of_a_peaked_state(L, levels, sweep, symmetry):
    """One large entry among thousands below 1e-3 in the state and in the
    target: the gradient comes from products with the small ones.  One step,
    solved to the format's resolution (rtol 1e-19): an entry of either stage
    vector, or of its neighbour combinations, is off by at most 8 units of 2^-59
    of its state's largest; each error meets the other state's entries, whose
    magnitudes sum to below 2 of its largest one, with ladder factors of at
    most 4 sqrt(3) in all."""
    N = int(np.prod(levels))
    p = W.random_problem(815, levels=levels, n_states=1, n_steps=1, T_ns=0.01, amp=0.004, ckpt_every=0)
    rng = np.random.default_rng(816)

    def peaked(k):
        v = 1e-3 * W.random_pure_state(rng, N)
        v[k] = 1.0
        return W.synthetic.pure_density(v)[None]

    p.rho0, p.targets, p.weights = peaked(0), peaked(N - 1), None
    s = _sys(p, sweep=sweep, symmetry=symmetry, rtol=1e-19)
    _, g = s.gradient()
    _fixed(s)
    go, lmax = _long_gradient(p)
    unit = 2.0**-59 * lmax * 2.0 * np.pi * p.system.T_ns
    err, tol = float(np.abs(g - go).max()), unit * 2 * 8 * 2 * 4 * np.sqrt(3.0) + 4e-16 * float(np.abs(go).max())
    print(levels, sweep, symmetry, "error", err, "bound", tol)
    assert err < tol


@gpu
@pytest.mark.parametrize("hermitian,K", [(True, 0), (False, 4)])
def test_a_zero_adjoint_state_beside_a_small_one(L, hermitian, K):
    """The grid sweep brings every state's gradient sums to one scale: a state
    of weight zero must not set it.  With the other's weight 2^-40 the integers
    are the same as with weight 1, so the gradient is 2^-40 of that one, bitwise."""
    p = W.random_problem(819, levels=(3, 3), n_states=2, n_steps=12, T_ns=0.12, amp=0.02, hermitian=hermitian, ckpt_every=K)
    res = []
    for w in (1.0, 2.0**-40):
        p.weights = np.array([w, 0.0])
        s = _sys(p, sweep=L.LB_SWEEP_GRID)
        res.append(s.gradient())
        _fixed(s)
    assert res[1][0] == res[0][0] * 2.0**-40 and np.array_equal(res[1][1], res[0][1] * 2.0**-40)
    Go, go, _ = imr.gradient(p)
    assert _rel(res[1][1], go) < 1e-9


def _mode(n_steps, levels=(64,), n_states=2, hermitian=False):
    """One mode of many levels, its phases and decay small."""
    p = W.random_problem(818, levels=levels, n_states=n_states, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.004,
                         hermitian=hermitian, ckpt_every=0)
    Q = len(levels)
    p.system.detuning_ghz[:] = 0.01
    p.system.selfkerr_ghz[:] = 1e-4
    p.system.crosskerr_ghz[:] = 0.0
    p.system.t1_us, p.system.t2_us = np.full(Q, 40.0), np.full(Q, 30.0)
    return p


@gpu
@pytest.mark.parametrize("n,hermitian,fits", [(58, False, True), (58, True, True), (62, True, True), (64, True, False),
                                              (59, False, False)])
def test_one_mode_of_many_levels_in_one_cta(L, n, hermitian, fits):
    """One mode's decay tables beside its state: the largest that fit one CTA,
    against the Neumann iteration (FP64) or, where that does not fit, the grid;
    the first that do not are refused by the launch, as by the FP64 sweep's."""
    p = _mode(4, (n,), hermitian=hermitian)
    s = _sys(p, sweep=L.LB_SWEEP_RESIDENT)
    if not fits:
        with pytest.raises(L.LBError) as e:
            s.gradient()
        assert e.value.code == L.LB_ECUDA
        return
    G, g = s.gradient()
    _fixed(s)
    other = dict(sweep=L.LB_SWEEP_RESIDENT, solver=L.LB_SOLVER_NEUMANN) if n <= 58 else dict(sweep=L.LB_SWEEP_GRID)
    Gn, gn = _sys(p, **other).gradient()
    assert abs(G - Gn) <= 1e-12 * abs(Gn) and _rel(g, gn) < 1e-11
    x = torch.from_numpy(p.rho0).cuda()
    if not hermitian:  # steps on vectors take every element
        assert _rel(s.propagate(x, 0, 4).cpu().numpy(),
                    _sys(p, sweep=L.LB_SWEEP_GRID).propagate(x, 0, 4).cpu().numpy()) < 1e-13


def _torch_model(p):
    """The operator of a problem in plain torch: perf.cases' 64-bit matrix form."""
    from perf.cases import _Model

    return _Model(p, "cuda")


def _apply_ref(p, x, step, adj):
    """M x and the sum of the magnitudes of its terms, entry by entry."""
    m = _torch_model(p)
    X = x.reshape((-1,) + tuple(m.lev) * 2)
    y = m.off(X, step, adj) + m.diag(adj) * X
    return y.reshape(x.shape)


def _term_bound(p, x, step):
    """A bound of the sum of the magnitudes of the terms of an entry of M x, per
    vector: twice the row sums' bound times the vector's largest entry."""
    m = _torch_model(p)
    row = float(m.D.abs().max())
    for q, n in enumerate(m.lev):
        row += abs(complex(m.d[q][step])) * 2.0 * (np.sqrt(n - 1.0) + np.sqrt(n - 2.0)) + m.g1[q] * (n - 1.0)
    return 2.0 * row * x.abs().amax(dim=(1, 2))


def _vectors(n, N, seed=5):
    g = torch.Generator().manual_seed(seed)
    a = torch.randn((n, N, N), dtype=torch.complex128, generator=g)
    return a.cuda()


@gpu
@pytest.mark.parametrize("levels,n_steps,sweep", [((2,), 300, 1), ((2,), 300, 0), ((2, 5), 120, 1), ((2, 5), 120, 0),
                                                  ((3, 2, 3), 80, 1), ((3,), 300, 2), ((3, 2, 2), 100, 2)])
def test_a_coherence_that_halves_and_more_each_step(L, levels, n_steps, sweep):
    """A dephasing first subsystem, the slowest decay of its coherences 0.4 of
    themselves per step: hundreds of powers of ten over the run, far below
    2^-60 within the length of a chunk.  Every solve keeps the state's own scale."""
    p = W.random_problem(820, levels=levels, n_states=1, n_steps=n_steps, T_ns=float(n_steps), amp=0.0,
                         hermitian=False, ckpt_every=0)
    Q = len(levels)
    p.system.detuning_ghz[:] = 1e-4
    p.system.selfkerr_ghz[:] = 1e-4
    p.system.crosskerr_ghz[:] = 0.0
    n = levels[0] - 1
    p.system.t1_us = np.full(Q, np.inf)
    p.system.t2_us = np.r_[1e-3 * 0.5 * n * n / 0.85, np.full(Q - 1, np.inf)]  # decay h n^2 / (2 T2) = 0.85
    p.controls.alpha[:] = 0.0
    N = int(np.prod(levels))
    p.rho0 = np.zeros((1, N, N), dtype=np.complex128)
    p.rho0[0, 0, N - 1] = 0.3  # levels 0 and n of the first subsystem
    p.weights = None
    s = _sys(p, sweep=sweep)
    _, rho = s.forward(want_states=True)
    _fixed(s)
    h = 1.0
    m = _torch_model(p)
    d = complex(m.D.reshape(N, N)[0, N - 1])
    want = 0.3 * ((1 + 0.5 * h * d) / (1 - 0.5 * h * d)) ** n_steps
    assert 0.0 < abs(want) < 1e-25
    assert abs(complex(rho[0, 0, N - 1]) - want) <= 1e-12 * abs(want)
    x = torch.from_numpy(p.rho0).cuda()
    y = s.propagate(x, 0, n_steps, adjoint=True)
    assert abs(complex(y[0, 0, N - 1]) - np.conj(want / 0.3) * 0.3) <= 1e-12 * abs(want)


@gpu
def test_products_where_control_and_decay_factors_are_alike(L):
    """Drives as weak as the decay: scaled up together, the two control factors
    and the decay factor of one sum must not pass 64 bits.  The bound is that of
    test_large_products_match_fp64."""
    p = _mode(3, (4, 4, 4, 4), n_states=6)
    Q = 4
    p.controls.carriers_ghz = [np.zeros(1) for _ in range(Q)]
    # (dt/2) 2 pi |d| 2^3 (the ladder's scale) = (dt/2) 3 / T1
    p.controls.alpha = np.full(2 * p.controls.n_splines * Q, 3.0 / 40e3 / (2.0 * np.pi * 8.0))
    s = _sys(p, sweep=L.LB_SWEEP_GRID)
    x = _vectors(6, 256)
    for adj in (False, True):
        y, ref = s.apply(x, 1, adjoint=adj), _apply_ref(p, x, 1, adj)
        assert bool(((y - ref).abs().amax(dim=(1, 2)) <= 2.0**-50 * _term_bound(p, x, 1)).all())


# edges of the product's dispatch: the fewest vectors it takes and one less, the unrolled
# loops (4 and 6 subsystems) and the general one, odd N, tables above 48 KB of
# shared memory, fewer vectors than states
@gpu
@pytest.mark.parametrize("levels,M,n", [
    ((4, 4, 4, 4), 4, 4), ((4, 4, 4, 4), 4, 3), ((3, 3, 3, 3, 3), 4, 4), ((3,) * 6, 1, 1), ((5, 5, 5), 21, 21),
    ((5, 5, 5), 21, 20), ((7, 3, 7), 20, 15), ((2, 2, 56), 15, 15), ((2, 64), 84, 84)])
@pytest.mark.parametrize("decay", [True, False])
def test_large_products_match_fp64(L, levels, M, n, decay):
    """FP64's and the integers' rounding of at most 2^-50 of the terms."""
    p = _mode(3, levels, n_states=M)
    if not decay:
        p.system.t1_us[:] = np.inf
    s = _sys(p, sweep=L.LB_SWEEP_GRID)
    N = int(np.prod(levels))
    x = _vectors(n, N)
    x[0] *= 1e-200
    if n > 2:
        x[1] *= 1e150
        x[2] = 0.0
    for adj in (False, True):
        y, ref = s.apply(x, 1, adjoint=adj), _apply_ref(p, x, 1, adj)
        err = (y - ref).abs().amax(dim=(1, 2))
        assert bool((err <= 2.0**-50 * _term_bound(p, x, 1)).all())
    if n > 2:
        x[2, 1, 1] = complex(float("nan"), 0.0)
        y = s.apply(x, 1)
        assert bool(torch.isnan(y[2]).any()) and bool(torch.isfinite(y[[0, 1]].abs()).all())


@gpu
def test_products_beside_a_gradient_and_each_other_on_other_streams(L):
    """Products on two streams while a gradient runs on a third: all as alone."""
    p = W.prefix(W.config4(n_states=6), 60)
    s = _sys(p)
    x, x2 = _vectors(6, 256, 6), _vectors(6, 256, 7)
    G, g = s.gradient()
    _fixed(s)
    y, y2 = s.apply(x, 7), s.apply(x2, 9)
    streams = [torch.cuda.Stream() for _ in range(3)]
    Gd = torch.zeros(1, dtype=torch.float64, device="cuda")
    gd = torch.zeros(s.n_params, dtype=torch.float64, device="cuda")
    bufs = [t.transpose(1, 2).contiguous() for t in (x, x2)]
    outs = [[torch.zeros_like(b) for _ in range(6)] for b in bufs]
    torch.cuda.synchronize()
    s.gradient_async(Gd, gd, stream=streams[0])
    for k in range(6):
        for i in range(2):
            L.check(s.lib.lb_apply(s.h, streams[1 + i].cuda_stream, 0, (7, 9)[i], bufs[i].data_ptr(),
                                   outs[i][k].data_ptr(), 6))
    torch.cuda.synchronize()
    assert float(Gd) == G and np.array_equal(gd.cpu().numpy(), g)
    for i, want in enumerate((y, y2)):
        for o in outs[i]:
            assert torch.equal(o.transpose(1, 2), want)


@gpu
def test_a_recorded_product_is_replayed(L):
    """Recorded, the product is FP64 (its own buffer would be shared by replays)."""
    p = W.prefix(W.config4(n_states=6), 20)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = _sys(p)
        x = _vectors(6, 256, 6).transpose(1, 2).contiguous()
        y, z = torch.zeros_like(x), torch.zeros_like(x)
        L.check(s.lib.lb_apply(s.h, st.cuda_stream, 0, 7, x.data_ptr(), y.data_ptr(), 6))
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            L.check(s.lib.lb_apply(s.h, st.cuda_stream, 0, 7, x.data_ptr(), z.data_ptr(), 6))
        graph.replay()
        torch.cuda.synchronize()
    assert _rel(z.cpu().numpy(), y.cpu().numpy()) < 1e-14


@gpu
@pytest.mark.parametrize("levels,sweep", [((3, 3), 0), ((3, 3), 1), ((3, 2, 3), 1), ((3, 3), 2), ((4, 4, 4), 2)])
def test_fp64_sweeps_on_request(L, levels, sweep):
    """The FP64 Jacobi sweeps at full length beside the fixed-point ones."""
    p = W.random_problem(822, levels=levels, n_states=2, n_steps=150, T_ns=1.5, amp=0.02, ckpt_every=0)
    s, f = _sys(p, sweep=sweep), _sys(p, sweep=sweep, arithmetic=L.LB_ARITH_F64)
    G, g = _fixed_after(s)
    Gf, gf = f.gradient()
    assert f.stats()["arithmetic"] == "f64" and f.workspace_bytes <= s.workspace_bytes
    assert abs(G - Gf) <= 1e-12 * abs(Gf) and _rel(g, gf) < 1e-11
    with pytest.raises(L.LBError):
        L.check(f.lib.lb_set_arithmetic(f.h, L.LB_ARITH_FIXED))  # a workspace is bound


def _fixed_after(s):
    r = s.gradient()
    _fixed(s)
    return r


def test_arithmetic_values():
    from paper_2110_10310_gb300 import _lib as L

    if not os.path.exists(L.lib_path()):
        pytest.skip("library not built")
    lib = L.load()
    assert lib.lb_set_arithmetic(None, L.LB_ARITH_F64) == L.LB_EINVAL


@gpu
@pytest.mark.parametrize("n_steps,sweep", [(24, 1), (80, 0)])
def test_a_penalty_source_that_overflows_is_reported(L, n_steps, sweep):
    p = W.random_problem(821, levels=(2, 2), n_states=1, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.02, ckpt_every=0)
    p.gamma1, p.penalty_a, p.weights = 1.7e308, 0.1, np.array([1e5])
    s = _sys(p, sweep=sweep)
    with pytest.raises(L.LBError) as e:
        s.gradient()
    assert e.value.code == L.LB_ENAN and str(e.value).endswith(f"time step {n_steps - 2}")


@gpu
@pytest.mark.parametrize("levels,n_steps,K,sweep", [((3, 3), 2000, 0, "cluster"), ((2,), 2000, 0, "cluster"),
                                                     ((3, 3), 300, 25, "resident")])
def test_autotune_within_the_fixed_point_range(L, levels, n_steps, K, sweep):
    """The kernels that run are the ones timed: chunks over a long horizon; with
    checkpoints one CTA per state, whose forward sweep predicts.  choice[2] is
    theirs: chunks of about 0.8 sqrt(steps), or two threads per element."""
    p = W.random_problem(823, levels=levels, n_states=2, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.01, ckpt_every=K)
    s = _sys(p)
    G, g = s.gradient()
    c = s.autotune(probe_steps=20)
    assert (c["sweep"], c["solver"]) == (sweep, "jacobi")
    if sweep == "cluster":
        per = round(0.8 * np.sqrt(n_steps))
        assert c["shape"] == -(-n_steps // per)
    else:
        assert c["shape"] == (2 * 45 + 31) // 32 * 32
    Gt, gt = _fixed_after(s)
    assert abs(Gt - G) <= 1e-12 * abs(G) and _rel(gt, g) < 1e-11


def _large(state, n_states=1):
    """Four four-level qudits (N^2 = 65536) from and to peaked or spread matrices."""
    p = W.prefix(W.config4(n_states=n_states), 12)
    if state != "spread":
        p.rho0 = np.stack([_basis((4,) * 4, 0, k) for k in range(n_states)])
        if state == "peaked":
            p.targets = np.stack([_basis((4,) * 4, 255, 254 - k) for k in range(n_states)])
    return p


@gpu
def test_peaked_states_of_large_systems_keep_fp64(L):
    """Entries are rounded to their state's largest: on the large grids a state
    of one entry is served by FP64, and is its results; small systems and spread
    states stay in fixed point.  The caller's vectors decide for lb_propagate."""
    for state, want in (("spread", "fixed"), ("peaked", "f64"), ("from", "f64")):
        p = _large(state)
        s, f = _sys(p), _sys(p, arithmetic=L.LB_ARITH_F64)
        G, g = s.gradient()
        assert s.stats()["arithmetic"] == want
        Gf, gf = f.gradient()
        assert abs(G - Gf) <= 1e-12 * abs(Gf) and _rel(g, gf) < 1e-9
        if want == "f64":
            assert G == Gf and np.array_equal(g, gf)
    s = _sys(_large("spread", 3))
    x = _vectors(3, 256)
    s.propagate(x, 0, 3)
    assert s.stats()["arithmetic"] == "fixed"
    x[1] = torch.from_numpy(_basis((4,) * 4, 3, 7)).cuda()
    y = s.propagate(x, 0, 3, adjoint=True)
    assert s.stats()["arithmetic"] == "f64"
    f = _sys(_large("spread", 3), arithmetic=L.LB_ARITH_F64)
    assert torch.equal(y, f.propagate(x, 0, 3, adjoint=True))
    q = W.random_problem(824, levels=(4, 4, 4), n_states=1, n_steps=5, T_ns=0.05, amp=0.02, ckpt_every=0)
    q.rho0 = _basis((4, 4, 4), 0, 0)[None]
    t = _sys(q, sweep=L.LB_SWEEP_GRID)
    t.gradient()
    _fixed(t)


@gpu
def test_products_of_peaked_vectors(L):
    """Per vector: one of spread entries, one of a single large entry among
    entries of 1e-13, whose products keep their own 53 bits away from it."""
    p = _large("spread", 6)
    s = _sys(p)
    x = _vectors(6, 256)
    x[1] *= 1e-13
    x[1, 0, 0] = 1.0
    for adj in (False, True):
        y, ref = s.apply(x, 5, adjoint=adj), _apply_ref(p, x, 5, adj)
        err = (y - ref).abs()
        assert float(err[0].amax()) <= 2.0**-50 * float(_term_bound(p, x, 5)[0])
        # entries that neither the large one nor its neighbours reach
        small = x.clone()
        small[1, 0, 0] = 0.0
        far = torch.ones(256, 256, dtype=torch.bool, device="cuda")
        far[0, :] = far[:, 0] = False
        far[:, :2] = far[:2, :] = False
        for st in (1, 4, 16, 64):
            far[st, :] = far[:, st] = False
        assert float(err[1][far].amax()) <= 2.0**-48 * float(_term_bound(p, small, 5)[1])


@gpu
@pytest.mark.parametrize("levels,penalty", [((2,), 0.0), ((3, 3), 0.0), ((3, 3), 0.3), ((11,), 0.0)])
@pytest.mark.parametrize("n_steps", [23, 24, 25, 40])
def test_the_shortest_horizons_in_chunks(L, levels, penalty, n_steps):
    """Three chunks of eight steps and around: a last chunk of one step, none."""
    p = W.random_problem(825, levels=levels, n_states=2, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.01, hermitian=False,
                         ckpt_every=0)
    if levels == (11,):
        p.system.selfkerr_ghz[:] = 0.01
    p.gamma1, p.penalty_a = penalty, 0.1
    s = _sys(p)
    G, g = s.gradient()
    assert (_fixed(s).stats()["kernel_launches"] > 8) == (n_steps >= 24)
    Go, go, _ = imr.gradient(p)
    assert abs(G - Go) <= 1e-10 * abs(Go)
    assert _rel(g, go) < 1e-9


@gpu
@pytest.mark.parametrize("K", [0, 100])
def test_fp64_sweeps_over_the_whole_cnot_horizon(L, K):
    """The CNOT workload's 10000 steps in both arithmetics, to the method's targets."""
    p = W.config2()
    s, f = _sys(p, ckpt_every=K), _sys(p, ckpt_every=K, arithmetic=L.LB_ARITH_F64)
    G, g = _fixed_after(s)
    Gf, gf = f.gradient()
    assert f.stats()["arithmetic"] == "f64"
    assert abs(G - Gf) <= 1e-10 * abs(Gf) and _rel(g, gf) < 1e-9


@gpu
def test_batch_statistics_name_the_arithmetic(L):
    """Of the sweeps that ran: the graph's, or FP64 while the controls are out of
    the fixed-point range, or while one member asks for FP64."""
    from paper_2110_10310_gb300.system import LindbladBatch

    ps = [W.random_problem(826 + k, levels=lv, n_states=2, n_steps=12, T_ns=0.12, amp=0.02, ckpt_every=0)
          for k, lv in enumerate([(2,), (3, 2)])]
    ss = [_sys(p, sweep=L.LB_SWEEP_RESIDENT) for p in ps]
    b, st = LindbladBatch(ss), torch.cuda.Stream()
    for capture in (False, True):
        if capture:
            b.capture(1, stream=st)
        for scale, want in ((1.0, "fixed"), (40.0, "f64"), (1.0, "fixed")):
            ss[1].set_alpha(scale * ps[1].controls.alpha)
            b.gradient(stream=st)
            assert b.stats()["arithmetic"] == want
    m = LindbladBatch([ss[0], _sys(ps[1], sweep=L.LB_SWEEP_RESIDENT, arithmetic=L.LB_ARITH_F64)])
    m.gradient()
    assert m.stats()["arithmetic"] == "f64"

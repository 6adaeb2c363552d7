"""The fixed-point sweeps at the limits of their arithmetic: states that grow,
cancel, vanish or decay between two rescalings, peaked states, tables that do
not fit, and the calls that share their buffers.

Tolerances: the method's accuracy targets against the oracle (states and
objective 1e-10, gradient 1e-9 of the largest entry) unless a test derives its
own."""

import copy
import ctypes

import numpy as np
import pytest

import workloads as W
from oracle import imr, model

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
@pytest.mark.parametrize("n_steps,theta,weight,sweep", [(24, 0.7796, 1.0, "resident"), (64, np.pi / 4.5, 1.06, "cluster")])
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
@pytest.mark.parametrize("levels,n_steps,sweep", [((2, 2), 24, 1), ((2, 2), 80, 0), ((3, 2, 3), 10, 1), ((3, 3), 20, 2)])
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

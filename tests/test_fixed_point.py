"""The fixed-point sweeps: their arithmetic (lb_fixed.cuh, compiled for the
host from the kernel source) against exact integers, and the kernels against
the oracle at the sizes where their plans change.

Tolerances: a product is its exact value to within two units (its rounding and
the left-out low product); the sweeps' rounding is below FP64's, so the
method's accuracy targets (states and objective 1e-10, gradient 1e-9) and the
agreement of two orderings of the same arithmetic (1e-11, the solver's
tolerance of 1e-15 per step over some hundred steps) hold as for FP64."""

import copy
import importlib
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "lb_fixed.cuh"
int main() {
  long long ax, ay, x, y;
  while (std::scanf("%lld %lld %lld %lld", &ax, &ay, &x, &y) == 4) {
    const lbk::Fx a = lbk::fx_coef(ax), b = lbk::fx_coef(ay), s = lbk::fx_split(x);
    lbk::Cx t; t.x = x; t.y = y;
    const lbk::Cx r = lbk::fx_cmul(a, b, t);
    std::printf("%d %d %d %d %lld %lld %u %u %lld %lld\n", a.h, a.l, s.h, s.l, r.x, r.y, lbk::fx_hi_abs(x),
                lbk::fx_abs_sat(y), lbk::fx_shift(x, 2), lbk::fx_shift(x / 8, -2));
  }
  return 0;
}
"""


def test_products_are_exact_to_two_units(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    B = importlib.import_module("paper_2110_10310_gb300.build")
    src, exe = tmp_path / "h.cu", str(tmp_path / "h")
    src.write_text(HARNESS)
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-I", B.CSRC, "-o", exe, str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    rng = random.Random(5)
    one, top = 1 << 64, 1 << 61
    big = int(0.47 * one)
    cases = [(-big, 0, top, -top), (big, 0, top, top), (0, -big, -top, 1), (0, big, top, -top), (1, -1, -1, 0),
             (0, 0, 0, 0), (int(0.33 * one), -int(0.33 * one), top, -top)]
    for _ in range(2000):
        a = [rng.randrange(-big, big) * 0.7 for _ in range(2)]
        k = rng.randrange(0, 62)
        cases.append((int(a[0]) >> k, int(a[1]) >> k, rng.randrange(-top, top) >> rng.randrange(0, 40),
                      rng.randrange(-top, top)))
    inp = "\n".join(" ".join(str(v) for v in c) for c in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, timeout=60).stdout.split("\n")
    low = 0.0
    for (ax, ay, x, y), line in zip(cases, out):
        ah, al, sh, sl, rx, ry, hx, ya, d2, u2 = (int(v) for v in line.split())
        assert ah * 2**32 + al == ax and sh * 2**32 + sl == x
        assert -2**31 <= min(al, sl) and max(al, sl) < 2**31
        ex, ey = ax * x - ay * y, ax * y + ay * x  # times 2^64
        assert abs(rx * one - ex) <= 2 * one and abs(ry * one - ey) <= 2 * one
        low += (rx * one - ex) / one
        assert hx == ((abs(x) if x >= 0 else -x - 1) >> 32) and ya == min(abs(y), 2**32 - 1)
        assert d2 == (x + 2) >> 2 and u2 == int(x / 8) * 4 if abs(x) < 2**53 else True
    assert abs(low / len(cases)) < 0.1  # unbiased


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


def _problem(levels, n_steps, herm, K=-1, n_states=2, **kw):
    """A driven, decaying problem with the iteration-matrix bound below 1/16."""
    p = W.random_problem(801, levels=levels, n_states=n_states, n_steps=n_steps, T_ns=0.01 * n_steps, amp=0.02,
                         hermitian=herm, ckpt_every=K, **kw)
    return p


def _against_oracle(p, **kw):
    from oracle import imr

    s = _sys(p, **kw)
    G, rho = s.forward(want_states=True)
    Gg, g = s.gradient()
    Go, go, fw = imr.gradient(p)
    assert abs(G - Go) <= 1e-10 * abs(Go) and abs(Gg - Go) <= 1e-10 * abs(Go)
    assert _rel(rho.cpu().numpy(), fw["rhoT"]) < 1e-10
    assert _rel(g, go) < 1e-9
    return s, G, g


# the edges of the plans: one element; a chunk's last step alone (65 steps of
# at least 8); the largest state in chunks (144) and the first past it; 256
# elements, the register plan's last; the table path with one and two elements
@gpu
@pytest.mark.parametrize("levels,n_steps,herm,K", [
    ((2,), 63, False, 0), ((2,), 64, True, 0), ((2,), 65, False, 0), ((3, 3), 81, False, 0), ((3, 3), 81, True, 7),
    ((3, 4), 66, False, 0), ((11,), 70, False, 0), ((13,), 64, False, 0), ((2, 2, 2, 2), 20, False, 0),
    ((4, 4), 64, True, 0), ((17,), 12, False, 0), ((3, 2, 3), 12, False, 5), ((5, 5), 10, True, 0),
    ((2, 2, 2, 2, 2), 6, True, 0)])
def test_small_states_match_the_oracle(L, levels, n_steps, herm, K):
    sweep = L.LB_SWEEP_RESIDENT if int(np.prod(levels)) >= 32 else L.LB_SWEEP_AUTO
    _against_oracle(_problem(levels, n_steps, herm, K), sweep=sweep)


# objectives, couplings and the penalty in chunks of steps, against the
# sequential one-CTA sweep too
@gpu
@pytest.mark.parametrize("objective,jc,penalty,zero_pen", [
    ("frob", 0.0, 0.3, 3.0), ("trace", 0.0, 0.2, 0.004), ("frob", 0.02, 0.0, 1.0), ("trace", 0.02, 0.3, 1.0)])
def test_chunks_match_the_sequential_sweep(L, objective, jc, penalty, zero_pen):
    p = _problem((3, 2), 150, False, 0, n_states=3, objective=objective, jc=jc)
    p.gamma1, p.penalty_a = penalty, zero_pen  # a narrow penalty is zero on all but the last steps
    s, G, g = _against_oracle(p)
    assert s.stats()["sweep"] == "cluster"
    r = _sys(p, sweep=L.LB_SWEEP_RESIDENT)
    Gr, gr = r.gradient()
    assert abs(G - Gr) <= 1e-12 * abs(Gr) and _rel(g, gr) < 1e-11


@gpu
def test_largest_one_cta_state_and_its_scale(L):
    """N = 64 on every element plan (all elements, k <= l) against the FP64
    sweep (the Neumann iteration), from states and targets of magnitudes that
    move the scale: 1e-200 and 1e200 in one problem."""
    for herm in (False, True):
        p = _problem((4, 4, 4), 24, herm, 0, n_states=2)
        p.rho0[0] *= 1e-3
        p.weights = np.array([1.0, 2.0])
        G, g = _sys(p, sweep=L.LB_SWEEP_RESIDENT).gradient()
        Gn, gn = _sys(p, sweep=L.LB_SWEEP_RESIDENT, solver=L.LB_SOLVER_NEUMANN).gradient()
        assert abs(G - Gn) <= 1e-12 * abs(Gn) and _rel(g, gn) < 1e-11
    p = _problem((3, 2), 40, False, 0)
    s = _sys(p, sweep=L.LB_SWEEP_RESIDENT)
    _, rho = s.forward(want_states=True)
    for f in (1e-200, 1e200):
        q = copy.deepcopy(p)
        q.rho0 = p.rho0 * f
        q.targets = p.targets * f
        _, r2 = _sys(q, sweep=L.LB_SWEEP_RESIDENT).forward(want_states=True)
        assert _rel(r2.cpu().numpy() / f, rho.cpu().numpy()) < 1e-13


@gpu
@pytest.mark.parametrize("sweep", ["auto", "resident"])
def test_scale_follows_states_that_decay_or_gather(L, sweep):
    """A coherence that decays to 4e-7 and a mixed state that gathers into one
    entry (24 shifts of the scale and more)."""
    p = W.random_problem(803, levels=(3,), n_states=2, n_steps=600, T_ns=90.0, amp=0.0005, hermitian=False,
                         ckpt_every=0)
    p.system.t1_us, p.system.t2_us = np.array([0.01]), np.array([0.01])
    p.system.detuning_ghz[:] = 0.01
    p.system.selfkerr_ghz[:] = 0.01
    p.rho0 = np.zeros((2, 3, 3), dtype=np.complex128)
    p.rho0[0, 0, 2] = 1.0
    p.rho0[1] = np.eye(3) / 3.0
    _against_oracle(p, sweep=L.LB_SWEEP_RESIDENT if sweep == "resident" else L.LB_SWEEP_AUTO)


@gpu
def test_batch_in_and_out_of_the_fixed_point_range(L):
    """A batch whose controls leave the fixed-point sweeps' range after its
    graph was captured runs the FP64 sweeps, and comes back."""
    from paper_2110_10310_gb300.system import LindbladBatch

    ps = [_problem(lv, 30, True, 0) for lv in [(2,), (3, 2), (4, 4), (4, 2, 3), (4, 4, 2)]]
    ss = [_sys(p, sweep=L.LB_SWEEP_RESIDENT) for p in ps]
    b = LindbladBatch(ss)
    st = torch.cuda.Stream()
    G0, g0 = b.gradient()
    b.capture(1, stream=st)
    G1, g1 = b.gradient(stream=st)
    assert np.array_equal(G0, G1) and np.array_equal(g0, g1)
    ss[1].set_alpha(40.0 * ps[1].controls.alpha)
    G2, g2 = b.gradient(stream=st)
    off = ss[0].n_params
    one, gone = _sys(ps[1], sweep=L.LB_SWEEP_RESIDENT), None
    one.set_alpha(40.0 * ps[1].controls.alpha)
    Go, gone = one.gradient()
    assert abs(G2[1] - Go) <= 1e-12 * abs(Go) and _rel(g2[off:off + len(gone)], gone) < 1e-11
    assert np.all(np.abs(G2[[0, 2, 3, 4]] - G0[[0, 2, 3, 4]]) <= 1e-12 * np.abs(G0[[0, 2, 3, 4]]))
    ss[1].set_alpha(ps[1].controls.alpha)
    G3, g3 = b.gradient(stream=st)
    assert np.array_equal(G3, G0) and np.array_equal(g3, g0)


# the grid sweep in fixed point: elements packed or not, several states per
# block and one state over many, checkpoints, subsystem counts with an unrolled
# loop (3, 4) and without
@gpu
@pytest.mark.parametrize("levels,n_states,herm,K,objective", [
    ((3, 3), 3, True, 0, "frob"), ((2, 3), 9, False, 5, "trace"), ((3, 2, 4), 2, True, 7, "frob"),
    ((2, 2, 2, 2), 5, False, 0, "frob"), ((2, 3, 2, 2), 2, True, 4, "trace"), ((5,), 40, True, 0, "frob")])
def test_grid_sweep_matches_the_oracle(L, levels, n_states, herm, K, objective):
    p = _problem(levels, 23, herm, K, n_states=n_states, objective=objective)
    s, G, g = _against_oracle(p, sweep=L.LB_SWEEP_GRID)
    st = s.stats()
    assert st["sweep"] == "grid" and st["phase_diff_iterations"] == [0, 0, 0]
    r = _sys(p, sweep=L.LB_SWEEP_RESIDENT)
    Gr, gr = r.gradient()
    assert abs(G - Gr) <= 1e-12 * abs(Gr) and _rel(g, gr) < 1e-11
    # steps on given vectors, both directions, against the one-CTA sweep
    rng = np.random.default_rng(4)
    N = int(np.prod(levels))
    x = torch.from_numpy(rng.standard_normal((2, N, N)) + 1j * rng.standard_normal((2, N, N))).cuda()
    for adj in (False, True):
        a = s.propagate(x, 3, 17, adjoint=adj).cpu().numpy()
        b = r.propagate(x, 3, 17, adjoint=adj).cpu().numpy()
        assert _rel(a, b) < 1e-13


# The last checkpoint segment's stage vectors come from the forward sweep: the
# gradient is bitwise the full tape's with the same predictor restarts, whether
# the last segment is the only one, full, or a single step.
@gpu
@pytest.mark.parametrize("levels,sweep", [((2, 2), "resident"), ((3, 2, 3), "resident"), ((7, 4), "resident"),
                                          ((3, 3), "grid")])
@pytest.mark.parametrize("K", [1, 8, 11, 23, 24, 60])
def test_last_segment_kept_by_the_forward_sweep(L, levels, sweep, K):
    p = _problem(levels, 24, True, 0, n_states=2)
    sw = {"resident": L.LB_SWEEP_RESIDENT, "grid": L.LB_SWEEP_GRID}[sweep]
    G0, g0 = _sys(p, ckpt_every=0, predictor=K, sweep=sw).gradient()
    s = _sys(p, ckpt_every=K, sweep=sw)
    for _ in range(2):
        G, g = s.gradient()
        assert G == G0 and np.array_equal(g, g0)
        st = s.stats()
        assert st["phase_steps"][1] == st["phase_steps"][0] and st["phase_iterations"][1] == st["phase_iterations"][0]


# A recorded call serves controls of any size on replay: it is the FP64 sweeps
# that are recorded, whatever the controls were then.
@gpu
@pytest.mark.parametrize("sweep", ["auto", "resident", "grid"])
def test_recorded_gradient_replays_with_larger_controls(L, sweep):
    sw = {"auto": L.LB_SWEEP_AUTO, "resident": L.LB_SWEEP_RESIDENT, "grid": L.LB_SWEEP_GRID}[sweep]
    p = _problem((3, 2), 70, True, 0)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = _sys(p, sweep=sw)
        G, g = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros(s.n_params, dtype=torch.float64,
                                                                               device="cuda")
        s.gradient()
        assert s.stats()["arithmetic"] == "fixed"
        s.set_alpha(p.controls.alpha)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            s.gradient_async(G, g, stream=st)
        for scale in (1.0, 40.0):
            s.set_alpha(scale * p.controls.alpha)
            graph.replay()
            torch.cuda.synchronize()
            q = copy.deepcopy(p)
            q.controls.alpha = scale * p.controls.alpha
            Go, go = _sys(q, sweep=sw).gradient()
            assert abs(float(G) - Go) <= 1e-12 * abs(Go) and _rel(g.cpu().numpy(), go) < 1e-11

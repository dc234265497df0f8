"""The full-velocity-grid step's fixed-point kernel against the FP64 CPU
oracle where it can go wrong: velocity counts that fill neither lanes nor
warps, more columns than lanes, shifts beyond the domain, grids it leaves to
the FP64 kernel, and states out of its range.  Tolerances as in
test_gpu_fixed.py."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_0903_4044_gb300 import bgk as B
from paper_0903_4044_gb300 import build, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    oracle.build()
    B.lib()


def pair(nv, nx=9, **over):
    w = dict(mach=1.5, nx=nx, length=0.5 * nx, nv=nv, vx=(-4.5, 6.0), vt=(-4.5, 4.5), omega=0.74, dt=0.09)
    w.update(over)
    s = solver.make_shock3v(w)
    prob, f = oracle.shock3v_problem(**w)
    rng = np.random.default_rng(5)
    f = f * (1.0 + 0.01 * rng.uniform(-1, 1, f.shape))
    return s, prob, f


def check(s, prob, f, steps=2, signed=False):
    s.set_state(np.ascontiguousarray(f))
    s.step(steps)
    want, mom = oracle.step3v(prob, f.copy(), steps)
    got, m = s.get_state(), s.moments(which=1)
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
    if not signed:
        # the effective parameters stop within 1e-13 of each other and a value
        # moves |c - U|^2 / theta <= 77 times as much (box corner): 8e-12
        bad = np.abs(got - want) > 8e-12 * np.abs(want)
        assert not bad.any(), (bad.sum(), (np.abs(got - want)[bad] / np.abs(want)[bad]).max(), np.abs(want)[bad].max())
    assert np.abs(m - mom).max() <= 1e-12 * np.abs(mom).max()
    s.sync()
    s.close()


@pytest.mark.parametrize("nv", [(16, 16, 16), (30, 30, 30), (13, 11, 9), (33, 10, 12), (64, 9, 10), (9, 64, 10), (10, 9, 17),
                                (65, 9, 9), (12, 14, 1), (22, 31, 19), (20, 31, 22), (13, 29, 19)])
def test_velocity_grids(nv):
    check(*pair(nv, conservative=0 if min(nv) == 1 else 1))


@pytest.mark.parametrize("over", [dict(dt=1.9), dict(conservative=0), dict(relax_exact=0), dict(nx=1), dict(mach=3.0, vx=(-8.0, 10.0))])
def test_options(over):
    check(*pair((18, 14, 14), **over))


@pytest.mark.parametrize("what", ["negative", "zero", "front", "off-axis"])
def test_states_out_of_range(what):
    s, prob, f = pair((14, 12, 13), conservative=0)
    j = np.arange(f.shape[1])
    if what == "negative":
        f[4, j % 17 == 0] *= -0.01
    elif what == "zero":
        f[4, j % 3 == 0] = 0.0
    elif what == "front":
        f[5:] *= 1e9
    else:
        f[4, 3] += 20 * f.max()  # above the sampled range; more would leave theta a difference of large terms
    check(s, prob, f, 1, what == "negative")

@pytest.mark.parametrize("nv", [(16, 16, 16), (49, 16, 16), (16, 49, 16), (14, 16, 49)])
def test_symmetric_state_has_the_velocity_of_the_box_centre(nv):
    # as in test_gpu_fixed.py: f2 - f1 = 0 in a uniform state, so f~ = f exactly
    rest = (1.0, 0.0, 0.0, 0.0, 1.0)
    s = solver.Solver3v(B.make_config3v(nx=8, lx=4.0, nv=nv, vmin=(-4.0,) * 3, vmax=(4.0,) * 3, cfl=0.5, conservative=0,
                                        inflow=(rest, rest)))
    c = [-4.0 + (np.arange(n) + 0.5) * (8.0 / n) for n in nv]
    x, y, z = (np.exp(-np.maximum(np.abs(a), np.abs(a[::-1])) ** 2) for a in c)
    f = (z[:, None, None] * y[:, None] * x).ravel()
    s.set_state(np.tile(f, (8, 1)))
    s.step(1)
    mid = np.array([float(Fraction(-4) + n * Fraction(8.0 / n) / 2) for n in nv])
    assert np.abs(s.moments(which=1)[2:-2, 1:4] - mid).max() <= 2.0 ** -54
    s.close()


def test_effective_parameters_at_the_range_end():
    # as in test_gpu_1d_fixed.py (the other end is the sums' own, which lie further out)
    n = 2.0 ** 97 * 0.99
    c = -8.0 + (np.arange(12) + 0.5) * (16.0 / 12)
    e = np.exp(-c * c)
    f = (e[:, None, None] * e[:, None] * e).ravel()
    f *= n / (f.sum() * (16.0 / 12) ** 3)
    end = (n, 0.0, 0.0, 0.0, 1.0)
    s = solver.Solver3v(B.make_config3v(nx=8, lx=4.0, nv=(12,) * 3, vmin=(-8.0,) * 3, vmax=(8.0,) * 3, cfl=0.5, omega=1.0,
                                        inflow=(end, end)))
    s.set_state(np.tile(f, (8, 1)))
    s.step(1)
    s.sync()
    assert np.abs(s.moments(which=1)[2:-2, 0] / n - 1.0).max() <= 1e-12
    s.close()

"""The 1D FP64 step that keeps a cell on one warp against the FP64 CPU oracle:
every number of velocities per lane and its remainders, grids it leaves to the
FP64-only kernel, shifts, options, and states out of its range.  Tolerances as
in test_gpu_fixed.py."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_0903_4044_gb300 import bgk as B
from paper_0903_4044_gb300 import build, solver
from paper_0903_4044_gb300 import workloads as W
from test_gpu_fixed import tail_state
from test_gpu_parity import assert_moments_close, assert_state_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    oracle.build()
    B.lib()


def pair(**over):
    w = W.scaled(W.SHOCK_M2, **{**dict(nx=23, length=8.0), **over})
    s = solver.make_shock(w)
    prob, g, h = oracle.shock_problem(**w)
    rng = np.random.default_rng(2)
    return s, prob, g * (1.0 + 0.01 * rng.uniform(-1, 1, g.shape)), h * (1.0 + 0.01 * rng.uniform(-1, 1, h.shape))


def run(s, prob, g, h, steps=3):
    s.set_state(np.ascontiguousarray(np.stack([g, h], -1)))
    s.step(steps)
    g1, h1, mom = oracle.step(prob, g, h, steps)
    return s.get_state(), s.moments(which=1), g1, h1, mom


@pytest.mark.parametrize("nvx,vbox", [(24, 6.0), (31, 6.0), (32, 6.0), (33, 7.0), (64, 8.0), (65, 8.0), (97, 9.0), (128, 9.0),
                                      (129, 10.0), (160, 10.0), (161, 10.0), (200, 10.0)])
def test_velocity_counts(nvx, vbox):
    s, prob, g, h = pair(nvx=nvx, vx=(-vbox, vbox + 1.0), tile_cells=(1, 2, 4, 8)[nvx % 4])
    st, m, g1, h1, mom = run(s, prob, g, h)
    assert_state_close(st, g1, h1)
    assert_moments_close(m, mom, vscale=1.0)
    s.close()


@pytest.mark.parametrize("over", [dict(cfl=2.6), dict(omega=0.74), dict(omega=0.74, mach=5.0, nvx=96, vx=(-19.0, 19.0)),
                                  dict(conservative=0), dict(relax_exact=0), dict(nx=1), dict(length=4000.0)])
def test_options(over):
    s, prob, g, h = pair(**over)
    st, m, g1, h1, mom = run(s, prob, g, h)
    if "length" in over or "mach" in over:
        # the effective parameters stop within 1e-13 of each other and a value
        # moves |c - U|^2 / theta times as much (64 and 555 at the box's end)
        bound = 7e-12 if "length" in over else 6e-11
        assert (np.abs(st[..., 0] - g1) <= bound * np.abs(g1)).all()
    else:
        assert_state_close(st, g1, h1)
    assert_moments_close(m, mom, vscale=1.0)
    s.close()


@pytest.mark.parametrize("what", ["negative", "zero", "front", "scale"])
def test_states_out_of_range(what):
    s, prob, g, h = pair(conservative=0)
    j = np.arange(prob.nv)
    if what == "negative":
        g[9, j % 13 == 0] *= -0.01
        h[12, j % 7 == 0] *= -0.01
    elif what == "zero":
        g[9, j % 3 == 0] = 0.0
        h[13] = 0.0
    elif what == "front":
        g[12:] *= 1e9
        h[12:] *= 1e9
    else:
        g[8:15] *= 1e60
        h[8:15] *= 1e60
    st, m, g1, h1, mom = run(s, prob, g, h, 1)
    for a, b in ((st[..., 0], g1), (st[..., 1], h1)):
        assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
        if what != "negative":
            assert (np.abs(a - b) <= 1e-12 * np.abs(b)).all()
    assert_moments_close(m, mom, vscale=1.0)
    s.close()


@pytest.mark.parametrize("nvx", [32, 64, 96, 160])
def test_sums_of_a_tail_on_a_wide_box(nvx):
    # as in test_gpu_fixed.py, in the cells that the ends do not reach
    box, nx = 20.0, 12
    rest = (1.0, 0.0, 0.0, 1.0)
    s = solver.Solver(B.make_config(dim=1, nx=nx, lx=6.0, nvx=nvx, vx=(-box, box), cfl=0.5, conservative=0,
                                    bc=[(B.BGK_BC_INFLOW, *rest)] * 2))
    g, h, n, theta = tail_state((nvx,), box, nx)
    s.set_state(np.ascontiguousarray(np.stack([g, h], -1)))
    s.step(1)
    m = s.moments(which=1)[2:-2]
    assert np.abs(m[:, 0] / n - 1.0).max() <= 8 * 2.0 ** -53
    assert np.abs(m[:, 3] / theta - 1.0).max() <= 8 * 2.0 ** -53
    s.close()

@pytest.mark.parametrize("nvx", [32, 49])
def test_symmetric_state_has_the_velocity_of_the_box_centre(nvx):
    # as in test_gpu_fixed.py; the streaming weights are mirrored within a rounding only
    rest = (1.0, 0.0, 0.0, 1.0)
    s = solver.Solver(B.make_config(dim=1, nx=12, lx=6.0, nvx=nvx, vx=(-4.0, 4.0), cfl=0.5, conservative=0,
                                    bc=[(B.BGK_BC_INFLOW, *rest)] * 2))
    c = -4.0 + (np.arange(nvx) + 0.5) * (8.0 / nvx)
    g = np.exp(-np.maximum(np.abs(c), np.abs(c[::-1])) ** 2)
    s.set_state(np.tile(np.stack([g, 0.5 * g], -1), (12, 1, 1)))
    s.step(1)
    mid = float(Fraction(-4) + nvx * Fraction(8.0 / nvx) / 2)
    assert np.abs(s.moments(which=1)[2:-2, 1] - mid).max() <= 2.0 ** -54
    s.close()


@pytest.mark.parametrize("n,nvx", [(2.0 ** -95 * 1.003, 11), (2.0 ** 97 * 0.997, 12)])
def test_effective_parameters_at_the_range_ends(n, nvx):
    # on 11 velocities a Maxwellian's sum exceeds its integral by 2 %, on 12 it falls short by 1 to 2 %: the effective
    # density leaves the range of the FP32 starts when the density is just inside
    c = -8.0 + (np.arange(nvx) + 0.5) * (16.0 / nvx)
    g = np.exp(-c * c)
    g *= n / (g.sum() * (16.0 / nvx))
    s = solver.Solver(B.make_config(dim=1, nx=8, lx=4.0, nvx=nvx, vx=(-8.0, 8.0), cfl=0.5, omega=1.0,
                                    bc=[(B.BGK_BC_INFLOW, n, 0.0, 0.0, 1.0)] * 2))
    s.set_state(np.tile(np.stack([g, g], -1), (8, 1, 1)))
    s.step(1)
    s.sync()
    assert np.abs(s.moments(which=1)[2:-2, 0] / n - 1.0).max() <= 1e-12
    s.close()


def test_collisions_keep_density_and_temperature():
    # as in test_gpu_fixed.py, in cells that the ends do not reach (FP64-only form: 0.058 and 0.046)
    drift = []
    for box in (5.6, 5.7, 5.83, 6.0, 6.1, 6.25):
        for n, theta in ((24, 1.0), (28, 0.93), (31, 1.07)):
            s = solver.Solver(B.make_config(dim=1, nx=220, lx=8800.0, nvx=n, vx=(-box, box), cfl=0.5,
                                            bc=[(B.BGK_BC_INFLOW, 1.0, 0.0, 0.0, theta)] * 2))
            c = -box + (np.arange(n) + 0.5) * (2 * box / n)
            for density in np.linspace(1.0, 1.9, 10):
                g = density * np.exp(-c * c / theta) / np.sqrt(np.pi * theta)
                s.set_state(np.tile(np.stack([g, theta * g], -1), (220, 1, 1)))
                s.step(1)
                m0 = s.moments(which=1)[105:115]
                s.step(100)
                drift.append((s.moments(which=1)[105:115, [0, 3]] / m0[:, [0, 3]] - 1.0).mean(0) / 100 * 2.0 ** 53)
            s.close()
    rms = np.sqrt((np.array(drift) ** 2).mean(0))
    assert (rms <= 0.065).all(), rms

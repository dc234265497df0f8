"""The 2D FP64 step's fixed-point kernels against the FP64 CPU oracle where
they can go wrong: velocity rows that fill no lane count, columns and rows
past the grid, c = 0, Courant number 1, boxes off centre, every number of
warps per cell, and states that leave the fixed-point range (negative and
zero values, steep fronts, densities far from one, relaxation weights beyond
one), for which the kernels fall back to FP64.

Tolerances as in test_gpu_parity.py: 1e-13 of the largest value and 1e-12 of
each value per step.  Each rounds at most five times a step (streaming 3,
relaxation 1, parameters), each to half an ulp of a sum of positive terms.
"""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_0903_4044_gb300 import bgk as B
from paper_0903_4044_gb300 import build, solver
from paper_0903_4044_gb300 import workloads as W
from test_gpu_parity import assert_moments_close, assert_state_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    oracle.build()
    B.lib()


def pair(nx, ny, nvx, nvy, *, tile=0, vx=(-4.0, 4.0), vy=(-4.5, 4.5), cfl=0.6, cons=1, exact=1, kinds=(1, 1, 1, 1),
         omega=0.5, n=1.0, length=0.5, lx=None, ly=None):
    rest, lid = (n, 0.0, 0.0, 1.0), (n, 0.05, 0.0, 1.0)
    kw = dict(dim=2, nx=nx, ny=ny, lx=lx or nx * length, ly=ly or ny * length, nvx=nvx, nvy=nvy, vx=vx, vy=vy, cfl=cfl,
              conservative=cons, relax_exact=exact, omega=omega)
    cfg = B.make_config(**kw, bc=[(k, *s) for k, s in zip(kinds, (rest, rest, rest, lid))], tile_cells=tile)
    prob = oracle.Problem(oracle.make_config(**kw, bc_kind=kinds, bc_state=(rest, rest, rest, lid)))
    xi = W.perturbation(3, prob.ncell, prob.nv)
    g, h = oracle.init_uniform(prob, rest, xi, 1e-2)
    return solver.Solver(cfg), prob, g, h


def run(s, prob, g, h, steps=3):
    s.set_state(np.ascontiguousarray(np.stack([g, h], -1)))
    s.step(steps)
    g1, h1, mom = oracle.step(prob, g, h, steps)
    return s.get_state(), s.moments(which=1), g1, h1, mom


@pytest.mark.parametrize("tile", [1, 2, 4, 8])
@pytest.mark.parametrize("nvx,nvy", [(12, 11), (13, 17), (21, 20), (33, 12), (48, 16), (65, 20), (128, 9)])
def test_velocity_grids(nvx, nvy, tile):
    s, prob, g, h = pair(5, 4, nvx, nvy, tile=tile)
    st, m, g1, h1, mom = run(s, prob, g, h)
    assert_state_close(st, g1, h1)
    assert_moments_close(m, mom, vscale=0.05)
    s.close()


@pytest.mark.parametrize("case", [
    dict(cfl=1.0), dict(cfl=1.0, vx=(-4.2, 4.2), vy=(-3.9, 3.9)), dict(vx=(-4.0, 6.0), vy=(-5.0, 4.0), kinds=(0, 0, 1, 1)),
    dict(kinds=(2, 2, 2, 2)), dict(omega=0.74), dict(cons=0), dict(exact=0), dict(n=1e60), dict(n=1e-60),
    dict(n=40.0, exact=0), dict(n=3000.0), dict(vx=(-40.0, 40.0), vy=(-40.0, 40.0), cons=0)])
def test_options(case):
    # nvx and nvy odd: a zero velocity per axis; n = 40 with the Euler form
    # makes the relaxation weight of f~ negative, n = 3000 makes it tiny; the
    # box of +-40 underflows to zeros at its corners
    s, prob, g, h = pair(6, 5, 21, 25, **case)
    steps = 1 if case.get("n") == 40.0 else 3
    st, m, g1, h1, mom = run(s, prob, g, h, steps)
    if case.get("n") == 40.0:  # f~ and Phi subtract: no bound relative to each value
        assert np.abs(st[..., 0] - g1).max() <= 1e-13 * np.abs(g1).max()
        assert np.abs(st[..., 1] - h1).max() <= 1e-13 * np.abs(h1).max()
    elif "vx" in case and case["vx"][1] == 40.0:
        # values below 2.2e-308 are spaced 4.9e-324 apart whatever their size:
        # four spacings (two products and two roundings) beside the 1e-12
        for a, b in ((st[..., 0], g1), (st[..., 1], h1)):
            assert (np.abs(a - b) <= 1e-12 * np.abs(b) + 2e-323).all()
    else:
        assert_state_close(st, g1, h1)
    assert_moments_close(m, mom, vscale=0.05)
    s.close()


@pytest.mark.parametrize("what", ["negative", "zero", "front", "fast"])
def test_states_out_of_range(what):
    s, prob, g, h = pair(6, 5, 24, 20, cons=0, kinds=(2, 2, 2, 2))
    j = np.arange(prob.nv)
    if what == "negative":
        g[7, j % 13 == 0] *= -0.01
        h[11, j % 7 == 0] *= -0.01
    elif what == "zero":
        g[7, j % 3 == 0] = 0.0
        h[8] = 0.0
        h[14, ::2] = 0.0
    elif what == "front":
        g[12:18] *= 1e9
        h[12:18] *= 1e9
    else:  # a beam in a few velocities between the sampled ones
        g[9, 37] += 1e5 * g.max()
        h[9, 38] += 1e5 * h.max()
    st, m, g1, h1, mom = run(s, prob, g, h, 1)
    for a, b in ((st[..., 0], g1), (st[..., 1], h1)):
        assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
        if what != "negative":
            assert (np.abs(a - b) <= 1e-12 * np.abs(b)).all()
    assert_moments_close(m, mom, vscale=0.05)
    s.close()


def test_nan_is_flagged():
    s, prob, g, h = pair(6, 5, 24, 20)
    g[9, 5] = np.nan
    s.set_state(np.ascontiguousarray(np.stack([g, h], -1)))
    s.step(1)
    with pytest.raises(B.BgkError) as e:
        s.sync()
    assert e.value.status == B.BGK_ERR_NUMERIC
    s.close()


@pytest.mark.parametrize("cfl", [1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("what", ["front", "zero"])
def test_small_time_steps(what, cfl):
    # weights far below one decide the values beside a front and where a cell is empty
    s, prob, g, h = pair(6, 5, 24, 20, cons=0, kinds=(2, 2, 2, 2), cfl=cfl)
    if what == "front":
        g[12:18] *= 1e9
        h[12:18] *= 1e9
    else:
        g[7, np.arange(prob.nv) % 3 == 0] = 0.0
        g[8] = 0.0
        g[8, 200:230] = g[9, 200:230]
        h[8] = 0.0
    st, _, g1, h1, _ = run(s, prob, g, h, 1)
    for a, b in ((st[..., 0], g1), (st[..., 1], h1)):
        assert (np.abs(a - b) <= 1e-12 * np.abs(b)).all()
    s.close()


@pytest.mark.parametrize("tile", [1, 8])
def test_sums_beside_a_steep_front(tile):
    # a cell takes 1e-7 of a neighbour 1e14 times as dense: the sums keep the bits of the cell's own values
    s, prob, g, h = pair(6, 5, 24, 20, cons=0, kinds=(2, 2, 2, 2), cfl=1e-7, tile=tile)
    g[12:18] *= 1e14
    h[12:18] *= 1e14
    st, m, g1, h1, mom = run(s, prob, g, h, 1)
    assert_moments_close(m, mom, vscale=0.05, tol=1e-14)
    s.close()


@pytest.mark.parametrize("nvx,nvy,cfl", [(32, 32, 0.5), (48, 48, 0.9), (20, 28, 0.5), (24, 24, 1.0)])
def test_uniform_state_does_not_drift(nvx, nvy, cfl):
    # the weights of f~ sum to one within their roundings, the same every step: without relaxation g, combined
    # in integers, stays as it is, and h, in three FP64 operations, moves by a sixtieth of 2^-53 a step (rms) at
    # most: most values round back.  Two roundings more a step double that
    n, steps = 1e-20, 200
    s = solver.Solver(B.make_config(dim=2, nx=12, ny=12, lx=10.0, ly=10.0, nvx=nvx, nvy=nvy, vx=(-5.0, 5.0), vy=(-5.0, 5.0),
                                    cfl=cfl, conservative=0, bc=[(2, n, 0.0, 0.0, 1.0)] * 4))
    g = n * np.exp(-8.0 * np.random.default_rng(0).random((nvy, nvx)))
    g = np.maximum(g, g[::-1])
    g = np.maximum(g, g[:, ::-1]).ravel()
    f = np.tile(np.stack([g, 0.5 * g], -1), (144, 1, 1))
    s.set_state(f)
    s.step(steps)
    out = s.get_state()
    assert (out[..., 0] == f[..., 0]).all()
    drift = (out[..., 1] / f[..., 1] - 1.0) / steps * 2.0 ** 53
    assert np.sqrt((drift ** 2).mean()) <= 0.02
    s.close()


def tail_state(counts, box, ncell):
    """A resting Maxwellian with a hot tail of 1e-9 on so many velocities per axis in +-box, the same in every cell,
    and its n and theta in extended precision (the centres too: in FP64 each is off by an ulp of the box, up to 4e-15
    of theta on the axis of 300)."""
    exact = [(2 * np.arange(k) + 1 - k) * (np.longdouble(box) / k) for k in counts]
    c = [x.astype(float) for x in exact]
    m = [np.exp(-x * x) for x in c]
    t = [np.exp(-x * x / 50.0) for x in c]
    g = m[0] + 1e-9 * t[0] if len(c) == 1 else m[1][:, None] * m[0] + 1e-9 * t[1][:, None] * t[0]
    h = (0.5 * g).ravel()
    e = exact[0] ** 2 if len(c) == 1 else exact[1][:, None] ** 2 + exact[0] ** 2
    G = g.astype(np.longdouble)
    dv = np.prod([2 * np.longdouble(box) / k for k in counts])
    theta = np.longdouble(2.0) / 3 * ((e * G).sum() + h.astype(np.longdouble).sum()) / G.sum()
    return np.tile(g.ravel(), (ncell, 1)), np.tile(h, (ncell, 1)), float(G.sum() * dv), float(theta)


@pytest.mark.parametrize("tile", [1, 2, 4, 8])
@pytest.mark.parametrize("nvx,nvy,box", [(16, 16, 20.0), (32, 32, 20.0), (64, 64, 20.0), (32, 32, 10.0), (128, 32, 20.0),
                                         (12, 300, 20.0)])
def test_sums_of_a_tail_on_a_wide_box(nvx, nvy, box, tile):
    # tail values 1e-9 of the peak carry most of sum c^2 g's rounding: the integer sums have to keep their low bits.
    # Eight roundings of 2^-53 lie between the sums and theta
    s, prob, *_ = pair(4, 3, nvx, nvy, cons=0, kinds=(2, 2, 2, 2), vx=(-box, box), vy=(-box, box), tile=tile)
    g, h, n, theta = tail_state((nvx, nvy), box, prob.ncell)
    s.set_state(np.ascontiguousarray(np.stack([g, h], -1)))
    s.step(1)
    m = s.moments(which=1)
    assert np.abs(m[:, 0] / n - 1.0).max() <= 8 * 2.0 ** -53
    assert np.abs(m[:, 3] / theta - 1.0).max() <= 8 * 2.0 ** -53
    s.close()

@pytest.mark.parametrize("tile", [1, 2, 4, 8])
@pytest.mark.parametrize("nvx,nvy,broad", [(32, 32, False), (49, 16, False), (16, 49, False), (64, 64, True), (12, 300, True)])
def test_symmetric_state_has_the_velocity_of_the_box_centre(nvx, nvy, broad, tile):
    # g mirrored in both axes: the integer sums over the indices cancel exactly whatever their order (sums in FP64
    # do not) where one warp has the cell (tile 8), else within a rounding of the warps' sums.  What is left is the
    # centre of the tabulated velocities -4 + (j + 1/2) dc, 3e-16 for 49.  broad: all values alike, the largest sums
    # a lane can meet
    s, prob, *_ = pair(4, 3, nvx, nvy, cons=0, kinds=(2, 2, 2, 2), vx=(-4.0, 4.0), vy=(-4.0, 4.0), tile=tile)
    c = [-4.0 + (np.arange(n) + 0.5) * (8.0 / n) for n in (nvx, nvy)]
    g = 0.5 + 0.5 * np.random.default_rng(1).random((nvy, nvx)) * (1 if broad else np.exp(-c[1][:, None] ** 2 - c[0] ** 2))
    g = np.maximum(g, g[::-1])
    g = np.maximum(g, g[:, ::-1]).ravel()
    f = np.tile(np.stack([g, 0.5 * g], -1), (prob.ncell, 1, 1))
    s.set_state(np.ascontiguousarray(f))
    s.step(1)
    m = s.moments(which=1)
    for u, n in ((m[:, 1], nvx), (m[:, 2], nvy)):
        mid = float(Fraction(-4) + n * Fraction(8.0 / n) / 2)
        assert np.abs(u - mid).max() <= 2.0 ** -51 * abs(mid) + (0.0 if tile == 8 else 2.0 ** -53)
    s.close()


def test_time_step_of_the_order_of_the_smallest_numbers():
    # an infinity stays one
    s, prob, g, h = pair(6, 5, 24, 20, cfl=1e-85, cons=0)
    h[9, 5] = np.inf
    s.set_state(np.ascontiguousarray(np.stack([g, h], -1)))
    s.step(1)
    with pytest.raises(B.BgkError) as e:
        s.sync()
    assert e.value.status == B.BGK_ERR_NUMERIC
    s.close()


@pytest.mark.parametrize("nvx", [21, 20])
@pytest.mark.parametrize("sides", [dict(lx=1e22), dict(ly=1e22)])
def test_courant_number_of_one_axis(sides, nvx):
    # cells 1e22 times as long as high or as high as long: the fastest velocity's weight along one axis is one
    s, prob, g, h = pair(6, 5, nvx, 16, cfl=1.0, vy=(-4.0, 4.0), **sides)
    st, m, g1, h1, mom = run(s, prob, g, h, 1)
    assert_state_close(st, g1, h1)
    assert_moments_close(m, mom, vscale=0.05)
    s.close()


@pytest.mark.parametrize("n,nvy", [(2.0 ** -95 * 1.003, 11), (2.0 ** 97 * 0.997, 12)])
def test_effective_parameters_at_the_range_ends(n, nvy):
    # on coarse velocities the effective density lies 1 to 2 % off the density: outside the range of the FP32
    # starts when the density is just inside
    s, prob, g, h = pair(6, 5, 12, nvy, vx=(-8.0, 8.0), vy=(-8.0, 8.0), n=n, kinds=(2, 2, 2, 2), omega=1.0, cfl=0.6)
    st, m, g1, h1, mom = run(s, prob, g, h, 1)
    s.sync()
    assert_moments_close(m, mom, vscale=0.05)
    s.close()


def test_collisions_keep_density_and_temperature():
    # a uniform gas that relaxes by e^-20 a step: its density and temperature are made anew every step by D(p) = q
    # and a Phi of the same p.  Roundings that differ from step to step average out (in units of 2^-53 a step 0.13 and
    # 0.09 rms here for the FP64-only form); a constant rounded once would not
    drift = []
    for box in (5.6, 5.7, 5.83, 6.0, 6.1, 6.25):
        for n, theta in ((24, 1.0), (28, 0.93), (31, 1.07)):
            s = solver.Solver(B.make_config(dim=2, nx=4, ny=4, lx=160.0, ly=160.0, nvx=n, nvy=n, vx=(-box, box),
                                            vy=(-box, box), cfl=0.5, bc=[(2, 1.0, 0.0, 0.0, 1.0)] * 4))
            c = -box + (np.arange(n) + 0.5) * (2 * box / n)
            for density in np.linspace(1.0, 1.9, 10):
                g = density * (np.exp(-(c * c + (c * c)[:, None]) / theta) / (np.pi * theta)).ravel()
                s.set_state(np.tile(np.stack([g, 0.5 * theta * g], -1), (16, 1, 1)))
                s.step(1)
                m0 = s.moments(which=1)
                s.step(100)
                drift.append((s.moments(which=1)[:, [0, 3]] / m0[:, [0, 3]] - 1.0).mean(0) / 100 * 2.0 ** 53)
            s.close()
    rms = np.sqrt((np.array(drift) ** 2).mean(0))
    assert (rms <= 0.16).all(), rms

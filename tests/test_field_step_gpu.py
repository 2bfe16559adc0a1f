"""The fused 2D field update and the current smoothing at the edges of their
strips and stencils (needs a GB300), in FP64 against the oracle: 1e-12 per
step as elsewhere.

The 2D update works in strips of 29 columns with recomputed halos, its walls
and the incoming wave included: grids one column around the strip's width,
one or two rows high, and walls that fall on a strip's first or last column.
The smoothing reaches up to nine cells along an axis: grids shorter than that,
where it wraps more than once.
"""
import math

import numpy as np
import pytest

from oracle import OracleSim
from paper_1503_02464_gb300 import synth
from paper_1503_02464_gb300.sim import Simulation

from _parity import compare_fields, j_floor

pytestmark = pytest.mark.gpu


def _seeded(o, s, seed, amplitude):
    """The same random E and B in both."""
    rng = np.random.default_rng(seed)
    for c in range(6):
        f = amplitude * rng.standard_normal(s.shape3)
        o.set_field(c, f)
        s.set_field(c, f)


@pytest.mark.parametrize("n", [(5, 1), (28, 2), (29, 3), (30, 17), (31, 5), (58, 33), (59, 1), (320, 95)])
def test_periodic_grid(n):
    wl = synth.small(2, n, 2, 1, 0.1, 11)
    o = OracleSim(2, wl.n, wl.d, wl.dt, 2)
    s = Simulation.from_workload(wl, precision="fp64")
    _seeded(o, s, 5, 0.1)
    for step in range(1, 5):
        o.step(1)
        s.step(1)
    fe = compare_fields(o, s)
    assert max(fe.values()) <= 4e-12, fe


@pytest.mark.parametrize("n", [(16, 1), (29, 4), (30, 9), (31, 16), (57, 3), (58, 8), (59, 40), (813, 2)])
@pytest.mark.parametrize("pol,angle", [(1, 0.0), (2, 0.0), (1, 0.4), (2, -0.3)])
def test_walls_and_wave(n, pol, angle):
    d = 0.1
    dt = 0.9 * synth.courant_limit((d, d), 2)
    laser = {"a0": 1.5, "waist": max(0.3 * n[1] * d, 0.2), "duration": 2 * math.pi, "pol": pol, "angle": angle}
    o = OracleSim(2, (*n, 1), (d, d, 1.0), dt, 2)
    o.set_absorbing_x(True)
    o.set_laser(laser["a0"], laser["waist"], laser["duration"], pol=pol, angle=angle)
    s = Simulation(2, n, (d, d), dt, 2, "fp64", absorbing_x=True, laser=laser)
    _seeded(o, s, 7, 0.3)
    for step in range(1, 13):
        o.step(1)
        s.step(1)
        fe = compare_fields(o, s)
        assert max(fe.values()) <= 1e-12 * step, (step, fe)


@pytest.mark.parametrize("dims,n", [(2, (3, 20)), (2, (33, 2)), (3, (5, 4, 3)), (3, (18, 7, 1))])
@pytest.mark.parametrize("passes,comp", [(1, False), (3, True), (8, True)])
def test_smoothing_wraps(dims, n, passes, comp):
    wl = synth.small(dims, n, 2, 3, 0.2, 13)
    p = wl.particles(0)
    o = OracleSim(wl.dims, wl.n, wl.d, wl.dt, wl.order)
    o.add_particles(p, -1.0, 1.0)
    o.set_filter(passes, comp)
    s = Simulation.from_workload(wl, precision="fp64", filter_passes=passes, filter_compensate=comp)
    k = s.add_species(-1.0, 1.0, len(p["x"]))
    s.load(k, p)
    o.step(2)
    s.step(2)
    # the compensating pass amplifies the floor by up to 1 + passes / 2 per axis
    jf = j_floor(wl, [p]) * ((1 + 0.5 * passes) ** dims if comp else 1.0)
    fe = compare_fields(o, s, j_abs=jf)
    assert max(fe.values()) <= 2e-12, fe


@pytest.mark.parametrize("walls", [False, True], ids=["periodic", "mur_walls"])
@pytest.mark.parametrize("n", [(16, 1), (28, 3), (29, 2), (30, 5), (31, 9), (58, 4), (59, 1), (60, 33), (814, 2)])
def test_reversed_field_step_is_the_transpose(n, walls):
    """<A x, y> = <x, A^T y> for one field step without particles, the adjoint's
    strips having their halo on the other side."""
    d = 0.1
    s = Simulation(2, n, (d, d), 0.9 * synth.courant_limit((d, d), 2), 2, "fp64", absorbing_x=walls)
    rng = np.random.default_rng(17)
    x = [rng.normal(size=s.shape3) for _ in range(6)]
    y = [rng.normal(size=s.shape3) for _ in range(6)]
    for c in range(6):
        s.set_field(c, x[c])
    s.tape_begin(1)
    s.step(1)
    ax = [s.field(c) for c in range(6)]
    s.adjoint_begin(1)
    for c in range(6):
        s.adjoint_set_field(c, y[c])
    s.adjoint_step(1)
    aty = [s.adjoint_field(c) for c in range(6)]
    lhs = sum(float((p * q).sum()) for p, q in zip(ax, y))
    rhs = sum(float((p * q).sum()) for p, q in zip(x, aty))
    scale = sum(float(np.abs(p * q).sum()) for p, q in zip(ax, y))
    assert abs(lhs - rhs) <= 1e-13 * scale, (lhs, rhs, scale)
    # (the sum could hide an entry: one unit seed per wall column)
    for c in (1, 2):
        for col in (0, 1, n[0] - 2, n[0] - 1):
            s.tape_begin(1)
            s.step(0)
            s.tape_record()
            s.adjoint_begin(1)
            seed = np.zeros(s.shape3)
            seed[0, 0, col] = 1.0
            s.adjoint_set_field(c, seed)
            s.adjoint_step(1)
            got = sum(float((p * s.adjoint_field(k)).sum()) for k, p in enumerate(x))
            assert abs(got - ax[c][0, 0, col]) <= 1e-13 * 30, (c, col)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [(9, 7, 5), (10, 7, 5), (11, 7, 5), (8, 8, 8), (75, 50, 43)])
def test_current_cleared_before_a_3d_step(n, precision):
    """J starts every step at zero up to its last value, whatever its bytes
    leave of the 16-byte stores (exact: nothing deposits)."""
    wl = synth.small(3, n, 2, 1, 0.1, 11)
    s = Simulation.from_workload(wl, precision=precision)
    for step in range(2):
        for c in (6, 7, 8):
            s.set_field(c, 1.0 + step)
        s.step(1)
        for c in range(9):
            assert not s.field(c).any(), (n, c)

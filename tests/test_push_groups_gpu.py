"""The push's deposit by groups of particles that share a nearest node or
cell (needs a GB300): group lengths around the eight particles one thread
sums at a time, a cell holding more particles than one work item, work items
just below, at and above their largest size, particles that do not move and
particles without weight.  Fields, J and momenta match the oracle, in FP64 to
1e-12 per step and in FP32 to the path's 1e-5.
"""
import numpy as np
import pytest

from paper_1503_02464_gb300 import synth
from paper_1503_02464_gb300.sim import Simulation

from _parity import build_oracle, compare_fields, compare_particles, j_floor, j_floor_fp32

pytestmark = pytest.mark.gpu

# a species of this capacity gets work items of the largest size (its slots
# over 16 items per SM), however few particles it holds
BIG = 7_000_000


def _particles(wl, counts, u_th, seed):
    """counts[c] particles in cell c of the grid; a fifth of them at rest and
    every seventh without weight."""
    one = [synth.particles_for_cells(np.array([c]), wl.n, wl.d, int(k), u_th, 1.0, seed + c, wl.dims)
           for c, k in enumerate(counts) if k > 0]
    p = {k: np.concatenate([q[k] for q in one]) for k in one[0]}
    p["id"] = np.arange(len(p["x"]), dtype=np.uint32)
    still = p["id"] % 5 == 0
    for k in ("ux", "uy", "uz"):
        p[k][still] = 0.0
    p["w"] = np.where(p["id"] % 7 == 3, 0.0, 0.05 + 0.01 * (p["id"] % 11))
    return p


def _compare(wl, p, precision, capacity, steps):
    o = build_oracle(wl, [p])
    s = Simulation.from_workload(wl, precision=precision, sort_every=1000)
    k = s.add_species(-1.0, 1.0, capacity)
    s.load(k, p)
    s.neutralize()
    o.step(steps)
    s.step(steps)
    floor = j_floor(wl, [p]) + (j_floor_fp32(wl, [p]) if precision == "fp32" else 0.0)
    fe = compare_fields(o, s, j_abs=floor)
    du, dx = compare_particles(o, s, wl)
    s.close()
    tol = 1e-12 * steps if precision == "fp64" else 1e-5
    assert max(fe.values()) <= tol and du <= tol, (fe, du)
    assert dx <= (1e-10 if precision == "fp64" else 1e-6)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("dims,n", [(3, (19, 12, 9)), (2, (37, 21))])
@pytest.mark.parametrize("u_th", [0.05, 0.8])
def test_group_lengths(dims, n, order, precision, u_th):
    wl = synth.small(dims, n, order, 1, u_th, 71)
    counts = np.arange(wl.ncells) % 20  # 0 .. 19 particles per cell
    counts[wl.ncells // 2] = 3000       # more than a work item holds
    _compare(wl, _particles(wl, counts, u_th, 500), precision, BIG, 3)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("total", [1, 31, 257, 1663, 1664, 1665, 2047, 2049, 2176, 2177, 2433, 4353])
def test_item_sizes(dims, total, precision):
    """One tile holding `total` particles."""
    n = (8, 8, 4) if dims == 3 else (16, 16)
    wl = synth.small(dims, n, 2, 1, 0.1, 73)
    counts = np.full(wl.ncells, total // wl.ncells)
    counts[: total % wl.ncells] += 1
    _compare(wl, _particles(wl, counts, 0.1, 900), precision, BIG, 2)

"""Work items of the push at their largest size (needs a GB300): ranks, the
task list, the staging copies and the window at full load.

The sort cuts every tile's run into pieces of one of thirty sizes, whichever
its estimate of the push's time (item_cost, restated here) finds least.  As
many tiles are filled as make exactly one round of items of the largest size:
runs four, three and one slot short of it, at it, and one and four beyond it,
spread over their tiles' cells or crowded into one cell.  Fields, J and
momenta match the oracle, in FP64 to 1e-12 per step and in FP32 to the path's
1e-5.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1503_02464_gb300 import synth
from paper_1503_02464_gb300.sim import Simulation

from _parity import compare_fields, compare_particles, j_floor, j_floor_fp32

pytestmark = pytest.mark.gpu

# (dims, order, precision): slots an item may hold, blocks per SM, an item's own cost in slots
LAYOUT = {(3, 2, "fp32"): (2176, 2, 400), (3, 1, "fp32"): (1216, 3, 400), (2, 2, "fp32"): (1920, 3, 400),
          (2, 1, "fp32"): (1920, 3, 400), (3, 2, "fp64"): (2432, 1, 120), (2, 2, "fp64"): (1664, 2, 120)}


def _sizes(cap, dims, precision):
    c = [int(cap * 2.0 ** (-j / 8.0)) // 4 * 4 for j in range(30)]
    return [max(v, 512) for v in c] if dims == 2 and precision == "fp32" else c


def _items(run, size):
    if run <= size:
        return int(run > 0)
    pieces = -(-run // size)
    piece = -(-(-(-run // pieces)) // 4) * 4
    return -(-run // piece)


def _cost(blocks, nsm, fixed, slots, items):
    per = blocks * nsm
    full, rem = items // per, items % per
    most = -(-rem // nsm) * nsm
    unit = items
    if full == 0:
        unit = (per + most) // 2
    elif rem > 0:
        unit += per - rem if blocks == 1 else 2 * per // (5 * full * full) + (most - rem) // 2
    return unit * (slots // items + fixed)


@pytest.mark.parametrize("dims,order,precision", sorted(LAYOUT))
def test_items_of_the_largest_size(dims, order, precision):
    cap, blocks, fixed = LAYOUT[dims, order, precision]
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    tile = (8, 8, 4) if dims == 3 else (16, 16, 1)
    beyond = blocks * nsm // 8  # runs that make two items
    ntile = blocks * nsm - beyond
    totals = np.where(np.arange(ntile) < beyond, cap + 1 + 3 * (np.arange(ntile) % 2),
                      cap - np.array([0, 4, 3, 1])[np.arange(ntile) % 4])
    runs = (totals + 3) // 4 * 4
    costs = [_cost(blocks, nsm, fixed, int(runs.sum()), sum(_items(int(r), size) for r in runs))
             for size in _sizes(cap, dims, precision)]
    assert costs[0] < min(costs[1:])

    nt = (8, 8, -(-ntile // 64)) if dims == 3 else (16, -(-ntile // 16), 1)
    wl = synth.small(dims, tuple(a * b for a, b in zip(nt, tile))[:dims], order, 1, 0.1, 23)
    rng = np.random.default_rng(29)
    cells = []
    for t in rng.permutation(nt[0] * nt[1] * nt[2])[:ntile]:
        k = len(cells)
        inside = np.arange(totals[k]) % (tile[0] * tile[1] * tile[2])
        if k % 16 == 5:
            inside[:] = rng.integers(tile[0] * tile[1] * tile[2])  # all of them in one cell
        first = np.array([t % nt[0], t // nt[0] % nt[1], t // (nt[0] * nt[1])]) * tile
        cells.append(first + np.stack([inside % tile[0], inside // tile[0] % tile[1], inside // (tile[0] * tile[1])], -1))
    cells = np.concatenate(cells)
    n = len(cells)
    x = (cells + rng.random((n, 3))) * wl.d
    u = rng.normal(0, 0.1, (n, 3))
    p = {"x": x[:, 0], "y": x[:, 1], "z": x[:, 2] if dims == 3 else np.zeros(n), "ux": u[:, 0], "uy": u[:, 1],
         "uz": u[:, 2], "w": rng.uniform(0.01, 0.02, n), "id": np.arange(n, dtype=np.uint32)}

    o = oracle.OracleSim(wl.dims, wl.n, wl.d, wl.dt, wl.order, parallel=True)
    o.add_particles(p, -1.0, 1.0)
    s = Simulation.from_workload(wl, precision=precision, sort_every=1000)
    s.load(s.add_species(-1.0, 1.0, n), p)
    o.step(2)
    s.step(2)
    floor = j_floor(wl, [p]) + (j_floor_fp32(wl, [p]) if precision == "fp32" else 0.0)
    fe = compare_fields(o, s, j_abs=floor)
    du, dx = compare_particles(o, s, wl)
    s.close()
    print(dims, order, precision, fe, du, dx)
    tol = 2e-12 if precision == "fp64" else 1e-5
    assert max(fe.values()) <= tol and du <= tol, (fe, du)
    assert dx <= (1e-10 if precision == "fp64" else 1e-6)

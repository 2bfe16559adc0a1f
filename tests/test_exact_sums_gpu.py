"""The FP32 current sums lose nothing but the window's quantum (needs a GB300).

Every tile holds three particles at one place with one momentum, of weights
W, 1 and -W in some order: their currents are those of the light one alone.
A contribution p q enters the sums as rint(p q 2^K) or finer, with 2^K above
2^36 / Q for the tile's bound Q = 1.01 (2 W + 1) |v|_1 on the sum (3D, cubic
cells: on |J|; other components have at most twice the quantum), so a node's
three contributions are off by at most 1.5 Q 2^-36, twice that in those, and the
sum by the rounding of the stored current.  FP32 sums of the same terms would
be off by 2^-25 W |v| times a shape weight, two hundred times the bound.
"""
import numpy as np
import pytest

from paper_1503_02464_gb300 import synth
from paper_1503_02464_gb300.sim import Simulation

pytestmark = pytest.mark.gpu

W = 1e5


def _opposite_weights(dims, n, d, dt, tile, order, largest_quantum):
    rng = np.random.default_rng(3)
    n3, d3 = tuple(n) + (1,) * (3 - len(n)), tuple(d) + (1.0,) * (3 - len(d))
    first = np.stack(np.meshgrid(*[np.arange(0, n3[a], tile[a]) for a in range(3)], indexing="ij"), -1).reshape(-1, 3)
    nt = len(first)
    # in the middle of the tile, 0.1 to 0.4 of a cell above its lower node, and
    # moves of at most 0.05 cells: the nearest node and the cell stay
    cell = first + [tile[0] // 2, tile[1] // 2, tile[2] // 2]
    x = (cell + rng.uniform(0.1, 0.4, (nt, 3))) * d3
    if dims == 2:
        x[:, 2] = 0.0
    u = rng.uniform(0.02, 0.05, (nt, 3)) * rng.choice([-1.0, 1.0], (nt, 3))
    w = rng.permuted(np.tile([W, 1.0, -W], (nt, 1)), axis=1).reshape(-1)
    p = {"x": x[:, 0], "y": x[:, 1], "z": x[:, 2], "ux": u[:, 0], "uy": u[:, 1], "uz": u[:, 2]}
    p = {k: np.repeat(v, 3) for k, v in p.items()}
    p["id"] = np.arange(3 * nt, dtype=np.uint32)
    J = []
    for weights in (w, np.where(w == 1.0, 1.0, 0.0)):
        s = Simulation(dims, n, d, dt, order, "fp32")
        k = s.add_species(-1.0, 1.0, 3 * nt)
        s.load(k, dict(p, w=weights))
        s.step(1)
        J.append(np.stack([s.field(c) for c in (6, 7, 8)]))
        s.close()
    v1 = (np.abs(u).sum(1) / np.sqrt(1.0 + (u * u).sum(1))).max()
    quantum = largest_quantum * 1.01 * (2 * W + 1) * v1 * 2.0 ** -36
    for c in range(3):
        largest = np.abs(J[1][c]).max()
        tol = 1.5 * quantum + 2.0 ** -23 * largest
        assert tol < 1e-3 * largest
        err = np.abs(J[0][c] - J[1][c]).max()
        print(dims, order, c, err, tol, largest)
        assert err <= tol, (c, err, tol)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("dims,n,tile", [(3, (64, 32, 16), (8, 8, 4)), (2, (128, 64), (16, 16, 1))])
def test_opposite_weights_cancel(dims, n, tile, order):
    d = (0.05,) * dims
    _opposite_weights(dims, n, d, 0.95 * synth.courant_limit(d, dims), tile, order, 1.0 if dims == 3 else 2.0)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("dims,n,d,dt,tile", [(3, (64, 32, 16), (0.05, 0.05, 5.0), 0.03, (8, 8, 4)),
                                              (3, (64, 32, 16), (5.0, 0.05, 0.5), 0.04, (8, 8, 4)),
                                              (2, (128, 64), (0.05, 2.5), 0.04, (16, 16, 1)),
                                              (2, (128, 64), (0.05, 0.05), 0.0005, (16, 16, 1))])
def test_in_flat_cells_and_small_steps(dims, n, d, dt, tile, order):
    """Components whose dt / dx is far below the largest lose nothing by it."""
    _opposite_weights(dims, n, d, dt, tile, order, 2.0)

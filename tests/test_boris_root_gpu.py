"""The FP32 push's rotation against 64 bits (needs a GB300).

3D FP32 runs take 1 / gamma and 1 / (1 + t^2) from the hardware's
approximations and one Newton step each, in place of the IEEE root and
quotients.  In a uniform B and no E, the new momenta are compared with the
Boris rotation of the stored FP32 ones in FP64.

Bound, with e = 2^-24 (a rounding to nearest is off by at most e): the field
weights sum to 1 within 9 e, the root is within 2 e and the quotient within
1.5 e, so t = h B / gamma and s = 2 t / (1 + t^2) are off by at most 16 e and
32 e of themselves (|ds| <= 2 |dt|, products and sums included).  A rotation by
2 atan |t| moves the momentum by at most |t| |ds| + |s| |dt| <= 64 e |t|, and
its own products and sums round six more times: (64 |t| + 8) e of |u|.
"""
import numpy as np
import pytest

from paper_1503_02464_gb300 import synth
from paper_1503_02464_gb300.sim import Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("u_th", [0.01, 0.5, 10.0])
@pytest.mark.parametrize("b", [0.1, 3.0, 30.0])
def test_rotation(u_th, b, order):
    wl = synth.small(3, (24, 16, 12), order, 6, u_th, 31)
    p = wl.particles(0)
    s = Simulation.from_workload(wl, precision="fp32")
    s.load(s.add_species(-1.0, 1.0, len(p["x"])), p)
    B = np.array([0.25, -0.5, 1.0]) * b
    for c in range(3):
        s.set_field(3 + c, B[c])
    before = s.particles(0)
    s.step(1)
    after = s.particles(0)
    s.close()
    i0, i1 = np.argsort(before["id"]), np.argsort(after["id"])
    u0 = np.stack([before[k][i0] for k in ("ux", "uy", "uz")], -1)
    u1 = np.stack([after[k][i1] for k in ("ux", "uy", "uz")], -1)
    h = -0.5 * wl.dt
    t = h * np.float32(B).astype(np.float64) / np.sqrt(1.0 + (u0 * u0).sum(1))[:, None]
    sv = 2.0 * t / (1.0 + (t * t).sum(1))[:, None]
    want = u0 + np.cross(u0 + np.cross(u0, t), sv)
    err = np.sqrt(((u1 - want) ** 2).sum(1)) / np.sqrt((u0 * u0).sum(1))
    tol = (64 * np.sqrt((t * t).sum(1)) + 8) * 2.0 ** -24
    print(u_th, b, order, (err / tol).max(), err.max() * 2 ** 24)
    assert (err <= tol).all()

"""The tape entries' copies at sizes whose field and particle blocks leave
remainders of the copy's passes (needs a GB300): FP64 gradients of runs with
every step recorded against central differences, at the bound of the adjoint
tests (1e-6), and FP32 gradients against the FP64 ones at theirs (1e-4).
"""
import dataclasses
import math

import numpy as np
import pytest

from paper_1503_02464_gb300 import diff

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, ny, ppc", [(40, 8, 2), (41, 9, 2), (43, 7, 3), (40, 131, 9)])
def test_gradients_from_recorded_steps(nx, ny, ppc):
    run = diff.SlabRun(nx=nx, ny=ny, ppc=ppc, steps=30, segment=10, slab=(8, 30), density=1.0, obj=(12, 20),
                       waist=1.5, duration=2 * math.pi, seed=7, precision="fp64", store_all=True)
    prof = run.default_profile()
    prof[8:30] = 1.0 + 0.3 * np.sin(np.arange(22) * 0.7)
    grads = {}
    for precision in ("fp64", "fp32"):
        F, sim = diff.forward_objective(dataclasses.replace(run, precision=precision), 0.8, prof, keep=True)
        grads[precision] = diff.backward_gradients(dataclasses.replace(run, precision=precision), sim)
        sim.close()
    h = 1e-6
    fd = (diff.forward_objective(run, 0.8 + h, prof)[0] - diff.forward_objective(run, 0.8 - h, prof)[0]) / (2 * h)
    assert abs(grads["fp64"][0] - fd) <= 1e-6 * abs(fd), (grads["fp64"][0], fd)
    assert abs(grads["fp32"][0] - grads["fp64"][0]) <= 1e-4 * abs(grads["fp64"][0])
    assert np.abs(grads["fp32"][1] - grads["fp64"][1]).max() <= 1e-4 * np.abs(grads["fp64"][1]).max()

"""Particle counts on both sides of the lines where the kernels change form: the radix
sort's chunks (65,536), the lanes per cell of P2G in single precision (58,368 in 3D and
311,296 in 2D on 152 SMs) and P2G in double precision, from random positions (cells with
no, one and many particles) against the FP64 oracle; every field read back.

Bounds as in the parity tests: FP64 1e-9, FP32 1e-4 of the largest value.
"""
import numpy as np
import pytest

import oracle
from paper_2507_04192_gb300 import inputs, mpm

pytestmark = pytest.mark.gpu


def scattered(dim, n, material, seed):
    cells = (128, 128) if dim == 2 else (24, 24, 24)
    dx = 1.0 / 32
    rng = np.random.default_rng(seed)
    hi = np.array(cells) * dx
    x = (0.1 + 0.8 * rng.random((n, dim))) * hi
    v = 0.5 * np.stack([np.sin(2.0 * x[:, a - 1] + a) for a in range(dim)], 1)
    return inputs.Workload(name="scattered", dim=dim, n_cells=cells, dx=dx, dt=2e-5, gravity=(0.0,) * (dim - 1) + (-9.81,),
                           material=dict(material), x=x, particle_volume=dx ** dim * 0.64 * np.prod(cells) / n, steps=3,
                           sort_every=2, v=v)


@pytest.mark.parametrize("dim,n,material,precision,tol", [
    (2, 65536, inputs.FLUID_WATER, mpm.MPM_FP32, 1e-4), (2, 65537, inputs.SAND_DP, mpm.MPM_FP32, 1e-4),
    (2, 311296, inputs.FLUID_WATER, mpm.MPM_FP32, 1e-4), (2, 311329, inputs.FLUID_WATER, mpm.MPM_FP32, 1e-4),
    (3, 58368, inputs.SAND_DP, mpm.MPM_FP32, 1e-4), (3, 58399, inputs.SAND_DP, mpm.MPM_FP32, 1e-4),
    (3, 58401, inputs.FLUID_WATER, mpm.MPM_FP32, 1e-4),
    (2, 5001, inputs.SAND_DP, mpm.MPM_FP64, 1e-9), (3, 4999, inputs.FLUID_WATER, mpm.MPM_FP64, 1e-9),
    (3, 30001, inputs.SAND_DP, mpm.MPM_FP64, 1e-9)])
def test_counts_around_the_lines(dim, n, material, precision, tol):
    w = scattered(dim, n, material, n)
    orc = oracle.Oracle.from_workload(w)
    st = orc.initial_state(w.x, w.v)
    orc.step(st, w.steps)
    sim = mpm.Simulation.from_workload(w, precision)
    sim.step(w.steps)
    for f, ref in (("x", st.x), ("v", st.v), ("C", st.B * (4.0 / w.dx ** 2)), ("F", st.F), ("rho", st.rho)):
        got = sim.get(f).reshape(np.shape(ref))
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), f
    sim.close()

"""G2P's work items (runs of a tile's particles) at the edges of their cut: counts
around a particle block (32), a block's round (256) and several runs of one
tile, alone in the domain or after another tile's particles, against the FP64
oracle.  A particle that a run missed keeps its old state, far outside the
bounds (FP64 1e-9, FP32 1e-4 of the largest value, as in the parity tests).
"""
import numpy as np
import pytest

import oracle
from paper_2507_04192_gb300 import inputs, mpm

pytestmark = pytest.mark.gpu


def clustered(dim, counts, material, seed=5):
    """counts[i] particles at random in the cells of tile i along x, smooth velocities."""
    T = 16 if dim == 2 else 8
    cells = (3 * T,) + (T,) * (dim - 1)
    dx = 1.0 / 32
    rng = np.random.default_rng(seed)
    x = np.concatenate([(rng.uniform(1.0, T - 2.0, (c, dim)) + np.eye(dim)[0] * T * i) * dx
                        for i, c in enumerate(counts)])
    v = np.stack([np.sin(3.0 * x[:, a - 1] + a) for a in range(dim)], 1)
    return inputs.Workload(name="clustered", dim=dim, n_cells=cells, dx=dx, dt=1e-4,
                           gravity=(0.0,) * (dim - 1) + (-9.81,), material=dict(material), x=x,
                           particle_volume=dx ** dim / 8, steps=2, sort_every=8, v=v)


@pytest.mark.parametrize("dim,material", [(2, inputs.FLUID_WATER), (3, inputs.FLUID_WATER), (3, inputs.SAND_DP)])
@pytest.mark.parametrize("counts", [(1,), (31,), (33,), (257,), (1, 32), (5, 255), (17, 513, 31), (2049, 63)])
@pytest.mark.parametrize("precision,tol", [(mpm.MPM_FP64, 1e-9), (mpm.MPM_FP32, 1e-4)])
def test_every_particle_of_every_run_is_updated(dim, material, counts, precision, tol):
    w = clustered(dim, counts, material)
    orc = oracle.Oracle.from_workload(w)
    st = orc.initial_state(w.x, w.v)
    orc.step(st, w.steps)
    sim = mpm.Simulation.from_workload(w, precision)
    sim.step(w.steps)
    for f, ref in (("x", st.x), ("v", st.v), ("F", st.F), ("rho", st.rho)):
        got = sim.get(f).reshape(np.shape(ref))
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), f
    sim.close()

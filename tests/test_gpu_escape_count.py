"""The escape counter in double precision: every P2G pass adds the cells (of the last sort)
with a particle whose stencil lies outside the window of the cell's tile.  The expected
count comes from the oracle's positions; particles that left their cells but no window
count nothing.  The single-precision counter counts threads that met a particle outside its
cell: zero before any moved, positive after.
"""
import numpy as np
import pytest

import oracle
from paper_2507_04192_gb300 import inputs, mpm

pytestmark = pytest.mark.gpu


def block(dim, speed):
    """A block of water far from the walls, moving by about a cell per 1 / speed steps."""
    if dim == 2:
        w = inputs.dam_break_2d(64, 0.2, 0.2)
        w.x = w.x + 0.3
    else:
        cells, dx = (32, 32, 32), 1.0 / 32
        x = inputs.lattice_particles(cells, dx, 2, lambda p: (np.abs(p - 0.45) < 0.14).all(1), (0.0,) * 3, (1.0,) * 3, 0)
        w = inputs.Workload(name="block", dim=3, n_cells=cells, dx=dx, dt=1e-4, gravity=(0.0, 0.0, -9.81),
                            material=dict(inputs.FLUID_WATER), x=x, particle_volume=dx ** 3 / 8, steps=32, sort_every=64)
    w.v = np.tile(np.array([speed, 0.4 * speed, -0.5 * speed][:dim]) * w.dx / w.dt, (w.n, 1))
    return w


def places(x, w):
    """Sort coordinates (base cell + 1) per axis."""
    return np.clip(np.floor(x / w.dx - 0.5).astype(int), -1, np.array(w.n_cells[:w.dim]) - 1) + 1


def expected(w, steps):
    T = 16 if w.dim == 2 else 8
    orc = oracle.Oracle.from_workload(w)
    st = orc.initial_state(w.x, w.v)
    home = places(w.x, w)
    cell = np.ravel_multi_index(home.T, [c + 1 for c in w.n_cells[:w.dim]])
    total, moved = 0, False
    for _ in range(steps):
        s = places(st.x, w)
        l = s + 1 - home // T * T                    # window coordinate of the stencil's first node
        total += len(np.unique(cell[((l < 0) | (l > T + 1)).any(1)]))
        moved = moved or bool((s != home).any())
        orc.step(st, 1)
    return total, moved


def counted(w, precision, steps):
    sim = mpm.Simulation.from_workload(w, precision, sort_every=64)
    sim.step(steps)
    n = sim.stats()["escaped"]
    sim.close()
    return n


@pytest.mark.parametrize("dim", [2, 3])
def test_fp64_counts_cells_with_a_particle_outside_the_tile_window(dim):
    w = block(dim, 0.1)
    want, _ = expected(w, 24)                        # 2.4 cells
    assert want > 0
    assert counted(w, mpm.MPM_FP64, 24) == want


@pytest.mark.parametrize("dim", [2, 3])
def test_fp64_counts_nothing_inside_the_window(dim):
    w = block(dim, 0.02)
    want, moved = expected(w, 24)                    # half a cell
    assert want == 0 and moved
    assert counted(w, mpm.MPM_FP64, 24) == 0
    assert counted(w, mpm.MPM_FP32, 24) > 0
    assert counted(w, mpm.MPM_FP32, 1) == 0

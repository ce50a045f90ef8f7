"""Around the count where the single-precision P2G goes from several lanes per cell to one
(4 x 4 x 128 particles per SM in 2D, 3 x 128 in 3D: on the line, one above it), every
particle field against the FP64 oracle; and above the line a batch of 2D simulations with a
friction field each, whose particles leave their cells between sorts.

Bounds as in the parity tests: positions, velocities, affine matrix, deformation gradient
and density 1e-4 of the largest value, stress 1e-3 of the sand's largest (1e-4 and 1e-6 of
the bulk modulus for water, whose pressure amplifies the density's rounding), plastic
strain 2e-2.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_04192_gb300 import inputs, mpm

pytestmark = pytest.mark.gpu


def line(dim):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sms * 128 * (3 if dim == 3 else 16)


def scattered(dim, n, material):
    cells = (128, 128) if dim == 2 else (24, 24, 24)
    dx = 1.0 / 32
    rng = np.random.default_rng(n)
    hi = np.array(cells) * dx
    x = (0.1 + 0.8 * rng.random((n, dim))) * hi
    v = 0.5 * np.stack([np.sin(2.0 * x[:, a - 1] + a) for a in range(dim)], 1)
    return inputs.Workload(name="scattered", dim=dim, n_cells=cells, dx=dx, dt=2e-5,
                           gravity=(0.0,) * (dim - 1) + (-9.81,), material=dict(material), x=x, v=v,
                           particle_volume=dx ** dim * 0.64 * np.prod(cells) / n, steps=3, sort_every=2)


@pytest.mark.parametrize("dim,material", [(2, inputs.FLUID_WATER), (2, inputs.SAND_DP), (3, inputs.FLUID_WATER),
                                          (3, inputs.SAND_DP)])
@pytest.mark.parametrize("above", [0, 1])
def test_every_field_on_both_sides_of_the_line(dim, material, above):
    w = scattered(dim, line(dim) + above, material)
    orc = oracle.Oracle.from_workload(w)
    st = orc.initial_state(w.x, w.v)
    orc.step(st, w.steps)
    sim = mpm.Simulation.from_workload(w, mpm.MPM_FP32)
    sim.step(w.steps)
    sand = material["kind"] == 1
    bounds = {"x": 1e-4, "v": 1e-4, "C": 1e-4, "F": 1e-4, "rho": 1e-4, "sigma": 1e-3 if sand else 1e-4, "eps": 2e-2}
    for f, ref in (("x", st.x), ("v", st.v), ("C", orc.affine_C(st)), ("F", st.F), ("rho", st.rho),
                   ("sigma", st.sigma), ("eps", st.eps)):
        got = sim.get(f).reshape(np.shape(ref))
        slack = 1e-6 * material["bulk_K"] if f == "sigma" and not sand else 0.0
        assert np.abs(got - ref).max() <= bounds[f] * np.abs(ref).max() + slack, f
    sim.close()


def test_batched_2d_with_escapes_above_the_line():
    steps, per = 32, 18432
    B = line(2) // per + 2
    mus = [inputs.friction_field(32, s) for s in range(B)]

    def workload(mu):
        w = inputs.dam_break_inverse_2d(96, n_seg=32, steps=steps)
        w.friction = [(2, (32, 1), mu)]
        w.v = np.tile([4.0, -0.5], (w.n, 1))        # 1.2 cells before the next sort
        return w
    w = workload(mus[0])
    assert w.n == per and B * per > line(2)
    sim = mpm.Simulation(2, w.n_cells, w.dx, w.dt, w.gravity, w.material, mpm.MPM_FP32, steps, batch=B)
    sim.load(np.concatenate([w.x] * B), np.concatenate([w.v] * B), w.particle_volume,
             np.repeat(np.arange(B, dtype=np.int32), per))
    sim.set_friction(2, (32, 1), np.concatenate(mus))
    sim.step(steps)
    assert sim.stats()["escaped"] > 0
    x, v = sim.get("x").reshape(B, per, 2), sim.get("v").reshape(B, per, 2)
    sim.close()
    for b in (0, B // 2, B - 1):
        wb = workload(mus[b])
        orc = oracle.Oracle.from_workload(wb)
        st = orc.initial_state(wb.x, wb.v)
        orc.step(st, steps)
        assert np.abs(x[b] - st.x).max() <= 1e-4
        assert np.abs(v[b] - st.v).max() <= 2e-3 * np.abs(st.v).max()

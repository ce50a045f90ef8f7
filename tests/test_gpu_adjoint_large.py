"""The 3D sand adjoint of a problem large enough for the forms that small ones never
reach: one lane per cell in the forward P2G, its copy of the inputs and the v_bar
scatter of single precision, and several rounds of the reverse particle kernels'
persistent blocks (138,432 particles on 152 SMs: two rounds in single, four in double
precision).  Sorts and a checkpoint lie inside the horizon.  Against the FP64 oracle's
reverse recursion.

Bounds as in the tests of the small problems: FP64 1e-6 of the largest value, FP32 1e-3
in norm on a short horizon.  The sand starts moving (converging, sliding, downwards),
away from the apex of the yield cone and from the stick/slide threshold.
"""
import numpy as np
import pytest

import oracle
from paper_2507_04192_gb300 import inputs, mpm

pytestmark = pytest.mark.gpu

STEPS, OBS = 5, (3, 5)


@pytest.fixture(scope="module")
def problem():
    w = inputs.granular_inverse_3d((56, 56, 40), 14, 28, patches=(4, 4), n_track=64, n_obs=2, dt=4e-5, dx=1 / 64)
    cx, cy = w.extras["axis"]
    v0 = np.stack([0.4 - 2.0 * (w.x[:, 0] - cx), -2.0 * (w.x[:, 1] - cy), np.full(w.n, -0.2)], 1)
    ids = w.extras["track_ids"]
    orc = oracle.Oracle.from_workload(w)
    states = [orc.initial_state(w.x, v0)]
    for _ in range(STEPS):
        states.append(states[-1].copy())
        orc.step(states[-1], 1)
    z = np.stack([states[s].x[ids] + 2e-3 for s in OBS])
    lam = [np.zeros((w.n, 3)), np.zeros((w.n, 3)), np.zeros((w.n, 3, 3)), np.zeros(w.n), np.zeros((w.n, 3, 3))]
    loss, grad = 0.0, np.zeros(16)
    for t in range(STEPS, 0, -1):
        if t in OBS:
            e = states[t].x[ids] - z[OBS.index(t)]
            loss += float((e * e).sum())
            lam[0][ids] += 2.0 * e
        lam, mub = orc.step_vjp(states[t - 1], *lam)
        grad += mub[4]
    return w, v0, z, loss, grad, lam[1]


@pytest.mark.parametrize("precision", [mpm.MPM_FP32, mpm.MPM_FP64])
def test_large_sand_adjoint_matches_the_oracle(problem, precision):
    w, v0, z, ref_loss, ref_grad, ref_v = problem
    assert w.n > 100_000 and np.abs(ref_grad).max() > 0
    sim = mpm.Simulation(3, w.n_cells, w.dx, w.dt, w.gravity, w.material, precision, 2)
    sim.load(w.x, v0, w.particle_volume)
    sim.set_friction(4, (4, 4), w.extras["mu_true"])
    mpm.mpm_set_observations(sim.ctx, w.extras["track_ids"], OBS, z)
    loss, grad = mpm.mpm_step_adjoint(sim.ctx, STEPS, 3, 4, 16)
    dv0 = mpm.mpm_get_initial_adjoint(sim.ctx, "v")
    sim.close()
    if precision == mpm.MPM_FP64:
        assert loss == pytest.approx(ref_loss, rel=1e-9)
        np.testing.assert_allclose(grad, ref_grad, rtol=0, atol=1e-6 * np.abs(ref_grad).max())
        np.testing.assert_allclose(dv0, ref_v, rtol=0, atol=1e-6 * np.abs(ref_v).max())
    else:
        assert loss == pytest.approx(ref_loss, rel=1e-3)
        assert np.linalg.norm(grad - ref_grad) <= 1e-3 * np.linalg.norm(ref_grad)
        assert np.linalg.norm(dv0 - ref_v) <= 1e-3 * np.linalg.norm(ref_v)

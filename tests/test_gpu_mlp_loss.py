"""The loss of a training step is the mean of (y - t)^2 over all outputs, whatever the
number of blocks that add it up: against the outputs of an inference on the same
parameters, differences in single precision as the kernel takes them, the sum in double
(rounding of a few hundred thousand additions: 1e-12 relative)."""
import numpy as np
import pytest

from paper_2507_04192_gb300 import mpm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_out,batch", [(8, 8), (40, 72), (32, 264), (1032, 8), (1024, 264)])
@pytest.mark.parametrize("out", [mpm.MPM_OUT_SIGMOID, mpm.MPM_OUT_LINEAR])
def test_loss_is_the_mean_over_all_outputs(n_out, batch, out):
    rng = np.random.default_rng(n_out + batch)
    net = mpm.MLP([24, n_out], batch, output=out)
    net.set_params((0.3 * rng.standard_normal(net.num_params)).astype(np.float32))
    x = rng.standard_normal((batch, 24)).astype(np.float32)
    t = rng.uniform(0.1, 0.6, (batch, n_out)).astype(np.float32)
    y = net.infer(x)
    loss = net.train_step(x, t, lr=0.0, update=False)
    net.close()
    e = (y - t).astype(np.float64)
    assert loss == pytest.approx((e * e).mean(), rel=1e-12)

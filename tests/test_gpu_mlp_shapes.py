"""The tile widths of the tensor-core GEMM (32, 64, 128 columns by the number of tiles)
at ragged sizes and an output that is not 16-byte aligned, and a training step of
networks whose layers end inside a tile.

Bounds as in the tests of the GEMM and the network: |C - A B^T| <= 2e-5 |A| |B|^T
elementwise, gradients within 2e-2 relative L2 per layer; Adam's first step from the
returned gradient within 2e-6.
"""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2507_04192_gb300 import mpm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(129, 33, 8), (257, 250, 264), (1280, 632, 200), (1300, 600, 72), (2560, 640, 136),
                                   # 256 columns, the last wave in two and in four parts (152 SMs)
                                   (6390, 1000, 136), (4990, 1016, 72)])
@pytest.mark.parametrize("shift", [0, 1])
def test_gemm_tile_widths(M, N, K, shift):
    g = torch.Generator().manual_seed(M + N)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, generator=g).to(torch.bfloat16)
    dA, dB = A.cuda(), B.cuda()
    buf = torch.full((M * N + 2,), float("nan"), device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    mpm.mpm_gemm_bf16(M, N, K, dA.data_ptr(), K, dB.data_ptr(), K, buf.data_ptr() + 4 * shift, N, st.data_ptr(),
                      torch.cuda.current_stream().cuda_stream)
    out = buf.cpu().double().numpy()
    assert int(st.item()) == 0
    a, b = A.double().numpy(), B.double().numpy()
    C = out[shift:shift + M * N].reshape(M, N)
    assert (np.abs(C - a @ b.T) <= 2e-5 * (np.abs(a) @ np.abs(b).T) + 1e-30).all()
    assert np.isnan(out[:shift]).all() and np.isnan(out[shift + M * N:]).all()


@pytest.mark.parametrize("widths,batch", [([8, 8], 8), ([8, 8, 8], 8), ([40, 264, 72, 8], 136), ([136, 40, 520, 16], 264)])
@pytest.mark.parametrize("hidden,out", [("gelu", "sigmoid"), ("relu", "linear")])
def test_training_step_of_ragged_networks(widths, batch, hidden, out):
    rng = np.random.default_rng(batch)
    p = omlp.pack([(rng.standard_normal((n, k)) / np.sqrt(k), 0.1 * rng.standard_normal(n))
                   for k, n in zip(widths, widths[1:])]).astype(np.float32)
    x = rng.standard_normal((batch, widths[0])).astype(np.float32)
    t = rng.uniform(0.1, 0.6, (batch, widths[-1])).astype(np.float32)
    net = mpm.MLP(widths, batch, hidden=mpm.MPM_ACT_RELU if hidden == "relu" else mpm.MPM_ACT_GELU,
                  output=mpm.MPM_OUT_LINEAR if out == "linear" else mpm.MPM_OUT_SIGMOID)
    net.set_params(p)
    loss = net.train_step(x, t, lr=1e-3, update=True)
    g, p1 = net.get_params(1).astype(np.float64), net.get_params(0).astype(np.float64)
    net.close()
    rl, rg = omlp.loss_and_grad(p.astype(np.float64), widths, x.astype(np.float64), t.astype(np.float64),
                                hidden=hidden, out=out)
    assert loss == pytest.approx(rl, rel=1e-2)
    o = 0
    for k, n in zip(widths, widths[1:]):
        for m in (n * k, n):
            assert np.linalg.norm(g[o:o + m] - rg[o:o + m]) <= 2e-2 * np.linalg.norm(rg[o:o + m])
            o += m
    np.testing.assert_allclose(p1, p - 1e-3 * g / (np.abs(g) + 1e-8), rtol=0, atol=2e-6)

"""The tensor-core GEMM where its tiles begin to outnumber the SMs: outputs of at most 32
columns take rings of 4 stages (two CTAs per SM) from there on, and the backward products
of a network whose 128 x 256 tiles fill the chip take the persistent kernel.

Values: |C - A B^T| <= 2e-5 |A| |B|^T elementwise, gradients within 2e-2 relative L2 per
layer, as in the other tests of GEMM and network.  Time: one tile more than SMs must not
cost a second wave of tiles (the ratio is 1.6 when it does, 1.0 when it does not).
"""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2507_04192_gb300 import mpm

pytestmark = pytest.mark.gpu


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def operands(M, N, K, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16),
            torch.randn(N, K, generator=g, device="cuda").to(torch.bfloat16))


def gemm(a, b, c_ptr, status):
    (M, K), N = a.shape, b.shape[0]
    mpm.mpm_gemm_bf16(M, N, K, a.data_ptr(), K, b.data_ptr(), K, c_ptr, N, status.data_ptr(),
                      torch.cuda.current_stream().cuda_stream)


def median_us(fn, calls=20, reps=7):
    for _ in range(3):
        fn()
    out = []
    for _ in range(reps):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        torch.cuda._sleep(1_000_000)                 # the calls queue up behind it
        start.record()
        for _ in range(calls):
            fn()
        end.record()
        torch.cuda.synchronize()
        out.append(start.elapsed_time(end) * 1000.0 / calls)
    return float(np.median(out))


@pytest.mark.parametrize("tiles,ragged,N,K", [(0, 0, 24, 72), (0, 1, 24, 72), (1, 0, 8, 8), (1, -5, 32, 640),
                                              (160, 37, 17, 264)])
@pytest.mark.parametrize("shift", [0, 1])
def test_narrow_outputs_in_more_tiles_than_sms(tiles, ragged, N, K, shift):
    M = 128 * (sms() + tiles) + ragged
    a, b = operands(M, N, K, seed=M)
    buf = torch.full((M * N + 2,), float("nan"), device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    gemm(a, b, buf.data_ptr() + 4 * shift, st)
    assert int(st.item()) == 0
    C = buf[shift:shift + M * N].reshape(M, N).double()
    ad, bd = a.double(), b.double()
    assert ((C - ad @ bd.T).abs() <= 2e-5 * (ad.abs() @ bd.abs().T) + 1e-30).all()
    assert torch.isnan(buf[:shift]).all() and torch.isnan(buf[shift + M * N:]).all()


def test_one_tile_more_than_sms_is_no_second_wave():
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    times = []
    for tiles in (sms(), sms() + 1):
        a, b = operands(128 * tiles, 24, 640)
        c = torch.empty(128 * tiles, 24, device="cuda")
        times.append(median_us(lambda: gemm(a, b, c.data_ptr(), st)))
    assert times[1] <= 1.3 * times[0], times


def tiles(M, N):
    return -(-M // 128) * -(-N // 256)


@pytest.mark.parametrize("widths,batch,wide", [([40, 2312, 40], 2056, (2056, 2312)),     # dA of layer 1
                                               ([2056, 2312, 8], 264, (2312, 2056))])    # dW of layer 0
@pytest.mark.parametrize("hidden", ["gelu", "relu"])
def test_wide_backward_products(widths, batch, wide, hidden):
    assert tiles(*wide) >= sms()
    rng = np.random.default_rng(batch)
    p = omlp.pack([(rng.standard_normal((n, k)) / np.sqrt(k), 0.1 * rng.standard_normal(n))
                   for k, n in zip(widths, widths[1:])]).astype(np.float32)
    x = rng.standard_normal((batch, widths[0])).astype(np.float32)
    t = rng.uniform(0.1, 0.6, (batch, widths[-1])).astype(np.float32)
    net = mpm.MLP(widths, batch, hidden=mpm.MPM_ACT_RELU if hidden == "relu" else mpm.MPM_ACT_GELU)
    net.set_params(p)
    loss = net.train_step(x, t, lr=1e-3, update=False)
    g = net.get_params(1).astype(np.float64)
    net.close()
    rl, rg = omlp.loss_and_grad(p.astype(np.float64), widths, x.astype(np.float64), t.astype(np.float64), hidden=hidden)
    assert loss == pytest.approx(rl, rel=1e-2)
    o = 0
    for k, n in zip(widths, widths[1:]):
        for m in (n * k, n):
            assert np.linalg.norm(g[o:o + m] - rg[o:o + m]) <= 2e-2 * np.linalg.norm(rg[o:o + m])
            o += m

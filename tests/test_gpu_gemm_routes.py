"""The tensor-core GEMM where its tiles begin to outnumber the SMs: outputs of at most 32
columns take rings of 4 stages (two CTAs per SM) from there on.

Values: |C - A B^T| <= 2e-5 |A| |B|^T elementwise, as in the other GEMM tests.  Time: one
tile more than SMs must not cost a second wave of tiles (the ratio is 1.6 when it does,
1.0 when it does not).
"""
import numpy as np
import pytest
import torch

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

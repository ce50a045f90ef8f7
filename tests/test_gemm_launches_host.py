"""Which products of a network layer's backward pass share a launch of narrow tiles and
which go through the persistent kernel (a host rule on sizes, compiled alone).

The rule must send a layer whose products both fill the chip to the persistent kernel,
keep small layers in one launch, and keep the weight gradient of a small layer beside the
other product however large the batch is.
"""
import subprocess

import pytest

from paper_2507_04192_gb300 import build

SRC = r"""
#include <cstdio>
#include "mpm_umma.cuh"
using namespace mpm;
int main()
{
    int in, out, batch;
    while (scanf("%d %d %d", &in, &out, &batch) == 3) {
        UmmaGemm dw{}, da{};
        dw.M = out; dw.N = in; dw.K = batch;
        da.M = batch; da.N = in; da.K = out;
        printf("%d %d %d\n", (int)umma_wide(dw.M, dw.N, 152), (int)umma_wide(da.M, da.N, 152),
               (int)umma_share_launch(dw, da, 152));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cu").write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, str(d / "rule.cu"), "-o", str(d / "rule")], check=True)

    def ask(layers):
        out = subprocess.run([str(d / "rule")], input="\n".join("%d %d %d" % l for l in layers), capture_output=True,
                             text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return ask


def test_wide_layers_take_the_persistent_kernel(rule):
    # (inputs, outputs, batch): dW wide, dA wide, shared launch
    assert rule([(4096, 4096, 4096), (8192, 8192, 512), (4096, 32, 19456), (1024, 1024, 65536), (2304, 2304, 128)]) == [
        (1, 1, 0), (1, 0, 0), (0, 1, 0), (0, 1, 0), (1, 0, 0)]


def test_small_layers_share_a_launch(rule):
    layers = [(256, 32, 256), (256, 256, 256), (640, 256, 256), (512, 512, 512), (1024, 1024, 512)]
    assert rule(layers) == [(0, 0, 1)] * len(layers)


def test_small_weight_gradients_over_large_batches_share_a_launch(rule):
    layers = [(256, 256, 65536), (256, 256, 19456), (512, 512, 65536), (768, 768, 16384), (256, 32, 65536)]
    assert rule(layers) == [(0, 1, 1)] * len(layers)


def test_a_layer_with_neither_product_wide_always_shares(rule):
    layers = [(8 * i, 8 * o, 8 * b) for i in (1, 31, 32, 200) for o in (1, 32, 129) for b in (1, 17, 640)]
    for w1, w2, shared in rule(layers):
        assert shared or w1 or w2
        assert not (w1 and w2 and shared)

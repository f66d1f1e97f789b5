"""GPU: a layer that has just been written is read whole by the call behind it, which requests it before it waits."""
import pytest
import torch

from paper_2405_14917_b200 import binding as slim
from paper_2405_14917_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 5, 40])
@pytest.mark.parametrize("g", [64, 128, 256])
@pytest.mark.parametrize("N,K", [(64, 512), (2048, 2048)])
def test_a_layer_used_right_after_it_was_written(N, K, M, g):
    weights = [wl.make_weight_and_norms_device((6, 3, i), N, K, "cuda") for i in range(4)]
    x = torch.randn((M, K), device="cuda").half()
    layers = [slim.QuantLinear.from_weight(W, a, 2, g=g) for W, a in weights]
    ws = [slim.new_workspace(M, N, K, L.bits, g=g) for L in layers]
    codes = [slim.quantize_minmax(W, L.bits, g=g)[0] for (W, _), L in zip(weights, layers)]
    torch.cuda.synchronize()
    want = [L.forward(x, w) for L, w in zip(layers, ws)]
    torch.cuda.synchronize()
    got = []
    for i in range(24):
        W, a = weights[i % 4]
        L = slim.QuantLinear.from_weight(W, a, 2, g=g)               # buffers that held another layer a moment ago
        got.append((i % 4, L.forward(x, ws[i % 4])))
        del L
        same = layers[i % 4]                                         # and a layer whose codes are written over in place
        slim.pack_weights(torch.zeros_like(codes[i % 4]), same.bits, same.packed, g=g)
        slim.pack_weights(codes[i % 4], same.bits, same.packed, g=g)
        got.append((i % 4, same.forward(x, ws[i % 4])))
    torch.cuda.synchronize()
    for k, y in got:
        assert torch.equal(y, want[k])

"""GPU: weights that are Inf or NaN get the codes that the fp64 quantizer gives them, on every way to a layer."""
import numpy as np
import pytest
import torch

from paper_2405_14917_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _slim():
    from paper_2405_14917_b200 import binding
    return binding


def _weights(N, K, g):
    """A row of every kind in every group: Inf, -Inf, both, NaN, NaN with Inf, all NaN, the largest finite values; the others as they are."""
    W, a = wl.make_weight_and_norms_device((9, 2, g), N, K, "cuda")
    inf, nan = float("inf"), float("nan")
    rng = np.random.default_rng(g)
    for j in range(K // g):
        for r, values in enumerate(([inf], [-inf], [inf, -inf], [nan], [nan, inf], [nan, -inf, nan], [65504.0, -65504.0])):
            for v in values:
                W[(r + 3 * j) % N, g * j + int(rng.integers(g))] = v
        W[(7 + 3 * j) % N, g * j:g * (j + 1)] = nan
    return W, a


@pytest.mark.parametrize("g", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("avg", [2, 3])
def test_a_layer_in_one_call_is_the_layer_of_the_separate_calls(g, avg):
    slim = _slim()
    N, K = 48, 2048
    W, a = _weights(N, K, g)
    L = slim.QuantLinear.from_weight(W, a, avg, g=g)
    codes, scales, zeros = slim.quantize_minmax(W, L.bits, g=g)
    assert torch.equal(L.scales.view(torch.int16), scales.view(torch.int16)) and torch.equal(L.zeros.view(torch.int16), zeros.view(torch.int16))
    assert torch.equal(L.packed, slim.pack_weights(codes, L.bits, g=g))


@pytest.mark.parametrize("g", [32, 128, 512])
@pytest.mark.parametrize("bits", [1, 2, 3, 4])
def test_the_first_group_of_the_compensated_layer(g, bits):
    """Nothing has been added to the first group, so its codes are the quantizer's."""
    slim = _slim()
    N, K = 48, 512
    W, _ = _weights(N, K, g)
    b = np.full(K // g, bits, dtype=np.uint8)
    x = torch.randn((64, K), device="cuda").half()
    codes, scales, zeros = slim.gptq_quantize(W, x, b, quantizer="minmax", g=g)
    want_codes, want_scales, want_zeros = slim.quantize_minmax(W, b, g=g)
    assert torch.equal(codes[:, :g], want_codes[:, :g])
    assert torch.equal(scales[0].view(torch.int16), want_scales[0].view(torch.int16)) and torch.equal(zeros[0].view(torch.int16), want_zeros[0].view(torch.int16))


@pytest.mark.parametrize("g", [32, 128, 512])
def test_calibrated_quantizer(g):
    """No candidate has a finite loss in such a group; the codes follow from the scale and zero point that are returned."""
    slim = _slim()
    N, K = 48, 1024
    W, _ = _weights(N, K, g)
    b = np.array([1 + j % 4 for j in range(K // g)], dtype=np.uint8)
    codes, scales, zeros, _ = slim.quantize_sqc(W, b, g=g)
    w, G = W.double().view(N, K // g, g), K // g
    s, z = scales.double().t().unsqueeze(2), zeros.double().t().unsqueeze(2)
    levels = torch.from_numpy(2.0 ** b - 1).cuda().view(1, G, 1)
    q = torch.round(w / s) + z
    q = torch.where(torch.isnan(q), torch.zeros_like(q), torch.minimum(torch.clamp(q, min=0.0), levels))
    assert torch.equal(codes.view(N, G, g).double(), q)

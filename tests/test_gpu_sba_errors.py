"""GPU: the errors that the SBA search returns, against the same quantities in fp64 from torch on the device."""
import numpy as np
import pytest
import torch

from paper_2405_14917_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# norm of the difference of two error curves over the norm of the curve.  What is left between the device and fp64 are the
# fp32 sums of a product (a few 1e-6 of the error at 11008 columns) and the outputs, a few in a thousand, that those sums put
# on the other side of an fp16 rounding; leaving out the fp16 rounding of the outputs moves the curves below by 7e-5 to 1.5e-4
CURVE_RTOL = 4e-5


def _slim():
    from paper_2405_14917_b200 import binding
    return binding


def _kl(y, y_q):
    log_p = torch.log_softmax(y, dim=1)
    return (log_p.exp() * (log_p - torch.log_softmax(y_q, dim=1))).sum(dim=1).mean().item()


def _errors(W, x, a, avg, g):
    """Every candidate as the layer it would become: fp16 outputs, and from 17 tokens on fp16 weights."""
    slim = _slim()
    N, K = W.shape
    M, G = x.shape[0], K // g
    sal = slim.group_salience(W, a, g).cpu().numpy()
    xd = x.double()
    y = xd @ W.double().t()
    out = []
    for p in range(G // 2 + 1):
        codes, s, z = slim.quantize_minmax(W, slim.allocate_bits(sal, avg, p), g=g)
        w = (s.t().double().unsqueeze(2) * (codes.view(N, G, g).double() - z.t().double().unsqueeze(2))).reshape(N, K)
        if M > slim.GEMV_MAX_M:
            w = w.half().double()
        out.append(_kl(y, (xd @ w.t()).half().double()))
    return np.array(out)


def _inputs(N, K, M, seed, scale=1.0):
    W, a = wl.make_weight_and_norms_device((seed, 5, 0), N, K, "cuda")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = (scale * torch.randn((M, K), generator=gen, device="cuda")).half()
    return W, a, x


@pytest.mark.parametrize("N,K,M,g,avg", [(2048, 4096, 36, 128, 3), (2048, 11008, 24, 128, 2), (2048, 8192, 12, 64, 2), (512, 8192, 16, 256, 3),
                                         (1024, 8192, 17, 512, 2)])
def test_a_candidate_is_the_layer_it_would_become(N, K, M, g, avg):
    W, a, x = _inputs(N, K, M, seed=N + K + M)
    _, _, got = _slim().sba_search(W, x, a, avg, g=g)
    want = _errors(W, x, a, avg, g)
    assert np.linalg.norm(got - want) <= CURVE_RTOL * np.linalg.norm(want), (np.linalg.norm(got - want) / np.linalg.norm(want))


@pytest.mark.parametrize("std", [1e-2, 1e-3])
@pytest.mark.parametrize("N,K,M", [(512, 512, 16), (4096, 1024, 40)])
def test_errors_of_small_outputs_keep_their_digits(N, K, M, std):
    """The divergence is second order in the outputs' difference: 1e-7 and less here, with no absolute floor in the comparison."""
    W, a, x = _inputs(N, K, M, seed=7 + K, scale=std / (0.02 * np.sqrt(2 * K)))
    _, _, got = _slim().sba_search(W, x, a, 2)
    want = _errors(W, x, a, 2, 128)
    assert np.linalg.norm(got - want) <= CURVE_RTOL * np.linalg.norm(want), (np.linalg.norm(got - want) / np.linalg.norm(want))


@pytest.mark.parametrize("M", [12, 20])
def test_errors_of_outputs_that_are_far_apart(M):
    """One input per token, a power of two: every output is one product, exact before it is rounded to fp16, so the two sides
    have the same outputs and only the divergence is compared.  It is computed from e = exp(y - m) in fp32, whose argument
    is off by 2^-24 |y - m|: 1e-5 where |y - m| is 200, beyond which e weighs nothing."""
    N, K = 320, 1024
    W, a, _ = _inputs(N, K, M, seed=3)
    x = torch.zeros((M, K), dtype=torch.float16, device="cuda")
    for t in range(M):
        x[t, 37 * t + 5] = 2.0 ** (t if t < 8 else 13 - t % 3)       # outputs from 0.02 to 1000 and more, differences likewise
    _, _, got = _slim().sba_search(W, x, a, 2)
    want = _errors(W, x, a, 2, 128)
    assert want.max() > 10
    assert np.abs(got - want).max() <= 2e-5 * want.max(), (got, want)
    for t in (0, 11):                                                # a token of each kind by itself
        _, _, got = _slim().sba_search(W, x[t:t + 1].contiguous(), a, 2)
        want = _errors(W, x[t:t + 1], a, 2, 128)
        assert np.abs(got - want).max() <= 2e-5 * want.max(), (t, got, want)


@pytest.mark.parametrize("N,K,M,g,avg,include_uniform", [(512, 4096, 256, 32, 2, True), (512, 4096, 130, 32, 3, False), (16, 8192, 250, 32, 2, True)])
def test_a_small_workspace_means_several_walks_and_the_same_errors(N, K, M, g, avg, include_uniform):
    slim = _slim()
    W, a, x = _inputs(N, K, M, seed=11)
    G = K // g
    layer = N * K + N * K * (avg + 1) // 8 + 4 * N * G + 6 * M * N + 8 * M * (G // 2 + 1)      # codes, packed, scales, zeros, outputs, errors
    full = slim.sba_workspace_bytes(M, N, K, avg, g)
    assert full > 1.3 * layer                                        # the shapes are ones where it matters
    results = []
    for size in (full, layer, (full + layer) // 2):
        ws = torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda")
        results.append(slim.sba_search(W, x, a, avg, include_uniform, workspace=ws, g=g))
    for p, bits, errors in results[1:]:
        assert p == results[0][0] and (bits == results[0][1]).all() and (errors == results[0][2]).all()
    with pytest.raises(slim.SlimError):
        slim.sba_search(W, x, a, avg, workspace=torch.empty(layer - 256, dtype=torch.uint8, device="cuda"), g=g)


# A CTA of the search takes 16, 32, 48, 64 or 80 rows, whatever fills the last wave of 148 CTAs per 128 tokens best.  Below: every one of
# them at each width of the operand's chunk (groups of 32, 64, 128 columns, and several chunks per group), with a last CTA that
# is full, ends in its first half, or reaches into the second, and with a second and third block of tokens.
@pytest.mark.parametrize("rows,N,M", [(16, 1184, 129), (32, 3280, 20), (32, 1200, 200), (48, 4752, 20), (48, 2384, 200), (64, 7120, 20),
                                      (80, 9488, 20), (80, 3168, 300), (80, 4752, 129)])
@pytest.mark.parametrize("g", [32, 64, 128, 256])
def test_every_form_of_the_search_kernel(rows, N, M, g):
    K = 768
    W, a, x = _inputs(N, K, M, seed=rows + N + g)
    _, _, got = _slim().sba_search(W, x, a, 2 + (g >> 6 & 1), g=g)
    want = _errors(W, x, a, 2 + (g >> 6 & 1), g)
    assert np.linalg.norm(got - want) <= CURVE_RTOL * np.linalg.norm(want), (np.linalg.norm(got - want) / np.linalg.norm(want))

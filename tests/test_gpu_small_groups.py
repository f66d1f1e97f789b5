"""Groups of 32 and 64 columns: the linear layer at the edges of its token and row tiles."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from paper_2405_14917_b200 import workloads as wl
from tests.helpers import check_output

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [32, 64])
@pytest.mark.parametrize("N,K,M", [(16, 128, 1), (48, 640, 8), (48, 1152, 9), (80, 640, 16), (48, 640, 17), (16, 2048, 33), (112, 384, 70),
                                   (48, 3968, 3), (48, 4096, 3), (16, 4224, 12), (32, 10112, 1), (16, 10240, 9)])
def test_tiles_of_tokens_and_rows(N, K, M, g):
    """Row tiles that are odd in number, token tiles of 8, 16 and 32 with remainders, more and fewer groups than warps, as many
    groups as 32 warps are taken from and fewer, every width, zero points that are no integers."""
    rng = np.random.default_rng(N + K + M + g)
    G = K // g
    bits = rng.permutation(np.resize(np.array([2, 3, 1, 4], np.uint8), G))
    codes = np.concatenate([rng.integers(0, 1 << b, (N, g)) for b in bits], axis=1).astype(np.uint8)
    scales = rng.uniform(0.01, 0.1, (G, N)).astype(np.float16)
    zeros = rng.uniform(0, 3, (G, N)).astype(np.float16)
    x = rng.normal(0, 1, (M, K)).astype(np.float16)
    ws = slim.new_workspace(M, N, K, bits, g=g)
    packed = slim.pack_weights(torch.from_numpy(codes).cuda(), bits, g=g)
    call = slim.mpq_gemv if M <= slim.GEMV_MAX_M else slim.mpq_gemm
    y = call(torch.from_numpy(x).cuda(), packed, bits, torch.from_numpy(scales).cuda(), torch.from_numpy(zeros).cuda(), N, ws, g=g)
    slim.workspace_status(ws)
    W = np.repeat(scales.astype(np.float64), g, axis=0).T * (codes - np.repeat(zeros.astype(np.float64), g, axis=0).T)
    check_output(y.cpu().numpy(), x.astype(np.float64) @ W.T, f"{N}x{K} M={M} g={g}")


@pytest.mark.parametrize("g", [32, 64])
@pytest.mark.parametrize("N,M", [(16 * 148, 1), (16 * 149, 8), (16 * 148, 9), (16 * 149, 16), (32 * 148, 32), (32 * 148 + 16, 17), (32 * 49 + 16, 70)])
def test_blocks_that_share_an_sm_and_blocks_that_do_not(N, M, g):
    """As many blocks as SMs and one more (148 of them; two row tiles per block from 17 tokens on), every width; the first
    rows by themselves, which take the form for a block per SM, give the same bits."""
    K = 384
    rng = np.random.default_rng(N + M + g)
    bits = rng.permutation(np.resize(np.array([2, 3, 1, 4], np.uint8), K // g))
    codes = np.concatenate([rng.integers(0, 1 << b, (N, g)) for b in bits], axis=1).astype(np.uint8)
    scales = rng.uniform(0.01, 0.1, (K // g, N)).astype(np.float16)
    zeros = rng.uniform(0, 3, (K // g, N)).astype(np.float16)
    x = rng.normal(0, 1, (M, K)).astype(np.float16)
    ws = slim.new_workspace(M, N, K, bits, g=g)

    def run(n):
        packed = slim.pack_weights(torch.from_numpy(codes[:n]).cuda(), bits, g=g)
        call = slim.mpq_gemv if M <= slim.GEMV_MAX_M else slim.mpq_gemm
        s, z = (torch.from_numpy(np.ascontiguousarray(t[:, :n])).cuda() for t in (scales, zeros))
        return call(torch.from_numpy(x).cuda(), packed, bits, s, z, n, ws, g=g)

    y = run(N)
    slim.workspace_status(ws)
    W = np.repeat(scales.astype(np.float64), g, axis=0).T * (codes - np.repeat(zeros.astype(np.float64), g, axis=0).T)
    check_output(y.cpu().numpy(), x.astype(np.float64) @ W.T, f"{N}x{K} M={M} g={g}")
    assert torch.equal(run(64), y[:, :64])                          # a few rows: one block per SM


def test_more_tokens_than_one_launch_takes():
    """65535 blocks of 32 tokens are the second grid dimension's limit; a second launch does the rest."""
    N, K, g, M = 16, 128, 64, 65535 * 32 + 45
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    W, norms = wl.make_weight_and_norms_device((5, N, K), N, K, "cuda")
    L = slim.QuantLinear.from_weight(W, norms, 2, g=g)
    x = torch.randn((M, K), generator=gen, device="cuda", dtype=torch.float16)
    y = L.forward(x, slim.new_workspace(M, N, K, L.bits, g=g))
    for m0 in (0, 65535 * 32 - 100, M - 300):                       # the same tokens by themselves
        part = x[m0:m0 + 200].contiguous()
        assert torch.equal(L.forward(part, slim.new_workspace(200, N, K, L.bits, g=g)), y[m0:m0 + 200])

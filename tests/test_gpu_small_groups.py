"""Groups of 32 and 64 columns: the linear layer at the edges of its token and row tiles."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from tests.helpers import check_output

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [32, 64])
@pytest.mark.parametrize("N,K,M", [(16, 128, 1), (48, 640, 8), (48, 1152, 9), (80, 640, 16), (48, 640, 17), (16, 2048, 33), (112, 384, 70)])
def test_tiles_of_tokens_and_rows(N, K, M, g):
    """Row tiles that are odd in number, token tiles of 8, 16 and 32 with remainders, more and fewer groups than warps, every
    width, zero points that are no integers."""
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

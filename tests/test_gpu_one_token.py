"""The single-token kernel at the edges of its staging and of its tile counts, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim

from tests.helpers import check_output, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,avg", [
    (32, 128, 2), (32, 384, 3),          # fewer K-tiles than the four that a warp stages at once
    (48, 640, 3), (32, 8576, 2),         # a remainder of one; 67 K-tiles: a second pass of some warps, 3 in the last one
    (20800, 256, 2), (23680, 128, 3),    # 1300 and 1480 row tiles: five tile pairs per CTA, the last size that is one wave on 148 SMs
])
def test_staging_remainders_and_tile_pairs(N, K, avg):
    L = oracle_layer(N, K, avg, 1, seed_name="one-token")
    packed = torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda()
    ws = slim.new_workspace(1, N, K, L["bits"])
    y = slim.mpq_gemv(torch.from_numpy(L["x"]).cuda(), packed, L["bits"], torch.from_numpy(L["scales"]).cuda(),
                      torch.from_numpy(L["zeros"]).cuda(), N, ws)
    slim.workspace_status(ws)
    check_output(y.cpu().numpy(), orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"]), f"{N}x{K}")


@pytest.mark.parametrize("bits", [[1, 1, 1, 1, 1], [4, 4, 4, 4, 3], [1, 2, 3, 4, 4, 3, 2, 1], [3, 3, 2, 2, 1]])
def test_every_mixture_of_widths_in_a_warp(bits):
    """Four neighbouring K-tiles share a warp; what its lanes do differs with the width."""
    rng = np.random.default_rng(sum(b << (2 * i) for i, b in enumerate(bits)))
    G, N = len(bits), 64
    codes = np.concatenate([rng.integers(0, 1 << b, (N, 128)) for b in bits], axis=1).astype(np.uint8)
    scales = rng.uniform(0.01, 0.1, (G, N)).astype(np.float16)
    zeros = np.stack([rng.integers(0, 1 << b, N) for b in bits]).astype(np.float16)
    x = rng.normal(0, 1, (1, 128 * G)).astype(np.float16)
    b = np.array(bits, np.uint8)
    ws = slim.new_workspace(1, N, 128 * G, b)
    y = slim.mpq_gemv(torch.from_numpy(x).cuda(), torch.from_numpy(orc.pack(codes, b)).cuda(), b, torch.from_numpy(scales).cuda(),
                      torch.from_numpy(zeros).cuda(), N, ws)
    slim.workspace_status(ws)
    check_output(y.cpu().numpy(), orc.linear_f64(x, codes, scales, zeros), str(bits))

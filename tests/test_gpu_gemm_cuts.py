"""Few tiles on the batched path: several CTA pairs per tile, each of which finishes some of the tile's 32-token pieces."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from tests.helpers import check_output, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M", [
    (16, 8192, 17),       # the kernel for a few tokens takes this one
    (272, 4096, 40),      # fewer pieces than pairs; a second row block of one tile
    (512, 8192, 200),     # seven pieces in a tile of 256 tokens
    (256, 2048, 300),     # a second token tile with two pieces, the last one of 12 tokens
    (80, 16384, 128),     # the most pairs
    (1024, 1024, 330),    # tiles narrower than they could be, a last one of fewer tokens
    (1296, 512, 700),     # whole tiles of equal width
])
def test_pieces_and_pairs(N, K, M):
    _check(N, K, M)


@pytest.mark.parametrize("N,K,M", [(16, 8320, 17), (272, 8320, 32)])
def test_one_piece_and_several_pairs(N, K, M):
    """65 K-tiles are too many for the kernel for a few tokens, so these are tiles of the batched one with a single piece: the
    pair that has it finishes the tile, the others only hand over theirs."""
    assert slim.workspace_bytes(M, N, K, np.full(K // 128, 3, dtype=np.uint8)) >= 4 * ((N + 255) // 256) * 128 * 128 * 4     # two pairs per tile at least
    _check(N, K, M)


def _check(N, K, M):
    L = oracle_layer(N, K, 3, M, seed_name="gemm-cuts")
    ref = orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"])
    x, packed = torch.from_numpy(L["x"]).cuda(), torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda()
    sc, zp = torch.from_numpy(L["scales"]).cuda(), torch.from_numpy(L["zeros"]).cuda()
    ws = slim.new_workspace(M, N, K, L["bits"])
    first = slim.mpq_gemm(x, packed, L["bits"], sc, zp, N, ws)
    check_output(first.cpu().numpy(), ref, f"{N}x{K} M={M}")
    for _ in range(3):                                   # the flags are back at zero, and the order of the sums is fixed
        y = torch.full_like(first, float("nan"))
        slim.mpq_gemm(x, packed, L["bits"], sc, zp, N, ws, y)
        assert torch.equal(y, first)
    slim.workspace_status(ws)
    words = ws[256:256 + 1024].cpu().numpy()
    assert not words.any()

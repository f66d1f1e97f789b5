"""GPU: 2 to 16 tokens on both sides of every line between the kernel that cuts a layer over the GPU and the general one."""
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from tests.helpers import check_output, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M", [
    (2048, 128, 2), (4096, 128, 3), (512, 512, 3), (528, 512, 3), (512, 512, 4),        # one K-tile, 2^18 weights, two and three tokens
    (512, 8192, 9), (1168, 8192, 9), (512, 8064, 16), (512, 8192, 8), (16, 8192, 16),   # a pair of row tiles, 64 K-tiles, more than 8 tokens
    (1024, 28672, 9), (1040, 32768, 16), (512, 32768, 9),                               # K-tiles and warps that the longest K leaves room for
])
def test_both_kernels(N, K, M):
    L = oracle_layer(N, K, 3, M, seed_name="few-or-general")
    ref = orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"])
    x, packed = torch.from_numpy(L["x"]).cuda(), torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda()
    sc, zp = torch.from_numpy(L["scales"]).cuda(), torch.from_numpy(L["zeros"]).cuda()
    ws = slim.new_workspace(M, N, K, L["bits"])
    y = slim.mpq_gemv(x, packed, L["bits"], sc, zp, N, ws)
    check_output(y.cpu().numpy(), ref, f"{N}x{K} M={M}")
    small = torch.zeros(256, dtype=torch.uint8, device="cuda")
    check_output(slim.mpq_gemv(x, packed, L["bits"], sc, zp, N, small).cpu().numpy(), ref, f"{N}x{K} M={M}, the smallest workspace")
    slim.workspace_status(ws)
    slim.workspace_status(small)

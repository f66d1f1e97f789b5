"""The kernel that cuts one layer of 2 to 16 tokens over the whole GPU, where its cuts have remainders."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from tests.helpers import check_output, oracle_layer

pytestmark = pytest.mark.gpu


def _run(x, codes, bits, scales, zeros, g=128):
    M, K = x.shape
    N = codes.shape[0]
    ws = slim.new_workspace(M, N, K, bits, g=g)
    packed = slim.pack_weights(torch.from_numpy(codes).cuda(), bits, g=g)
    y = slim.mpq_gemv(torch.from_numpy(x).cuda(), packed, bits, torch.from_numpy(scales).cuda(), torch.from_numpy(zeros).cuda(), N, ws, g=g)
    slim.workspace_status(ws)
    return y.cpu().numpy()


@pytest.mark.parametrize("M", [2, 3, 8, 9, 16])
@pytest.mark.parametrize("N,K,avg", [
    (16, 128, 2),           # one tile, one K-tile: CTAs without any
    (48, 1152, 3),          # an odd tile; nine K-tiles over the CTAs of a cluster
    (2416, 640, 2),         # 151 tiles: a last cluster with fewer rows, a last pair of one tile
    (1200, 8320, 3),        # 65 K-tiles over clusters of eight
])
def test_remainders(N, K, avg, M):
    L = oracle_layer(N, K, avg, M, seed_name="few-tokens")
    y = _run(L["x"], L["codes"], L["bits"], L["scales"], L["zeros"])
    check_output(y, orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"]), f"{N}x{K} M={M}")


@pytest.mark.parametrize("M", [17, 24, 25, 32])
@pytest.mark.parametrize("N,K,avg", [(528, 2048, 3), (1040, 8192, 2), (48, 2176, 3)])
def test_three_and_four_token_tiles(N, K, avg, M):
    """The batched entry point sends its fewest tokens here."""
    L = oracle_layer(N, K, avg, M, seed_name="few-batched")
    ws = slim.new_workspace(M, N, K, L["bits"])
    y = slim.mpq_gemm(torch.from_numpy(L["x"]).cuda(), torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda(), L["bits"],
                      torch.from_numpy(L["scales"]).cuda(), torch.from_numpy(L["zeros"]).cuda(), N, ws)
    slim.workspace_status(ws)
    check_output(y.cpu().numpy(), orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"]), f"{N}x{K} M={M}")


@pytest.mark.parametrize("N,K,M", [(8192, 8192, 8), (4096, 16384, 16), (13824, 2560, 12), (640, 32768, 1), (640, 32768, 16)])
def test_more_bytes_than_the_ring_holds(N, K, M):
    """K-tiles that take the slot of an earlier one, every width among them; 32768 columns, where one token does not fit
    the single-token kernel and sixteen do not fit this one.  Reference: the plain product in fp64."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N + K + M)
    G = K // 128
    bits = np.tile(np.array([2, 4, 3, 1, 4], np.uint8), G // 5 + 1)[:G]
    top = torch.from_numpy((1 << bits.astype(np.int64)) - 1).cuda()
    codes = (torch.rand((N, G, 128), device="cuda", generator=gen) * (top[None, :, None] + 1)).floor().clamp(max=top[None, :, None]).to(torch.uint8)
    scales = (0.01 + 0.05 * torch.rand((G, N), device="cuda", generator=gen)).to(torch.float16)
    zeros = (torch.rand((G, N), device="cuda", generator=gen) * top[:, None]).round().to(torch.float16)
    x = torch.randn((M, K), device="cuda", generator=gen).to(torch.float16)
    y = _run(x.cpu().numpy(), codes.reshape(N, K).cpu().numpy(), bits, scales.cpu().numpy(), zeros.cpu().numpy())
    ref = torch.zeros((M, N), dtype=torch.float64, device="cuda")
    for j in range(G):
        w = scales[j, :, None].double() * (codes[:, j].double() - zeros[j, :, None].double())
        ref += x[:, 128 * j:128 * (j + 1)].double() @ w.t()
    check_output(y, ref.cpu().numpy(), f"{N}x{K} M={M}")


@pytest.mark.parametrize("g", [256, 512])
def test_wider_groups(g):
    L = oracle_layer(160, 2048, 2, 5, seed_name="few-wide", bits=np.repeat(np.array([1, 3, 2, 4, 2, 2, 3, 1], np.uint8)[: 2048 // g], g // 128))
    step = g // 128
    scales, zeros = L["scales"][::step], L["zeros"][::step]            # one row per group of g columns
    y = _run(L["x"], L["codes"], L["bits"][::step].copy(), scales.copy(), zeros.copy(), g=g)
    ref = orc.linear_f64(L["x"], L["codes"], np.repeat(scales, step, axis=0), np.repeat(zeros, step, axis=0))
    check_output(y, ref, f"g={g}")


@pytest.mark.parametrize("M", [20, 24, 33, 41, 49, 57])
def test_sets_of_every_number_of_token_tiles(M):
    """Layer sets whose widest layer needs three, five, six, seven or eight MMA tiles, next to layers of fewer tokens; few
    row blocks, so that these are cut into parts."""
    layers = [oracle_layer(304, 1152, 3, M, seed_name="set-tiles", block=0), oracle_layer(512, 1024, 2, 3, seed_name="set-tiles", block=1)]
    entries = []
    for L in layers:
        layer = slim.QuantLinear(torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda(), L["bits"], torch.from_numpy(L["scales"]).cuda(),
                                 torch.from_numpy(L["zeros"]).cuda(), L["N"], L["K"])
        entries.append((layer, torch.from_numpy(L["x"]).cuda(), torch.full((L["M"], L["N"]), float("nan"), dtype=torch.float16, device="cuda")))
    s = slim.LayerSet(entries)
    assert s.info["token_tiles"] == (M + 7) // 8
    s.run()
    s.check()
    for L, (_, _, y) in zip(layers, entries):
        check_output(y.cpu().numpy(), orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"]), f"M={L['M']}")

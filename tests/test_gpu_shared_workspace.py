"""GPU: one workspace for calls of every kind in turn: the flags of the batched kernel are zero whenever it starts."""
import pytest
import torch

from paper_2405_14917_b200 import binding as slim
from paper_2405_14917_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _layer(N, K, avg=3, g=128):
    W, a = wl.make_weight_and_norms_device((8, N, K), N, K, "cuda")
    return slim.QuantLinear.from_weight(W, a, avg, g=g)


# (N, K) and tokens of calls whose workspace holds more than a status word: x staged for the general kernel, and for a layer of
# 32 MB and more its plan, counters, staged x and partial sums, with one and with several tokens
OTHERS = [(256, 8192, 12), (64, 16384, 16), (16384, 8192, 1), (16384, 8192, 5), (14336, 8192, 16)]


@pytest.mark.parametrize("N,K,M", [(512, 8192, 200), (1024, 4096, 40)])
def test_a_workspace_shared_by_all_calls(N, K, M):
    layer = _layer(N, K)
    others = [(_layer(n, k), torch.randn((m, k), device="cuda").half(), m) for n, k, m in OTHERS]
    x = torch.randn((M, K), device="cuda").half()
    size = max([layer.workspace_bytes(M)] + [o.workspace_bytes(m) for o, _, m in others])
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    slim.workspace_init(ws)
    want = layer.forward(x, slim.new_workspace(M, N, K, layer.bits))
    assert layer.workspace_bytes(M) > 4096                            # the tiles are cut: the flags are used
    for other, xo, m in others:
        own = slim.new_workspace(m, other.N, other.K, other.bits)
        y = other.forward(xo, own)
        assert torch.equal(other.forward(xo, ws), y)
        assert not ws[256:1280].any()                                 # before the call that would wait on them
        assert torch.equal(layer.forward(x, ws), want)
        slim.workspace_status(ws)


@pytest.mark.parametrize("N,K,M", [(16384, 8192, 1), (16384, 8192, 5), (256, 8192, 12)])
def test_a_workspace_without_room_for_the_flags(N, K, M):
    layer = _layer(N, K)
    x = torch.randn((M, K), device="cuda").half()
    want = layer.forward(x, slim.new_workspace(M, N, K, layer.bits))
    ws = torch.zeros(layer.workspace_bytes(M) - 1024, dtype=torch.uint8, device="cuda")
    assert torch.equal(layer.forward(x, ws), want)
    slim.workspace_status(ws)

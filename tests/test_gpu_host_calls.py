"""The two ways a call takes into the library (host module; general path for everything that needs converting) agree."""
import numpy as np
import pytest
import torch

from paper_2405_14917_b200 import binding as slim
from paper_2405_14917_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _layer(N, K, g):
    W, norms = wl.make_weight_and_norms_device((5, N, K), N, K, "cuda")
    return slim.QuantLinear.from_weight(W, norms, 2, g=g)


@pytest.mark.parametrize("M,g", [(1, 128), (1, 64), (5, 128), (40, 128)])
def test_bit_maps_outputs_and_streams(M, g):
    L = _layer(64, 512, g)
    x = torch.randn((M, 512), device="cuda").to(torch.float16)
    ws = slim.new_workspace(M, 64, 512, L.bits, g=g)
    call = slim.mpq_gemv if M <= slim.GEMV_MAX_M else slim.mpq_gemm
    args = (L.packed, L.bits, L.scales, L.zeros, 64, ws)
    y = call(x, *args, g=g)
    assert y.shape == (M, 64) and y.dtype == torch.float16 and not y.requires_grad
    # other forms of the same bit map, the output given, a tensor subclass, N as a numpy integer, another stream
    strided = np.repeat(L.bits, 2)[::2]
    for bits in (list(L.bits), L.bits.astype(np.int64), strided, torch.from_numpy(L.bits)):
        assert torch.equal(call(x, L.packed, bits, L.scales, L.zeros, 64, ws, g=g), y)
    out = torch.full((M, 64), float("nan"), dtype=torch.float16, device="cuda")
    assert call(x, *args, out, g) is out and torch.equal(out, y)
    assert torch.equal(call(torch.nn.Parameter(x, requires_grad=False), *args, g=g), y)
    assert torch.equal(call(x, L.packed, L.bits, L.scales, L.zeros, np.int64(64), ws, g=g), y)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        y2 = call(x, *args, g=g)
    torch.cuda.synchronize()
    assert torch.equal(y2, y)
    slim.workspace_status(ws)


def test_calls_that_must_fail():
    L = _layer(64, 512, 128)
    x = torch.zeros((1, 512), dtype=torch.float16, device="cuda")
    ws = slim.new_workspace(1, 64, 512, L.bits)
    ok = [x, L.packed, L.bits, L.scales, L.zeros, 64, ws]
    for at, bad in ((0, x.float()), (0, x.cpu()), (0, x.expand(2, 512)), (1, L.packed.to(torch.int8)), (3, L.scales.cpu()),
                    (4, L.zeros.t()), (6, ws.cpu())):
        args = list(ok)
        args[at] = bad
        with pytest.raises(TypeError):
            slim.mpq_gemv(*args)
    with pytest.raises(TypeError):
        slim.mpq_gemv(*ok, torch.empty((1, 64), device="cuda"))
    for at, bad in ((6, ws[:16]), (6, None), (2, L.bits + 4), (5, 63)):
        args = list(ok)
        args[at] = bad
        with pytest.raises((slim.SlimError, RuntimeError, TypeError)):
            slim.mpq_gemv(*args)
    with pytest.raises(slim.SlimError):
        slim.mpq_gemm(*ok)                              # one token is not the batched path's
    torch.cuda.synchronize()


def test_what_torch_raises_is_what_the_caller_gets():
    L = _layer(64, 512, 128)
    x = torch.zeros((1, 512), dtype=torch.float16, device="cuda")
    ws = slim.new_workspace(1, 64, 512, L.bits)
    ok = [x, L.packed, L.bits, L.scales, L.zeros, 64, ws]
    for at in (0, 1, 3, 6):                             # no strides to ask for
        args = list(ok)
        args[at] = ok[at].to_sparse()
        with pytest.raises((TypeError, RuntimeError)):
            slim.mpq_gemv(*args)
    many = torch.zeros((200, 512), dtype=torch.float16, device="cuda")
    with pytest.raises(torch.OutOfMemoryError):         # an output of 800 GB
        slim.mpq_gemm(many, L.packed, L.bits, L.scales, L.zeros, 2**31 - 16, ws)


def test_bytes_are_not_a_bit_map():
    L = _layer(64, 512, 128)
    x = torch.randn((1, 512), device="cuda").to(torch.float16)
    ws = slim.new_workspace(1, 64, 512, L.bits)
    with pytest.raises(ValueError):
        slim.mpq_gemv(x, L.packed, L.bits.tobytes(), L.scales, L.zeros, 64, ws)
    y = slim.mpq_gemv(x, L.packed, L.bits, L.scales, L.zeros, 64, ws)
    assert torch.equal(slim.mpq_gemv(x, L.packed, bytearray(L.bits), L.scales, L.zeros, 64, ws), y)

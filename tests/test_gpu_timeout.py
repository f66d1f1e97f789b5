"""GPU test of the device-side time-out path: a bounded wait that runs out is reported through the workspace
status word as SLIM_ERR_TIMEOUT, the word is cleared by the query, and the workspace and the context stay usable.
The wait that runs out belongs to a kernel made for this (slim_selftest_wait_timeout: a barrier that nothing
signals, a limit of a millisecond); no kernel of the hot path is starved or broken to get there."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from paper_2405_14917_b200 import workloads as wl
from tests.helpers import check_output, oracle_layer

pytestmark = pytest.mark.gpu


def quantised_layer(N, K, avg=2):
    W, a = wl.make_weight_and_norms_device((47, N, K), N, K, "cuda")
    return slim.QuantLinear.from_weight(W, a, avg)


def test_bounded_wait_runs_out_and_is_reported_once():
    from paper_2405_14917_b200 import binding as slim
    L = oracle_layer(256, 512, 2, 1)
    ws = slim.new_workspace(1, 256, 512, L["bits"])
    slim.workspace_status(ws)                                  # clean to begin with
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    slim.selftest_wait_timeout(ws, limit_us=1000)
    t1.record()
    with pytest.raises(slim.SlimError) as e:
        slim.workspace_status(ws)
    assert e.value.status == -6                                # SLIM_ERR_TIMEOUT
    assert 0.9 <= t0.elapsed_time(t1) <= 50.0                  # the kernel waited about the limit, then returned by itself
    slim.workspace_status(ws)                                  # reported once: the word is cleared
    # the same workspace serves an ordinary call afterwards
    packed = torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda()
    y = slim.mpq_gemv(torch.from_numpy(L["x"]).cuda(), packed, L["bits"], torch.from_numpy(L["scales"]).cuda(),
                      torch.from_numpy(L["zeros"]).cuda(), 256, ws)
    slim.workspace_status(ws)
    check_output(y.cpu().numpy(), orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"]), "after a time-out")


def test_selftest_arguments_are_validated():
    from paper_2405_14917_b200 import binding as slim
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    for bad in (0, 100001):
        with pytest.raises(slim.SlimError) as e:
            slim.selftest_wait_timeout(ws, limit_us=bad)
        assert e.value.status == -1
    with pytest.raises(slim.SlimError) as e:
        slim.selftest_wait_timeout(torch.zeros(64, dtype=torch.uint8, device="cuda"), limit_us=10)
    assert e.value.status == -4


@pytest.mark.parametrize("N,K,M", [(26624, 4096, 5), (28672, 8192, 24), (512, 8192, 200)])
def test_flags_that_a_kernel_left_behind_are_cleared_with_the_status(N, K, M):
    """The state that a kernel which gave up leaves (written from the host): its words of the header, and flags that are not zero.  The query that
    reports it leaves a workspace whose next call, large layers cut over the GPU in either form, is right."""
    layer, x = quantised_layer(N, K), torch.randn((M, K), device="cuda").half()
    ws = slim.new_workspace(M, N, K, layer.bits)
    y = layer.forward(x, ws)
    slim.workspace_status(ws)
    ws[:8].view(torch.int32).fill_(1)
    ws[256:1280].view(torch.int32).fill_(0x21212121)
    with pytest.raises(slim.SlimError) as e:
        slim.workspace_status(ws)
    assert e.value.status == -6
    assert not ws[:1280].any()
    assert torch.equal(layer.forward(x, ws), y)
    slim.workspace_status(ws)


def test_a_workspace_of_the_header_alone_is_cleared_no_further():
    buffer = torch.full((2048,), 7, dtype=torch.uint8, device="cuda")
    ws = buffer[:256]
    ws.zero_()
    ws[:4].view(torch.int32).fill_(1)                          # a kernel without flags reports in the first word
    with pytest.raises(slim.SlimError):
        slim.workspace_status(ws)
    assert not ws.any() and (buffer[256:] == 7).all()

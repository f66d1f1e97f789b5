"""GPU parity: a layer from its weight in one call (slim_quantize_layer) against the oracle's quantizer and packer."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _slim():
    from paper_2405_14917_b200 import binding
    return binding


def _check(W, a, avg, g, p=-1):
    slim = _slim()
    N, K = W.shape
    L = slim.QuantLinear.from_weight(torch.from_numpy(W).cuda(), torch.from_numpy(a).cuda(), avg, p=p, g=g)
    sal = slim.group_salience(torch.from_numpy(W).cuda(), torch.from_numpy(a).cuda(), g).cpu().numpy()
    assert (L.bits == slim.allocate_bits(sal, avg, p)).all()
    codes, scales, zeros = orc.quantize_minmax(W, L.bits, g)
    assert (L.scales.cpu().numpy().view(np.uint16) == scales.view(np.uint16)).all()
    assert (L.zeros.cpu().numpy().view(np.uint16) == zeros.view(np.uint16)).all()
    assert (L.packed.cpu().numpy() == orc.pack(codes, L.bits, g)).all()
    return L


# one tile and ragged numbers of tiles (a block is eight (tile, group) pairs), one group to 1024 of them
@pytest.mark.parametrize("g,N,K", [(128, 16, 128), (128, 272, 1408), (128, 1040, 4096), (32, 48, 384), (32, 16, 32768), (64, 272, 1152),
                                   (256, 144, 2304), (512, 80, 2560), (512, 16, 512)])
@pytest.mark.parametrize("avg", [2, 3])
def test_layer_from_weight_equals_the_oracle(g, N, K, avg):
    seed = wl.layer_seed("test", f"build-{N}x{K}-{g}", avg)
    _check(wl.make_weight(seed, N, K), wl.make_act_norms(seed, K), avg, g)


def test_layer_from_weight_edge_groups_and_ties():
    """Groups of one sign, of zeros (equal saliences: the lower index ranks higher), beyond the fp16 range of a one-bit
    scale, of subnormals, and weights exactly half-way between two codes; a weight that starts off a 32-byte boundary."""
    rng = np.random.default_rng(17)
    N, K = 48, 1024
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float16)
    W[:, 0:128] = np.abs(W[:, 0:128])
    W[:, 128:256] = -np.abs(W[:, 128:256])
    W[:, 256:512] = 0
    W[:, 512:640] = np.clip(rng.standard_normal((N, 128)) * 3e4, -6e4, 6e4).astype(np.float16)
    W[:, 640:768] = (rng.standard_normal((N, 128)) * 1e-7).astype(np.float16)
    for j, levels in ((6, 3), (7, 7)):                     # ties under two and three bits
        k = rng.integers(0, levels, (N, 128))
        w = (k + 0.5) * 2.0 ** -6
        w[:, 0], w[:, 1] = 0.0, levels * 2.0 ** -6
        w[1::2] *= -1
        W[:, 128 * j:128 * j + 128] = w
    a = wl.make_act_norms(wl.layer_seed("test", "build-edge", 0), K)
    for avg in (2, 3):
        for p in (0, 1, 2, 4):
            _check(W, a, avg, 128, p)
    buf = torch.empty(N * K + 8, dtype=torch.float16, device="cuda")
    off = buf[8:].view(N, K)
    off.copy_(torch.from_numpy(W))
    slim = _slim()
    A = slim.QuantLinear.from_weight(off, torch.from_numpy(a).cuda(), 2)
    B = _check(W, a, 2, 128)
    assert torch.equal(A.packed, B.packed) and torch.equal(A.scales, B.scales) and torch.equal(A.zeros, B.zeros)


def test_layer_from_weight_rejects_bad_arguments():
    slim = _slim()
    W, a = torch.zeros(32, 256, dtype=torch.float16, device="cuda"), torch.ones(256, device="cuda")
    for kw in (dict(avg_bits=4), dict(avg_bits=2, p=2), dict(avg_bits=2, g=96)):
        with pytest.raises(slim.SlimError):
            slim.QuantLinear.from_weight(W, a, **kw)
    L = slim.lib()
    pageable = np.zeros(2, dtype=np.uint8)
    t = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    args = (W.data_ptr(), a.data_ptr(), 2, -1, t.data_ptr(), t.data_ptr(), t.data_ptr(), pageable.ctypes.data, 32, 256, 128, t.data_ptr())
    assert L.slim_quantize_layer(*args, 4096, None) == -1          # the bit map has to go to page-locked memory
    assert L.slim_quantize_layer(*args, 64, None) == -4            # scratch too small

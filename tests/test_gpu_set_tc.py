"""GPU: the kernel for 2 to 64 tokens on raw codes (tcgen05, 8-bit floats), as a layer set and as one large layer, against the
oracle or an fp64 product with the dequantised weights."""
import numpy as np
import pytest
import torch

from oracle import slim_oracle as orc
from paper_2405_14917_b200 import binding as slim
from paper_2405_14917_b200 import workloads as wl
from tests.helpers import check_output, oracle_layer

pytestmark = pytest.mark.gpu


def _on_device(L):
    packed = torch.from_numpy(orc.pack(L["codes"], L["bits"])).cuda()
    return slim.QuantLinear(packed, L["bits"], torch.from_numpy(L["scales"]).cuda(), torch.from_numpy(L["zeros"]).cuda(), L["N"], L["K"])


def _quantised(N, K, avg, seed=0):
    W, a = wl.make_weight_and_norms_device((31, N, K + seed), N, K, "cuda")
    return slim.QuantLinear.from_weight(W, a, avg)


def _one_width(N, K, b):
    gen = torch.Generator(device="cuda").manual_seed(N + K + b)
    bits = np.full(K // 128, b, np.uint8)
    packed = torch.randint(0, 256, (slim.packed_bytes(N, K, bits),), dtype=torch.uint8, device="cuda", generator=gen)
    scales = (torch.rand((K // 128, N), device="cuda", generator=gen) * 0.02 + 0.01).half()
    return slim.QuantLinear(packed, bits, scales, torch.full_like(scales, (1 << b) // 2), N, K)


def _fp64(layer, x):
    What = slim.dequant(layer.packed, layer.bits, layer.scales, layer.zeros, layer.N, layer.K).double()
    return (x.double() @ What.T).cpu().numpy()


def _set(entries):
    s = slim.LayerSet(entries)
    s.run()
    s.check()
    return s


# every form (tokens rounded up to even, beyond 16 to a multiple of 8) with its last column used and not, and row blocks of one row tile, of one less and one more
# than a row of MMA tiles, and of more than 512 rows
@pytest.mark.parametrize("M", list(range(2, 17)) + [17, 24, 25, 32, 33, 40, 41, 48, 49, 56, 57, 64])
def test_every_form_on_ragged_row_blocks(M):
    layers = [oracle_layer(N, K, avg, m, block=i, seed_name="set-tc") for i, (N, K, avg, m) in enumerate(
        [(16, 128, 2, M), (112, 384, 3, max(1, M - 1)), (272, 256, 2, M), (528, 640, 3, 1), (1040, 128, 2, M)])]
    entries = [(_on_device(L), torch.from_numpy(L["x"]).cuda(), torch.full((L["M"], L["N"]), float("nan"), dtype=torch.float16, device="cuda")) for L in layers]
    s = _set(entries)
    assert s.info["tiles_per_warp"] == (4 if M <= 16 else 2)          # items of 512 or 256 rows
    for L, (_, _, y) in zip(layers, entries):
        check_output(y.cpu().numpy(), orc.linear_f64(L["x"], L["codes"], L["scales"], L["zeros"]), f"{L['N']}x{L['K']} M={L['M']} of {M}")


@pytest.mark.parametrize("M", [2, 9, 17, 33])
def test_each_bit_of_a_code_meets_its_activation(M):
    """One activation at a time: column k of the weights, exact up to the one rounding of the output."""
    bits = np.array([1, 2, 3, 4], dtype=np.uint8)
    L = oracle_layer(32, 512, 2, M, bits=bits, seed_name="set-tc-columns")
    What = orc.dequant_f64(L["codes"], L["scales"], L["zeros"])
    dl = _on_device(L)
    entries = []
    for k0 in range(0, 512, M):
        x = np.zeros((M, 512), np.float16)
        for m in range(M):
            x[m, (k0 + m) % 512] = 1.0
        entries.append((dl, torch.from_numpy(x).cuda(), torch.empty((M, 32), dtype=torch.float16, device="cuda")))
    _set(entries)
    for i, (_, _, y) in enumerate(entries):
        want = np.stack([What[:, (i * M + m) % 512] for m in range(M)]).astype(np.float16)
        assert (y.cpu().numpy().view(np.uint16) == want.view(np.uint16)).all(), i


def test_activations_of_any_size_are_taken_exactly():
    """Groups of x with sixteen exponents and of subnormals alone stay within the rounding of sums of 128 products (which x is taken exactly is tested
    above one activation at a time, and below); an infinity and a NaN spoil their token alone."""
    L = oracle_layer(16, 256, 2, 4, seed_name="set-tc-range")
    x = np.zeros((4, 256), np.float16)
    x[0, :128] = [(1 + (37 * i % 1024) / 1024) * 2.0 ** (i % 16 - 13) * (-1) ** i for i in range(128)]
    x[1, 130:140] = 6e-8 * np.arange(1, 11)                           # subnormals alone
    x[2, 5], x[3, 200] = np.inf, np.nan
    L["x"] = x
    y = torch.empty((4, 16), dtype=torch.float16, device="cuda")
    _set([(_on_device(L), torch.from_numpy(x).cuda(), y)])
    y = y.cpu().numpy().astype(np.float64)
    ref = orc.linear_f64(x[:2], L["codes"], L["scales"], L["zeros"])
    # one rounding to fp16 (a half unit, or half of the smallest subnormal) and fp32 sums of 128 products
    bound = 2.0 ** -11 * np.abs(ref) + 2.0 ** -25 + 2.0 ** -20 * np.abs(x[:2].astype(np.float64)).sum(axis=1)[:, None] * np.abs(orc.dequant_f64(L["codes"], L["scales"], L["zeros"])).max()
    assert (np.abs(y[:2] - ref) <= bound).all()
    assert np.isnan(y[2:]).all()


@pytest.mark.parametrize("M,avg", [(2, 2), (7, 3), (8, 3), (16, 2), (16, 3), (24, 3), (40, 2), (64, 3)])
def test_shares_that_end_inside_row_blocks_repeat_bit_for_bit(M, avg):
    """A set of more steps than four per CTA: equal shares, sums of cut row blocks added in the order of their parts.  A step read before it
    has landed, or sums added before they are written, would show as a run that differs."""
    entries = []
    for i, (N, K) in enumerate([(4096, 4096), (1040, 11008), (11008, 1024), (5120, 5120)]):
        layer = _quantised(N, K, avg, i)
        entries.append((layer, torch.randn((M, K), device="cuda").half(), torch.empty((M, N), dtype=torch.float16, device="cuda")))
    s = _set(entries)
    assert s.info["split"] > 1 and s.info["n_items"] > s.info["grid"]
    first = [y.clone() for (_, _, y) in entries]
    for (layer, x, _), y in zip(entries, first):
        check_output(y.cpu().numpy(), _fp64(layer, x), f"{layer.N}x{layer.K} M={M}")
    for _ in range(60):
        s.run()
        for (_, _, y), want in zip(entries, first):
            assert torch.equal(y, want)
    s.check()


@pytest.mark.parametrize("N,K,M,avg", [(14336, 8192, 2, 2), (14336, 8192, 8, 2), (26624, 4096, 5, 2), (16, 128, 2, 2), (28672, 8192, 16, 2), (8192, 28672, 13, 2), (14352, 8192, 9, 3),
                                       (14336, 8192, 18, 2), (8192, 14336, 32, 3), (28672, 8192, 40, 2), (24592, 8192, 56, 2)])
def test_one_large_layer_in_one_or_two_launches(N, K, M, avg):
    """Records of x in shared memory, or staged by a kernel ahead (many tokens and steps): the layer's own shares, twice into one workspace."""
    layer = _quantised(N, K, avg)
    x = torch.randn((M, K), device="cuda").half()
    ws = slim.new_workspace(M, N, K, layer.bits)
    y = layer.forward(x, ws)
    check_output(y.cpu().numpy(), _fp64(layer, x), f"{N}x{K} M={M}")
    for _ in range(40):
        assert torch.equal(layer.forward(x, ws), y)
    assert not ws[256:1280].any()                                     # the words that count the parts are zero again
    slim.workspace_status(ws)
    small = torch.zeros(256, dtype=torch.uint8, device="cuda")        # no room for parts: the other kernels
    check_output(layer.forward(x, small).cpu().numpy(), _fp64(layer, x), f"{N}x{K} M={M}, status word alone")


def test_a_kernel_ahead_that_outlasts_the_limit_of_the_waits():
    """A neighbour that lets the next kernel start at once and runs for longer than the two seconds that a wait of this library takes
    at most: its time is not this kernel's, whose ring is full until then."""
    hold = torch.cuda._compile_kernel("""extern "C" __global__ void hold(unsigned int us) {
        asm volatile("griddepcontrol.launch_dependents;");
        unsigned long long t0, t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
        for (int i = 0; i < 10000000; ++i) {
            __nanosleep(1000);
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
            if (t - t0 >= 1000ull * us) break;
        }
    }""", "hold")
    N, K, M = 26624, 4096, 5
    layer = _quantised(N, K, 2)
    assert 24 << 20 <= layer.packed.numel() < 32 << 20                # one launch that reads its slices ahead
    x = torch.randn((M, K), device="cuda").half()
    ws = slim.new_workspace(M, N, K, layer.bits)
    y = layer.forward(x, ws)
    out = torch.zeros_like(y)
    torch.cuda.synchronize()
    hold(grid=(1, 1, 1), block=(32, 1, 1), args=[2_500_000])
    layer.forward(x, ws, out)
    slim.workspace_status(ws)
    assert torch.equal(out, y)


@pytest.mark.parametrize("N,K,M,avg", [(131088, 1024, 2, 2), (131088, 1024, 9, 2), (152064, 2048, 16, 2), (65552, 2048, 20, 2), (131088, 2048, 40, 2)])
def test_one_large_layer_of_more_row_blocks_than_flags(N, K, M, avg):
    """An output head: the row blocks that are cut count their parts, of which there are fewer than shares."""
    layer = _quantised(N, K, avg)
    x = torch.randn((M, K), device="cuda").half()
    ws = slim.new_workspace(M, N, K, layer.bits)
    y = layer.forward(x, ws)
    check_output(y.cpu().numpy(), _fp64(layer, x), f"{N}x{K} M={M}")
    for _ in range(20):
        assert torch.equal(layer.forward(x, ws), y)
    assert not ws[256:1280].any()
    slim.workspace_status(ws)


# a megabyte less than the rule's 25, one row block of 512 fewer than its 6 and 8, and of 256 fewer than its 18 and 20; as many K-slices as leave gemv_few its shared memory
@pytest.mark.parametrize("N,K,M,avg", [(12288, 8192, 4, 2), (12288, 8192, 16, 2), (2560, 32768, 4, 3), (3584, 32768, 5, 2), (3584, 32768, 16, 0),
                                       (4352, 32768, 33, 3), (4864, 32768, 49, 3)])
def test_layers_that_other_kernels_are_sooner_at(N, K, M, avg):
    """Large layers of few row blocks, or little over 24 MB, take the kernels of a workspace without room for parts: the same bits.
    (0: two bits throughout, a K-slice per K-tile.)"""
    layer = _quantised(N, K, avg) if avg else _one_width(N, K, 2)
    x = torch.randn((M, K), device="cuda").half()
    size = slim.workspace_bytes(M, N, K, layer.bits)
    ws = slim.new_workspace(M, N, K, layer.bits)
    y = layer.forward(x, ws)
    check_output(y.cpu().numpy(), _fp64(layer, x), f"{N}x{K} M={M}")
    if M <= 16:
        assert torch.equal(layer.forward(x, torch.zeros(256, dtype=torch.uint8, device="cuda")), y)
    else:                                                             # no more than the batched kernel's flags and partial tiles
        assert size <= 1280 + 148 * 128 * 128 * 4
    slim.workspace_status(ws)


@pytest.mark.parametrize("N,K,M,avg", [(3072, 32768, 4, 3), (4096, 32768, 5, 2), (12288, 8192, 3, 2), (2304, 29184, 9, 3), (4608, 32768, 48, 3), (5120, 32768, 56, 3)])
def test_layers_of_few_row_blocks(N, K, M, avg):
    """The smallest layer and the fewest row blocks that the rule for large layers takes, and fewer of more K-slices: up to 15 parts to a row block."""
    layer = _quantised(N, K, avg)
    x = torch.randn((M, K), device="cuda").half()
    ws = slim.new_workspace(M, N, K, layer.bits)
    y = layer.forward(x, ws)
    check_output(y.cpu().numpy(), _fp64(layer, x), f"{N}x{K} M={M}")
    for _ in range(20):
        assert torch.equal(layer.forward(x, ws), y)
    assert ws[2048:].any() and not ws[256:1280].any()                 # parts were added through the workspace
    slim.workspace_status(ws)


@pytest.mark.parametrize("N,K,M,avg,share", [(28672, 4096, 6, 2, 0.94), (8192, 14336, 16, 3, 0.92), (65552, 2048, 24, 2, 0.95), (28672, 4096, 6, 2, 0.5), (8192, 24576, 56, 2, 0.93), (8192, 28672, 16, 2, 0.7)])
def test_a_workspace_short_of_a_few_parts(N, K, M, avg, share):
    """Fewer shares as long as that is a few, the other kernels in a workspace that is much smaller; nothing is written past its end."""
    layer = _quantised(N, K, avg)
    x = torch.randn((M, K), device="cuda").half()
    full = slim.workspace_bytes(M, N, K, layer.bits)
    buffer = torch.zeros(full, dtype=torch.uint8, device="cuda")
    size = int(share * (full - 1024)) // 16 * 16                      # (a thousand bytes less than asked for are as good)
    buffer[size:] = 7
    ws = buffer[:size]
    y = layer.forward(x, ws)
    check_output(y.cpu().numpy(), _fp64(layer, x), f"{N}x{K} M={M} in {share}")
    for _ in range(20):
        assert torch.equal(layer.forward(x, ws), y)
    assert (buffer[size:] == 7).all() and not ws[256:1280].any()
    slim.workspace_status(ws)


@pytest.mark.parametrize("N,K,M", [(28672, 8192, 24), (8192, 28672, 56), (38144, 16384, 56)])
def test_the_built_in_scratch_serves_large_layers_alike(N, K, M):
    """slim_mpq_gemm_static gives what slim_mpq_gemm gives in a workspace of the built-in scratch's size; all but the last ask for no more."""
    layer, size = _one_width(N, K, 2), 1280 + 148 * 256 * 128 * 4
    x = torch.randn((M, K), device="cuda").half()
    asked = slim.workspace_bytes(M, N, K, layer.bits)
    assert (asked - 1024 <= size) == (K != 16384)
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    y = layer.forward(x, ws)
    check_output(y[:, :512].cpu().numpy(), _fp64(layer, x)[:, :512], f"{N}x{K} M={M}")
    if asked <= size:
        assert torch.equal(layer.forward(x, slim.new_workspace(M, N, K, layer.bits)), y)
    out, status = torch.empty_like(y), torch.ones(1, dtype=torch.int32, device="cuda")
    for _ in range(3):
        slim.mpq_gemm_static(x, layer.packed, layer.bits, layer.scales, layer.zeros, N, out, status)
        assert torch.equal(out, y) and status.item() == 0


@pytest.mark.parametrize("M", [2, 7, 16, 17, 64])
@pytest.mark.parametrize("shapes,split", [([(4096, 4096)] * 3, None), ([(512, 28672)], 15), ([(1024, 8192), (16, 8192)], 8), ([(64, 1024)] * 16, 2), ([(1040, 2048)] * 6 + [(512, 128)], None)])
def test_small_sets_in_equal_parts(shapes, split, M):
    """A part of a row block per CTA, up to 15 of them: the sums are added in the order of the parts."""
    entries = []
    for i, (N, K) in enumerate(shapes):
        layer = _quantised(N, K, 2 + i % 2, i)
        entries.append((layer, torch.randn((M, K), device="cuda").half(), torch.empty((M, N), dtype=torch.float16, device="cuda")))
    s = _set(entries)
    assert s.info["n_items"] == s.info["grid"] <= torch.cuda.get_device_properties(0).multi_processor_count
    assert split is None or s.info["split"] == split
    first = [y.clone() for (_, _, y) in entries]
    for (layer, x, _), y in zip(entries, first):
        check_output(y.cpu().numpy(), _fp64(layer, x), f"{layer.N}x{layer.K} M={M}")
    for _ in range(20):
        s.run()
        for (_, _, y), want in zip(entries, first):
            assert torch.equal(y, want)
    s.check()


def _from_codes(codes, bits, scales, zeros):
    N, K = codes.shape
    packed = slim.pack_weights(torch.from_numpy(codes).cuda(), bits)
    return slim.QuantLinear(packed, bits, torch.from_numpy(scales).cuda(), torch.from_numpy(zeros).cuda(), N, K)


@pytest.mark.parametrize("M", list(range(2, 17, 2)) + list(range(24, 65, 8)))
def test_all_bits_of_an_activation_are_multiplied(M):
    """One activation at a time, of every exponent from -6 to 6 and a full significand of either sign, on every column: s (q - z) x up to the rounding to fp16
    (2^-11) and those of the two fp32 operations of the fold.  The third piece of x is up to 2^-8 of it, the second 2^-3."""
    L = oracle_layer(32, 512, 2, M, bits=np.array([1, 2, 3, 4], np.uint8), seed_name="set-tc-bits")
    What = orc.dequant_f64(L["codes"], L["scales"], L["zeros"])
    dl = _on_device(L)
    x = np.zeros((512 // M + 1, M, 512), np.float16)
    for i in range(x.shape[0]):
        for m in range(M):
            k = (i * M + m) % 512
            x[i, m, k] = (-1) ** (i + k) * (1 + (389 * k + 61 * m) % 1024 / 1024) * 2.0 ** ((i + 5 * m) % 13 - 6)
    entries = [(dl, torch.from_numpy(xi).cuda(), torch.empty((M, 32), dtype=torch.float16, device="cuda")) for xi in x]
    _set(entries)
    for xi, (_, _, y) in zip(x, entries):
        ref = xi.astype(np.float64) @ What.T
        assert (np.abs(y.cpu().numpy() - ref) <= 2.0 ** -11 * np.abs(ref) * (1 + 2.0 ** -9) + 2.0 ** -25).all()


@pytest.mark.parametrize("M", [4, 8, 12, 16, 24, 64])
@pytest.mark.parametrize("b", [1, 2, 3, 4])
def test_small_activations_beside_a_large_one(b, M):
    """A group whose largest activation meets a weight of exactly zero, and one other: exact down to 2^-(16 + b) of the largest, off by 2^-(27 + b) of it
    at most below."""
    rng = np.random.default_rng(10 * b + M)
    codes = rng.integers(1, 1 << b, (16, 128)).astype(np.uint8)
    codes[:, 77] = 0
    scales, zeros = np.full((1, 16), 1.0, np.float16), np.zeros((1, 16), np.float16)
    layer = _from_codes(codes, np.array([b], np.uint8), scales, zeros)
    large = 1.9990234375 * 2.0 ** 8
    entries, xs = [], []
    for i in range(0, 26 * 32, M):
        x = np.zeros((M, 128), np.float16)
        x[:, 77] = large if i % 2 else -1.0 * 2.0 ** 8                # the top and the bottom of a power of two
        for m in range(M):
            t, k = (i + m) % 26, (i + m) * 7 % 128
            if k != 77:
                x[m, k] = (-1) ** m * (1 + (331 * (i + m)) % 1024 / 1024) * 2.0 ** (8 - t)
        xs.append(x)
        entries.append((layer, torch.from_numpy(x).cuda(), torch.empty((M, 16), dtype=torch.float16, device="cuda")))
    _set(entries)
    for x, (_, _, y) in zip(xs, entries):
        small = x.astype(np.float64)
        top = np.abs(small).max(axis=1)[:, None]
        small[:, 77] = 0
        ref = small @ codes.astype(np.float64).T
        exact = np.abs(small).max(axis=1)[:, None] >= top * 2.0 ** -(16 + b)
        off = np.where(exact, 0.0, top * 2.0 ** -(27 + b) * codes.max())
        assert (np.abs(y.cpu().numpy() - ref) <= 2.0 ** -11 * np.abs(ref) * (1 + 2.0 ** -9) + 2.0 ** -25 + off).all()


@pytest.mark.parametrize("g,M", [(256, 2), (512, 8), (256, 16), (512, 24), (256, 40)])
def test_one_large_layer_of_wide_groups(g, M):
    """Two or four K-tiles that share a row of scales and zero points."""
    N, K = 24592, 8192
    W, a = wl.make_weight_and_norms_device((53, g, M), N, K, "cuda")
    layer = slim.QuantLinear.from_weight(W, a, 3 if M > 32 else 2, g=g)
    x = torch.randn((M, K), device="cuda").half()
    ws = slim.new_workspace(M, N, K, layer.bits, g=g)
    assert ws.numel() > 148 * M * (512 if M <= 16 else 256) * 4       # parts: the kernel for large layers
    y = layer.forward(x, ws)
    What = slim.dequant(layer.packed, layer.bits, layer.scales, layer.zeros, N, K, g=g).double()
    check_output(y.cpu().numpy(), (x.double() @ What.T).cpu().numpy(), f"{N}x{K} M={M} g={g}")
    slim.workspace_status(ws)

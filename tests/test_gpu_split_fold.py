"""The split fold: a layer whose workspace has room for the split-fold codes runs on one-limb weights (four of the factors of
H_raw folded into the weights, the others applied to the codes); the integers are the same sums, so its output is bit for bit
that of the same layer in a workspace of codes and scales alone, which runs on the two-limb weights.  The two-limb path is held
to the oracle by the other layer tests; here the split weights and codes are also checked against it through the product."""
import numpy as np
import pytest

from paper_2512_05746_b200 import inputs
from hq_testutil import decode_blob, weight_integers

CODE_BITS = [2, 3, 4, 1, 0]          # the index bits whose factors go to the codes, in this order


def hadamard_bits(n, mask):
    """The factors of the Hadamard matrix (Sylvester order) that belong to the index bits in `mask`."""
    i = np.arange(n)
    same = ((i[:, None] ^ i[None, :]) & ~mask) == 0
    par = np.array([bin(v).count("1") & 1 for v in range(n)])[(i[:, None] & i[None, :]) & mask]
    return np.where(same, 1 - 2 * par, 0).astype(np.int64)


@pytest.mark.parametrize("n", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("container", [0, 1])
def test_split_weights_times_split_codes_is_the_folded_product(n, container):
    from paper_2512_05746_b200 import binding as hq
    N, C, k = 130, 2 * n, n.bit_length() - 1
    pw = hq.hq_weight_prepare(inputs.weights((N, C), seed=n), 4, n, hq.HQ_W_FOLDED, container)
    d = pw.desc
    assert d.reserved == 1 and d.bytes == d.N_pad * d.C_pad * 3
    B = decode_blob(pw).reshape(N, C).astype(np.int64)
    B1 = pw.blob[d.N_pad * 2 * d.C_pad:].reshape(d.N_pad, d.C_pad)[:N, :C].astype(np.int64)
    mask = sum(1 << b for b in CODE_BITS[: k - 4])
    a_bits = 4 if k <= 8 else 3
    q = np.random.default_rng(n).integers(-(1 << (a_bits - 1)), 1 << (a_bits - 1), (64, C))
    z = q.reshape(64, -1, n) @ hadamard_bits(n, mask)
    assert np.abs(z + 0.5).max() < 128                         # fits a signed byte
    assert np.array_equal(z.reshape(64, C) @ B1.T, q @ B.T)
    # a blob buffer of the two-limb section alone is taken, and says that the other one is absent
    import ctypes
    blob, s_w, desc = np.zeros(d.N_pad * 2 * d.C_pad, np.int8), np.zeros(N, np.float32), hq.WeightDesc()
    w = np.ascontiguousarray(inputs.weights((N, C), seed=n), np.float32)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert hq.lib.hq_weight_prepare(ptr(w), N, 1, C, 4, n, hq.HQ_W_FOLDED, container, ptr(blob), blob.size, ptr(s_w),
                                    ctypes.byref(desc)) == 0
    assert desc.reserved == 0 and np.array_equal(blob, pw.blob[: blob.size])


def _codes_bytes(rows, cols, container):
    pitch = ((cols // 2 if container == 0 else cols) + 15) // 16 * 16
    return (rows * pitch + 255) // 256 * 256 + 4 * rows


def _both(torch, hq, rows, cols, container, call):
    """Outputs of the call in a workspace of codes and scales alone and in one with room for the split-fold codes, which must
    be written there (where the rule takes the one-limb product) and nothing behind them."""
    base = _codes_bytes(rows, cols, container)
    off = (base + 255) // 256 * 256
    full = off + rows * ((cols + 15) // 16 * 16)
    ws1 = torch.full((base,), 0x11, dtype=torch.uint8, device="cuda")
    ws2 = torch.full((full + 256,), 0x11, dtype=torch.uint8, device="cuda")
    y1, y2 = call(ws1), call(ws2[:full])
    torch.cuda.synchronize()
    assert torch.equal(ws1, ws2[:base])                         # the same codes and scales
    assert bool((ws2[full:] == 0x11).all())
    return y1, y2, ws2[off:full]


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,n,a_bits,dt,container,static", [
    (8192, 1152, 4608, 128, 4, "bf16", 1, False),      # nine blocks a row, streamed weights
    (20001, 512, 1288, 256, 4, "f32", 1, True),        # ragged rows and columns, resident weights; codes down to -8
    (16385, 96, 2056, 32, 4, "f32", 1, True),          # the smallest block, K not a multiple of 128
    (9000, 512, 2048, 512, 3, "f32", 0, True),         # the largest block, 3-bit codes down to -4, two codes per byte
    (9000, 192, 2048, 64, 4, "bf16", 0, False),
    (9000, 256, 2048, 256, 4, "bf16", 0, True),
])
def test_linear_on_one_limb_is_the_linear_on_two(M, K, N, n, a_bits, dt, container, static):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn((M, K), generator=gen, device="cuda")
    x[:, 3] *= 20
    if static:
        x[: M // 2] = x[: M // 2].abs() * torch.sign(torch.randn((1, K), generator=gen, device="cuda"))
    x = x if dt == "f32" else x.to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 4, n, hq.HQ_W_FOLDED, container).to_device()
    b = torch.from_numpy(inputs.bias(N, seed=3)).cuda()
    ss = torch.tensor([0.1], device="cuda") if static else None
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")

    def call(ws):
        y = torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
        hq.hq_qlinear(x, pw, b, a_bits, y, ws, static_scale=ss, dev_status=status)
        return y

    y1, y2, z = _both(torch, hq, M, K, container, call)
    hq.hq_check_status(status)
    assert torch.equal(y1, y2)
    assert not bool((z == 0x11).all()), "the layer was meant to run on one limb"
    # the split codes against the codes, on a few rows
    pitch = (K // 2 if container == 0 else K) // 1
    ws = torch.zeros((_codes_bytes(M, K, container),), dtype=torch.uint8, device="cuda")
    call(ws)
    pitch = (pitch + 15) // 16 * 16
    c = ws[: M * pitch].view(M, pitch)[:: max(1, M // 97)].cpu().numpy()
    if container == 0:
        q = np.stack([c & 15, c >> 4], axis=-1).reshape(c.shape[0], -1)[:, :K].astype(np.int64)
        q = np.where(q > 7, q - 16, q)
    else:
        q = c[:, :K].view(np.int8).astype(np.int64)
    if static:
        assert q.min() == -(1 << (a_bits - 1))
    mask = sum(1 << v for v in CODE_BITS[: n.bit_length() - 5])
    want = (q.reshape(q.shape[0], -1, n) @ hadamard_bits(n, mask)).reshape(q.shape[0], K)
    zp = (K + 15) // 16 * 16
    got = z.view(M, zp)[:: max(1, M // 97), :K].cpu().numpy().view(np.int8)
    assert np.array_equal(got, want)


@pytest.mark.gpu
@pytest.mark.parametrize("Nb,H,W,C,Cout,R,stride,container", [
    (64, 16, 16, 768, 768, 3, 1, 1),       # whole images per tile, six taps' K blocks odd in number per tap
    (19, 64, 64, 256, 512, 3, 2, 1),       # stride 2
    (40, 20, 24, 256, 520, 3, 1, 1),       # rows of a tile are not consecutive output rows: the general store path
    (33, 32, 32, 512, 1032, 1, 1, 0),      # 1x1, one scale per pixel, two codes per byte
])
def test_convolution_on_one_limb_is_the_convolution_on_two(Nb, H, W, C, Cout, R, stride, container):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randn((Nb, H, W, C), generator=gen, device="cuda").to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((Cout, R, R, C), seed=C), 4, 256, hq.HQ_W_FOLDED, container).to_device()
    b = torch.from_numpy(inputs.bias(Cout, seed=3)).cuda()
    ss = torch.tensor([0.4], device="cuda") if R == 3 else None
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    pad = R // 2

    def call(ws):
        y = torch.full((Nb, (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1, Cout), 7.0, dtype=torch.bfloat16,
                       device="cuda")
        hq.hq_qconv(x, pw, R, R, stride, pad, b, 4, y, ws, static_scale=ss, dev_status=status)
        return y

    y1, y2, z = _both(torch, hq, Nb * H * W, C, container, call)
    hq.hq_check_status(status)
    assert torch.equal(y1, y2)
    assert not bool((z == 0x11).all()), "the layer was meant to run on one limb"


@pytest.mark.gpu
@pytest.mark.parametrize("M", [3400, 7000, 7400])                  # 3.8, 7.7 and 8.2 MiB of codes and scales
@pytest.mark.parametrize("container", [0, 1])
def test_a_workspace_of_the_layer_query_takes_the_one_limb_route_at_any_size(M, container):
    import torch
    from paper_2512_05746_b200 import binding as hq
    K, N = 1152, 4608
    x = torch.randn((M, K), generator=torch.Generator(device="cuda").manual_seed(M), device="cuda").to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=1), 4, 128, hq.HQ_W_FOLDED, container).to_device()
    base, full = _codes_bytes(M, K, container), hq.hq_layer_workspace_size(pw, 4, M)
    assert full > base
    y = []
    for ws in (torch.full((full,), 0x11, dtype=torch.uint8, device="cuda"), torch.zeros((base,), dtype=torch.uint8, device="cuda")):
        y.append(torch.zeros((M, N), dtype=torch.bfloat16, device="cuda"))
        hq.hq_qlinear(x, pw, None, 4, y[-1], ws)
        assert ws.numel() == base or not bool((ws[(base + 255) // 256 * 256:] == 0x11).all())
    assert torch.equal(y[0], y[1])

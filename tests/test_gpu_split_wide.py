"""The split fold at blocks of 1024 to 4096 channels: four factors of H_raw go to the codes and the others stay with the weights,
as signed bytes where the integers fit and halved (with their common parities carried by further columns of the product) where
they do not.  The sums are the same integers, so a layer's output is bit for bit that of the same layer in a workspace of codes
and scales alone, which runs on the two-limb weights."""
import numpy as np
import pytest

import oracle
from paper_2512_05746_b200 import inputs
from hq_testutil import decode_blob
from test_gpu_split_fold import _both, _codes_bytes, hadamard_bits

CODE_MASK = 0b11110                  # channel bits 1 .. 4
HALVED = 128                         # bytes of further columns


def section(pw):
    """The one-limb section of a blob: its rows, the column parities (None: the integers themselves), or None without one."""
    d = pw.desc
    base, rows = d.N_pad * 2 * d.RS * d.C_pad, pw.blob
    more = int(d.bytes) - base
    if more == d.N_pad * d.RS * d.C_pad:
        return rows[base: base + more].reshape(d.N_pad, -1)[: d.N].astype(np.int64), None
    if more == d.N_pad * (d.C_pad + HALVED + 1):
        w = rows[base: base + d.N_pad * (d.C_pad + HALVED)].reshape(d.N_pad, -1)[: d.N].astype(np.int64)
        return w, rows[base + d.N_pad * (d.C_pad + HALVED): int(d.bytes)][: d.N].astype(np.int64)
    assert more == 0
    return None


def further_columns(q):
    """The bytes behind a row of split codes, from the row's codes (the statement of hq_fwht.cuh, in numpy)."""
    u = q.reshape(q.shape[0], -1, 16, 2).sum(axis=(1, 3))            # channel c belongs to sum (c >> 1) & 15
    h, U = (u + 8) >> 4, u.sum(axis=1)
    c1 = ((U >> 1) + 64) >> 7
    ext = np.zeros((q.shape[0], HALVED), np.int64)
    ext[:, :16], ext[:, 16:32] = h, u - 16 * h
    ext[:, 32] = ext[:, 33] = c1
    ext[:, 34], ext[:, 35] = (U >> 1) - 128 * c1, U & 1
    return ext


def layer_weights(N, n, kind):
    """`gaussian` as the other tests draw them; `wide`: a few quantized weights of seven in step, so that integers reach 8 bits
    and more; `top`: the largest there are, on one channel in all classes of equal sign."""
    w = inputs.weights((N, n), seed=n + N)
    if kind == "wide":
        w[::3, : n // 8] = np.abs(w[::3]).max(axis=1, keepdims=True)
    if kind == "top":
        w[1], w[2] = 1.0, -1.0
    return w


@pytest.mark.parametrize("n,kind,form", [(1024, "gaussian", "bytes"), (2048, "gaussian", None), (4096, "gaussian", "halved"),
                                         (1024, "wide", None), (2048, "wide", None), (4096, "top", "none")])
@pytest.mark.parametrize("container", [0, 1])
def test_wide_split_weights_times_split_codes_is_the_folded_product(n, kind, form, container):
    from paper_2512_05746_b200 import binding as hq
    N = 130
    pw = hq.hq_weight_prepare(layer_weights(N, n, kind), 4, n, hq.HQ_W_FOLDED, container)
    d = pw.desc
    assert d.reserved == 0 and d.bytes <= hq.hq_weight_blob_bytes(N, 1, n, 4, n, hq.HQ_W_FOLDED)
    sec = section(pw)
    # the two-limb section is what it is without the other, also where some of the weights keep the other away
    assert np.array_equal(decode_blob(pw).reshape(N, n), oracle.prepare_weights(layer_weights(N, n, kind), 4, n, "folded")[0].reshape(N, n))
    assert form is None or form == ("none" if sec is None else "bytes" if sec[1] is None else "halved")
    if sec is None:
        return
    B = decode_blob(pw).reshape(N, n).astype(np.int64)
    rng = np.random.default_rng(n)
    q = rng.integers(-8, 8, (64, n))
    q[0], q[1], q[2] = -8, 7, np.where(np.arange(n) & 2, -8, 7)
    z = q @ hadamard_bits(n, CODE_MASK)
    assert np.abs(z + 0.5).max() < 128
    if sec[1] is None:
        got = z @ sec[0].T
    else:
        ext = further_columns(q)
        assert ext.min() >= -128 and ext.max() <= 127
        got = 2 * (np.concatenate([z, ext], axis=1) @ sec[0].T) + ext[:, 35:36] * sec[1][None]
    assert np.array_equal(got, q @ B.T)
    # a buffer of the two-limb section alone is taken, and the descriptor then has no other
    import ctypes
    blob, s_w, desc = np.zeros(d.N_pad * 2 * d.C_pad, np.int8), np.zeros(N, np.float32), hq.WeightDesc()
    w = np.ascontiguousarray(layer_weights(N, n, kind), np.float32)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert hq.lib.hq_weight_prepare(ptr(w), N, 1, n, 4, n, hq.HQ_W_FOLDED, container, ptr(blob), blob.size, ptr(s_w),
                                    ctypes.byref(desc)) == 0
    assert desc.bytes == blob.size and np.array_equal(blob, pw.blob[: blob.size])


@pytest.mark.gpu
@pytest.mark.parametrize("M,n,N,a_bits,dt,container,static", [
    (9001, 1024, 2056, 4, "f32", 1, True),         # bytes; codes down to -8; ragged rows and columns
    (9000, 2048, 520, 3, "f32", 0, False),         # halved: one warp a row; two codes per byte
    (8001, 2048, 520, 4, "bf16", 1, True),
    (6000, 4096, 1032, 4, "bf16", 1, False),       # halved: two warps a row
    (4099, 4096, 1032, 4, "f32", 0, True),
    (16385, 4096, 1288, 3, "f32", 1, False),
])
def test_linear_on_wide_split_weights_is_the_linear_on_two_limbs(M, n, N, a_bits, dt, container, static):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(M + n)
    x = torch.randn((M, n), generator=gen, device="cuda")
    x[:, 3] *= 20
    if static:
        x[: M // 2] = x[: M // 2].abs() * torch.sign(torch.randn((1, n), generator=gen, device="cuda"))
        x[0], x[1] = -100.0, 100.0
    x = x if dt == "f32" else x.to(torch.bfloat16)
    w = layer_weights(N, n, "gaussian")
    if n == 2048:
        w[5, : n // 8] = np.abs(w[5]).max()        # integers beyond a byte: halved
    pw = hq.hq_weight_prepare(w, 4, n, hq.HQ_W_FOLDED, container)
    halved = section(pw)[1] is not None
    assert halved == (n > 1024)
    pw = pw.to_device()
    b = torch.from_numpy(inputs.bias(N, seed=3)).cuda()
    ss = torch.tensor([0.1], device="cuda") if static else None
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    base = _codes_bytes(M, n, container)
    off, pitch = (base + 255) // 256 * 256, n + (HALVED if halved else 0)
    full = off + M * pitch
    assert full <= hq.hq_workspace_size(M, n, container)

    def call(ws):
        y = torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
        hq.hq_qlinear(x, pw, b, a_bits, y, ws, static_scale=ss, dev_status=status)
        return y

    ws1 = torch.full((base,), 0x11, dtype=torch.uint8, device="cuda")
    ws2 = torch.full((full + 256,), 0x11, dtype=torch.uint8, device="cuda")
    y1, y2 = call(ws1), call(ws2[:full])
    torch.cuda.synchronize()
    hq.hq_check_status(status)
    assert torch.equal(ws1, ws2[:base]) and bool((ws2[full:] == 0x11).all())
    z = ws2[off:full].view(M, pitch)
    assert not bool((z == 0x11).all()), "the layer was meant to run on one limb"
    assert torch.equal(y1, y2)
    rows = slice(None, None, max(1, M // 97))
    cp = ((n // 2 if container == 0 else n) + 15) // 16 * 16
    c = ws1[: M * cp].view(M, cp)[rows].cpu().numpy()
    q = (np.stack([c & 15, c >> 4], axis=-1).reshape(c.shape[0], -1) if container == 0 else c.view(np.int8)).astype(np.int64)
    q = np.where(q > 7, q - 16, q)
    if static:
        assert q.min() == -(1 << (a_bits - 1))
    want = q @ hadamard_bits(n, CODE_MASK)
    if halved:
        want = np.concatenate([want, further_columns(q)], axis=1)
    assert np.array_equal(z[rows].cpu().numpy().view(np.int8), want)
    # fp32 outputs are not the pair kernel's: the call runs, on whichever weights, with the same sums
    yf = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    hq.hq_qlinear(x, pw, b, a_bits, yf, ws2[:full], static_scale=ss, dev_status=status)
    assert torch.equal(yf.to(torch.bfloat16), y1)


@pytest.mark.gpu
@pytest.mark.parametrize("M,n,N,container,taken", [
    (16384, 4096, 512, 1, False),       # two limbs / one: 103.5 / 108.5 us
    (32768, 4096, 512, 1, False),       # 194 / 204.5
    (16384, 4096, 1024, 1, True),
    (16384, 4096, 512, 0, True),        # 105.4 / 102.1
    (32768, 2048, 512, 1, False),       # 95.5 / 99.0
    (32768, 2048, 768, 1, True),        # 114.6 / 109
])
def test_one_limb_only_where_it_is_the_faster(M, n, N, container, taken):
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(layer_weights(N, n, "gaussian"), 4, n, hq.HQ_W_FOLDED, container)
    assert section(pw) is not None
    pw = pw.to_device()
    x = torch.randn((M, n), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda").to(torch.bfloat16)
    ws = torch.full((hq.hq_workspace_size(M, n, container),), 0x11, dtype=torch.uint8, device="cuda")
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    hq.hq_qlinear(x, pw, None, 4, y, ws)
    behind = ws[(_codes_bytes(M, n, container) + 255) // 256 * 256:]
    assert bool((behind[:n] != 0x11).any()) == taken

"""Fused layers with a residual connection: the sum is bit for bit that of hq_add on the layer's own output, whichever kernel runs
the product (a reduction divided over a cluster, streamed weights on pairs of SMs, and those that leave the addition to a launch
of its own)."""
import ctypes as C

import pytest

from paper_2512_05746_b200 import inputs


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,n,room", [
    (2, 1024, 1024, 256, False),        # divided eight ways, 16 columns a CTA; two rows of a tile
    (130, 768, 264, 256, False),        # ragged rows and columns, divided
    (200, 1024, 512, 256, False),       # two rows of tiles
    (4096, 1024, 1024, 256, True),      # pairs of SMs, one limb
    (1001, 2304, 1160, 256, True),      # ... rows of the last tile missing, a column tile cut off inside a 32-column store
    (16385, 768, 200, 256, True),       # ... one column tile, cut off inside a store
    (16001, 640, 1288, 128, True),      # ... tiles of 192 columns, six a pair
    (5000, 1024, 776, 256, False),      # ... two limbs
    (4096, 512, 512, 256, True),        # ... four K blocks, which a layer without a residual runs on one CTA
    (1001, 512, 200, 256, True),
    (9500, 512, 512, 256, True),        # ... beyond one round of tiles: a launch of its own, behind the one-CTA kernel that keeps the weights
    (20000, 256, 264, 256, True),       # two K blocks: likewise
    (6000, 512, 776, 512, False),       # two limbs, weights kept by pairs of SMs (168 tiles): likewise
    (8200, 2048, 520, 2048, True),      # halved weights: likewise
])
def test_linear_with_a_residual_is_the_linear_and_an_addition(M, K, N, n, room):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(M + K + N)
    x = torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16)
    r = (3 * torch.randn((M, N), generator=gen, device="cuda")).to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 4, n, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device()
    b = torch.from_numpy(inputs.bias(N, seed=3)).cuda()
    codes = (M * K + 255) // 256 * 256 + 4 * M
    ws = torch.zeros((max(codes, hq.hq_layer_workspace_size(pw, 4, M), hq.hq_workspace_size(M, K, 1)) if room else codes,),
                     dtype=torch.uint8, device="cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    y, want = (torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    guard = torch.full((M * N + 1024,), 7.0, dtype=torch.bfloat16, device="cuda")
    got = guard[512: 512 + M * N].view(M, N)
    hq.hq_qlinear(x, pw, b, 4, y, ws, dev_status=status)
    hq.hq_add(y.view(-1), r.view(-1), want.view(-1))
    hq.hq_qlinear(x, pw, b, 4, got, ws, dev_status=status, residual=r)
    torch.cuda.synchronize()
    hq.hq_check_status(status)
    assert torch.equal(got, want)
    assert bool((guard[:512] == 7).all()) and bool((guard[512 + M * N:] == 7).all())


@pytest.mark.gpu
@pytest.mark.parametrize("Nb,H,W,Cin,Cout,stride,static", [
    (2, 8, 8, 2048, 1024, 1, True),     # divided eight ways
    (3, 16, 16, 768, 776, 1, True),
    (5, 32, 32, 512, 512, 1, True),     # pairs of SMs; an odd number of row tiles
    (40, 32, 32, 256, 264, 1, True),
    (7, 64, 64, 256, 256, 2, True),
    (2, 20, 24, 256, 520, 1, True),     # rows of a tile are not consecutive output rows: a launch of its own
    (2, 16, 16, 256, 256, 1, False),    # one scale per pixel under the window: likewise
])
def test_convolution_with_a_residual_is_the_convolution_and_an_addition(Nb, H, W, Cin, Cout, stride, static):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(Cin + Nb)
    x = torch.randn((Nb, H, W, Cin), generator=gen, device="cuda").to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((Cout, 3, 3, Cin), seed=Cin), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device()
    b = torch.from_numpy(inputs.bias(Cout, seed=3)).cuda()
    g, bt = torch.ones(Cin, device="cuda"), torch.zeros(Cin, device="cuda")
    shape = (Nb, H // stride, W // stride, Cout)
    r = (3 * torch.randn(shape, generator=gen, device="cuda")).to(torch.bfloat16)
    ws = torch.zeros((max(hq.hq_layer_workspace_size(pw, 4, Nb * H * W, static, stride), hq.hq_workspace_size(Nb * H * W, Cin, 1)),),
                     dtype=torch.uint8, device="cuda")
    scr = torch.zeros((Nb * 32 * 24,), dtype=torch.uint8, device="cuda")
    ss = torch.tensor([0.3], device="cuda") if static else None
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    y, got = (torch.empty(shape, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    args = (x, 32, g, bt, 1e-5, pw, 3, 3, stride, 1, b, 4)
    hq.hq_gn_silu_qconv(*args, y, ws, scr, static_scale=ss, dev_status=status)
    want = torch.empty_like(y)
    hq.hq_add(y.view(-1), r.view(-1), want.view(-1))
    hq.hq_gn_silu_qconv(*args, got, ws, scr, static_scale=ss, dev_status=status, residual=r)
    torch.cuda.synchronize()
    hq.hq_check_status(status)
    assert torch.equal(got, want)


def test_residuals_that_cannot_be_added_are_refused_before_a_launch():
    from paper_2512_05746_b200 import binding as hq
    L, big = hq.lib, 1 << 30
    p = lambda v: C.c_void_p(v)
    odd = hq.hq_weight_prepare(inputs.weights((36, 256), seed=1), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)
    lin = hq.hq_weight_prepare(inputs.weights((64, 256), seed=1), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)

    def call(pw, residual, y):
        return L.hq_qlinear_add(p(0x1000), 1, 64, 256, 256, C.byref(pw.desc), p(0x1000), p(0x1000), None, 4, residual, y, p(0x1000),
                                big, None, None)
    assert call(lin, None, p(0x2000)) == 1
    assert call(lin, p(0x2000), p(0x2000)) == 1                       # the output itself
    assert call(odd, p(0x3000), p(0x2000)) == 2                       # 36 columns
    assert call(lin, p(0x3008), p(0x2000)) == 4
    assert call(lin, p(0x3000), p(0x2008)) == 4


def test_a_residual_of_another_type_or_shape_is_refused():
    import torch
    from paper_2512_05746_b200 import binding as hq
    lin = hq.hq_weight_prepare(inputs.weights((64, 256), seed=1), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device("cpu")
    conv = hq.hq_weight_prepare(inputs.weights((64, 3, 3, 256), seed=1), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device("cpu")
    x, px = torch.zeros((8, 256)), torch.zeros((1, 4, 4, 256))
    g, ws, scr = torch.zeros(256), torch.zeros(1 << 16, dtype=torch.uint8), torch.zeros(1 << 10, dtype=torch.uint8)

    class Stream:
        cuda_stream = 0

    def both(error, y, residual):
        with pytest.raises(error):
            hq.hq_qlinear(x, lin, None, 4, y, ws, residual=residual, stream=Stream)
        with pytest.raises(error):
            hq.hq_gn_silu_qconv(px, 32, g, g, 1e-5, conv, 3, 3, 1, 1, None, 4, y.view(1, -1, 4, y.shape[-1]), ws, scr, stream=Stream,
                                residual=residual.view(1, -1, 4, residual.shape[-1]))
    both(TypeError, *(torch.zeros((8, 64), dtype=torch.float16) for _ in range(2)))
    both(TypeError, *(torch.zeros((8, 64), dtype=torch.int16) for _ in range(2)))
    both(ValueError, *(torch.zeros((8, 64)) for _ in range(2)))
    both(ValueError, torch.zeros((8, 64), dtype=torch.bfloat16), torch.zeros((8, 64)))
    both(ValueError, *(torch.zeros((8, 72), dtype=torch.bfloat16) for _ in range(2)))        # rows longer than the layer's
    both(ValueError, torch.zeros((8, 64), dtype=torch.bfloat16), torch.zeros((4, 64), dtype=torch.bfloat16))


@pytest.mark.gpu
@pytest.mark.parametrize("Nb,H,W,Cin,Cout", [
    (3, 16, 16, 768, 776),              # statistics by runs of groups
    (7, 32, 32, 512, 512),
    (1, 256, 256, 256, 256),            # one wave over the pixels
])
def test_an_addend_with_a_pitch_of_its_own_is_its_dense_copy(Nb, H, W, Cin, Cout):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(Cin + Nb)
    x = torch.randn((Nb, H, W, Cin), generator=gen, device="cuda").to(torch.bfloat16)
    wide = (2 * torch.randn((Nb, 3 * Cin + 128), generator=gen, device="cuda")).to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((Cout, 3, 3, Cin), seed=Cin), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device()
    g, bt = torch.ones(Cin, device="cuda"), torch.zeros(Cin, device="cuda")
    r = (3 * torch.randn((Nb, H, W, Cout), generator=gen, device="cuda")).to(torch.bfloat16)
    ws = torch.zeros((hq.hq_workspace_size(Nb * H * W, Cin, 1),), dtype=torch.uint8, device="cuda")
    scr, ss = torch.zeros((Nb * 32 * 24,), dtype=torch.uint8, device="cuda"), torch.tensor([0.3], device="cuda")

    def call(e, residual):
        y = torch.zeros((Nb, H, W, Cout), dtype=torch.bfloat16, device="cuda")
        hq.hq_gn_silu_qconv(x, 32, g, bt, 1e-5, pw, 3, 3, 1, 1, None, 4, y, ws, scr, static_scale=ss, pre_bias=e, residual=residual)
        return y
    sliced = wide[:, Cin + 64: 2 * Cin + 64]
    want = torch.empty_like(r)
    hq.hq_add(call(sliced.contiguous(), None).view(-1), r.view(-1), want.view(-1))
    assert torch.equal(call(sliced, r), want) and torch.equal(call(sliced.contiguous(), r), want)


def test_an_addend_that_cannot_be_read_is_refused():
    """The calls without a pitch for it (no residual; codes alone; two inputs) would take its rows from the wrong places."""
    import torch
    from paper_2512_05746_b200 import binding as hq
    conv = hq.hq_weight_prepare(inputs.weights((64, 3, 3, 256), seed=1), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device("cpu")
    x, half = torch.zeros((2, 4, 4, 256)), torch.zeros((2, 4, 4, 128))
    g, ws, scr = torch.zeros(256), torch.zeros(1 << 16, dtype=torch.uint8), torch.zeros(1 << 10, dtype=torch.uint8)
    y, r = (torch.zeros((2, 4, 4, 64), dtype=torch.bfloat16) for _ in range(2))
    codes, sc = torch.zeros((32, 256), dtype=torch.uint8), torch.zeros(32)
    wide = torch.zeros((2, 512), dtype=torch.bfloat16)

    class Stream:
        cuda_stream = 0

    def conv_call(e, xs=(x, None), residual=None):
        hq.hq_gn_silu_qconv(xs[0], 32, g, g, 1e-5, conv, 3, 3, 1, 1, None, 4, y, ws, scr, stream=Stream, pre_bias=e, x2=xs[1], residual=residual)
    for e in (wide[:, :256], wide[:, ::2], wide.view(4, 256)[::2], wide[:1, :256].expand(2, 256)):
        with pytest.raises(ValueError):
            conv_call(e)
        with pytest.raises(ValueError):
            conv_call(e, (half, half))
        with pytest.raises(ValueError):
            hq.hq_gn_silu_quant(x, 32, g, g, 1e-5, 256, 4, codes, 1, scr, scales=sc, pre_bias=e, stream=Stream)
    with pytest.raises(ValueError):
        conv_call(wide[:, ::2], residual=r)


@pytest.mark.gpu
@pytest.mark.parametrize("stride", [0, 3, -1])
@pytest.mark.parametrize("with_residual", [False, True])
def test_a_stride_that_is_refused_is_refused(stride, with_residual):
    """The size of the output is worked out for the residual: not from a stride that the product has refused."""
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(inputs.weights((64, 3, 3, 256), seed=1), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device()
    x = torch.zeros((1, 8, 8, 256), dtype=torch.bfloat16, device="cuda")
    y, r = (torch.full((1, 8, 8, 64), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    g, ws = torch.ones(256, device="cuda"), torch.zeros((hq.hq_workspace_size(64, 256, 1),), dtype=torch.uint8, device="cuda")
    scr = torch.zeros((32 * 24,), dtype=torch.uint8, device="cuda")
    with pytest.raises(hq.HqError) as e:
        hq.hq_gn_silu_qconv(x, 32, g, g, 1e-5, pw, 3, 3, stride, 1, None, 4, y, ws, scr, static_scale=torch.tensor([0.3], device="cuda"),
                            residual=r if with_residual else None)
    assert e.value.status == 3 and bool((y == 7).all())

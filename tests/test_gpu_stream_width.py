"""Narrower column tiles of the streamed pair kernel (one weight limb, 192 or 128 operand rows per tile): bit for bit the one-CTA
kernel's output, at column counts that end inside a tile, at one and two K blocks per ring stage and for a convolution."""
import pytest

from paper_2512_05746_b200 import inputs
from test_gpu_splitk import both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [
    (16001, 1024, 1288),      # 192 wide, one K block per stage, ragged rows and columns
    (4096, 2048, 264),        # 128 wide, two K blocks per stage
    (4096, 1152, 264),        # 128 wide, an odd number of K blocks
    (5000, 4096, 520),        # 192 wide, two K blocks per stage
    (20000, 1280, 136),       # 192 wide, as many tiles as 256 wide ones
    (8192, 4608, 1152),       # 192 wide, whole tiles
    (53000, 512, 1288),       # four K blocks: the one-CTA kernel's weights stay in its shared memory up to 1024 tiles
])
def test_linear_on_narrow_tiles(M, K, N):
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 8, 128, hq.HQ_W_DOUBLE, hq.HQ_CODES_INT8).to_device()
    gen = torch.Generator(device="cuda").manual_seed(K)
    q = torch.randint(-128, 128, (M, K), generator=gen, device="cuda", dtype=torch.int8).view(torch.uint8)
    sa = torch.rand((M,), generator=gen, device="cuda") + 0.5
    b = torch.from_numpy(inputs.bias(N, seed=1)).cuda()
    both(torch, hq, lambda y, st: hq.hq_qgemm(q, hq.HQ_CODES_INT8, 8, K, pw, scale_a=sa, bias=b, y=y, dev_status=st), (M, N))


@pytest.mark.parametrize("Nb,H,C,Cout", [(16, 16, 768, 768), (40, 32, 256, 136), (9, 32, 640, 264)])
def test_convolution_on_narrow_tiles(Nb, H, C, Cout):
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(inputs.weights((Cout, 3, 3, C), seed=C), 4, 128, hq.HQ_W_PLAIN, hq.HQ_CODES_INT8).to_device()
    gen = torch.Generator(device="cuda").manual_seed(C)
    q = torch.randint(-128, 128, (Nb, H, H, C), generator=gen, device="cuda", dtype=torch.int8).view(torch.uint8)
    sa, b = torch.rand((1,), generator=gen, device="cuda") + 0.5, torch.from_numpy(inputs.bias(Cout, seed=1)).cuda()
    both(torch, hq, lambda y, st: hq.hq_qconv2d(q, hq.HQ_CODES_INT8, 8, Nb, H, H, C, pw, 3, 3, 1, 1, scale_a=sa, bias=b, y=y,
                                                dev_status=st), (Nb, H, H, Cout))


@pytest.mark.parametrize("M,K,N", [
    (16001, 640, 1288),       # 192 wide, six tiles a pair, five K blocks
    (16001, 1152, 1288),      # ... nine
    (50000, 640, 136),        # one column tile cut off inside a store, two to three tiles a pair
])
def test_narrow_tiles_one_after_the_other_keep_their_staging_apart(M, K, N):
    # three stores a tile and two staging buffers: the turn passes from tile to tile, and every pass gives the same bytes
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 8, 128, hq.HQ_W_DOUBLE, hq.HQ_CODES_INT8).to_device()
    gen = torch.Generator(device="cuda").manual_seed(K)
    q = torch.randint(-128, 128, (M, K), generator=gen, device="cuda", dtype=torch.int8).view(torch.uint8)
    sa = torch.rand((M,), generator=gen, device="cuda") + 0.5
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    ys = [torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(13)]
    hq.hq_set_pair_gemm(0)
    try:
        hq.hq_qgemm(q, hq.HQ_CODES_INT8, 8, K, pw, scale_a=sa, y=ys[0], dev_status=status)
    finally:
        hq.hq_set_pair_gemm(2)
    for y in ys[1:]:
        hq.hq_qgemm(q, hq.HQ_CODES_INT8, 8, K, pw, scale_a=sa, y=y, dev_status=status)
    assert int(status) == 0
    for y in ys[1:]:
        assert torch.equal(y, ys[0])


@pytest.mark.parametrize("Nb,H,W,C,Cout,stride,mode", [
    (8, 32, 32, 256, 256, 1, "folded"),      # two limbs, two K blocks a stage, one wave
    (5, 32, 32, 384, 264, 1, "folded"),      # ... three K blocks a tap, an odd number of row tiles, a column tile cut off
    (7, 16, 16, 256, 136, 2, "plain"),       # one limb, stride 2, two images a tile and one missing
    (40, 16, 16, 512, 520, 1, "plain"),      # ... several tiles a pair
    (3, 12, 16, 256, 136, 1, "folded"),      # tiles of 8 rows: four of the second tile lie below the image
    (3, 12, 16, 256, 264, 1, "plain"),
    (1, 6, 160, 256, 136, 1, "folded"),      # tiles of 128 pixels of a row: 96 of the second lie past it
    (1, 6, 160, 384, 264, 1, "plain"),
    (2, 24, 32, 256, 136, 2, "folded"),      # 12 x 16 outputs at stride 2
    (2, 6, 320, 256, 264, 2, "plain"),       # 3 x 160
])
@pytest.mark.parametrize("f32", [False, True])
def test_per_pixel_scales_on_pairs(Nb, H, W, C, Cout, stride, mode, f32):
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(inputs.weights((Cout, 3, 3, C), seed=C), 4, 128, hq.WEIGHT_MODES[mode], hq.HQ_CODES_INT8).to_device()
    gen = torch.Generator(device="cuda").manual_seed(C)
    q = torch.randint(-8, 8, (Nb, H, W, C), generator=gen, device="cuda", dtype=torch.int8).view(torch.uint8)
    sa = torch.rand((Nb * H * W,), generator=gen, device="cuda") + 0.5
    b = torch.from_numpy(inputs.bias(Cout, seed=1)).cuda()
    out = []
    for pair in (0, 2):
        n = Nb * (H // stride) * (W // stride) * Cout
        guard = torch.full((n + 1024,), 7.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
        y = guard[512: 512 + n].view(Nb, H // stride, W // stride, Cout)
        status = torch.zeros((1,), dtype=torch.int32, device="cuda")
        before = hq.hq_set_pair_gemm(pair)
        try:
            hq.hq_qconv2d(q, hq.HQ_CODES_INT8, 4, Nb, H, W, C, pw, 3, 3, stride, 1, scale_a=sa, bias=b, y=y, dev_status=status)
        finally:
            hq.hq_set_pair_gemm(before)
        assert int(status) == 0
        assert bool((guard[:512] == 7).all()) and bool((guard[512 + n:] == 7).all())
        out.append(y)
    assert torch.equal(out[0], out[1])

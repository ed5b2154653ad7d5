"""Products of few tiles, whose reduction the default dispatch divides over the CTAs of a cluster: the sums are integers, so the
output is bit for bit that of the one-CTA kernel (`hq_set_pair_gemm(0)`), which the other tests hold to the oracle.  Sizes at the
edges of tiles (rows and columns that end inside one, a tile of fewer rows than 128), of the shares (K blocks that 2, 4 and 8
do not divide) and at the largest number of tiles that still divides."""
import numpy as np
import pytest

from paper_2512_05746_b200 import inputs

pytestmark = pytest.mark.gpu


def both(torch, hq, call, shape):
    y = [torch.full(shape, 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    call(y[0], status)
    before = hq.hq_set_pair_gemm(0)
    try:
        call(y[1], status)
    finally:
        hq.hq_set_pair_gemm(before)
    torch.cuda.synchronize()
    hq.hq_check_status(status)
    assert torch.equal(y[0], y[1])
    assert float((y[0] == 7.0).float().mean()) < 0.5


@pytest.mark.parametrize("M,K,N,mode,scalar", [
    (1, 1024, 1024, "folded", False),      # one row, one K block per CTA of eight
    (2, 4608, 1152, "folded", True),       # 36 K blocks over eight: shares of four and five
    (127, 2048, 136, "plain", False),      # one limb, columns end inside a tile
    (129, 1408, 264, "folded", False),     # eleven K blocks, a second row tile of one row
    (256, 4608, 1152, "folded", False),    # four ways
    (2000, 4096, 200, "plain", False),     # two ways, ragged rows, columns not a multiple of 128
    (64, 5000, 130, "folded", False),      # a reduction that ends inside a K block, output rows that 16-byte stores cannot take
])
def test_linear_divided_over_a_cluster(M, K, N, mode, scalar):
    import torch
    from paper_2512_05746_b200 import binding as hq
    n = 8 if K % 128 else 128
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 4, n, hq.WEIGHT_MODES[mode], hq.HQ_CODES_INT8).to_device()
    gen = torch.Generator(device="cuda").manual_seed(K)
    ld = (K + 15) // 16 * 16
    q = torch.randint(-8, 8, (M, ld), generator=gen, device="cuda", dtype=torch.int8).view(torch.uint8)
    sa = torch.rand((1 if scalar else M,), generator=gen, device="cuda") + 0.5
    b = torch.from_numpy(inputs.bias(N, seed=1)).cuda()
    both(torch, hq, lambda y, st: hq.hq_qgemm(q, hq.HQ_CODES_INT8, 4, K, pw, scale_a=sa, bias=b, alpha=pw.alpha, y=y, dev_status=st),
         (M, N))


@pytest.mark.parametrize("Nb,H,W,C,Cout,R,stride,mode", [
    (1, 8, 8, 1024, 1024, 3, 1, "folded"),     # a tile of 64 pixels
    (2, 8, 8, 2048, 1024, 3, 1, "folded"),     # 144 K blocks, 64 CTAs
    (3, 8, 8, 512, 264, 3, 1, "plain"),        # the last tile holds one of two images
    (2, 16, 16, 768, 768, 3, 2, "folded"),     # stride 2
    (1, 32, 32, 512, 512, 3, 1, "folded"),     # several tiles per image
    (2, 16, 16, 1536, 768, 1, 1, "folded"),    # 1x1, one scale per pixel
    (5, 4, 4, 1024, 96, 3, 1, "plain"),        # eight images per tile, fewer exist
    (1, 6, 10, 640, 128, 3, 1, "folded"),      # a tile of 60 pixels
])
def test_convolution_divided_over_a_cluster(Nb, H, W, C, Cout, R, stride, mode):
    import torch
    from paper_2512_05746_b200 import binding as hq
    pw = hq.hq_weight_prepare(inputs.weights((Cout, R, R, C), seed=C), 4, 128, hq.WEIGHT_MODES[mode], hq.HQ_CODES_INT8).to_device()
    gen = torch.Generator(device="cuda").manual_seed(C)
    q = torch.randint(-8, 8, (Nb, H, W, C), generator=gen, device="cuda", dtype=torch.int8).view(torch.uint8)
    sa = torch.rand((1 if R == 3 else Nb * H * W,), generator=gen, device="cuda") + 0.5
    b = torch.from_numpy(inputs.bias(Cout, seed=1)).cuda()
    pad = R // 2
    both(torch, hq, lambda y, st: hq.hq_qconv2d(q, hq.HQ_CODES_INT8, 4, Nb, H, W, C, pw, R, R, stride, pad, scale_a=sa, bias=b,
                                                alpha=pw.alpha, y=y, dev_status=st),
         (Nb, (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1, Cout))

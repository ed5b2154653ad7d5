"""Linear layers of few rows run as one kernel: codes, scales and outputs are, bit for bit, those of the two kernels (which another
kernel choice brings back), in the workspace and the output and nowhere beside them."""
import numpy as np
import pytest

from paper_2512_05746_b200 import inputs


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,n,mode,w_bits,a_bits,dt,static,bias", [
    (256, 256, 256, 256, "folded", 4, 4, "f32", False, True),      # two limbs
    (1, 128, 2, 32, "folded", 4, 3, "bf16", False, False),         # one row, one pair of columns, the shortest reduction
    (17, 768, 130, 256, "folded", 4, 4, "bf16", True, True),       # 24 threads a row; a row tile and a column tile nearly empty
    (48, 1024, 200, 512, "folded", 4, 4, "f32", False, True),      # the longest reduction on two limbs: the shared memory is full
    (300, 512, 384, 128, "double", 4, 4, "f32", True, False),      # one limb; codes down to -8
    (33, 640, 1000, 128, "double", 8, 8, "bf16", False, True),     # eight bits a side
    (590, 384, 250, 64, "plain", 4, 4, "bf16", False, True),       # as many CTAs as there are SMs
    (64, 896, 64, 32, "folded", 4, 8, "f32", False, True),
    (520, 256, 640, 256, "folded", 4, 4, "bf16", False, True),     # more CTAs than SMs, all resident at once
])
def test_one_kernel_is_two(M, K, N, n, mode, w_bits, a_bits, dt, static, bias):
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(M + K + N)
    xs = torch.randn((M, K + 16), generator=gen, device="cuda") * 3
    xs[:, 7] *= 20
    if static:
        xs[0] = -100.0
    if M > 2:
        xs[1] = 0
    x = (xs if dt == "f32" else xs.to(torch.bfloat16))[:, 8:8 + K]
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), w_bits, n, hq.WEIGHT_MODES[mode], hq.HQ_CODES_INT8).to_device()
    b = torch.from_numpy(inputs.bias(N, seed=3)).cuda() if bias else None
    ss = torch.tensor([0.4], device="cuda") if static else None
    need = (M * K + 255) // 256 * 256 + 4 * M

    def call():
        ws = torch.full((need + 256,), 0x11, dtype=torch.uint8, device="cuda")
        y = torch.full((M + 2, N + 6), 7.0, dtype=torch.bfloat16, device="cuda")
        for _ in range(3):                                         # one behind the other in buffers of their own and the same
            hq.hq_qlinear(x, pw, b, a_bits, y[1:-1, 2:2 + N], ws[:need], static_scale=ss)
        torch.cuda.synchronize()
        return ws, y

    ws, y = call()
    before = hq.hq_set_pair_gemm(0)
    try:
        ws2, y2 = call()
    finally:
        hq.hq_set_pair_gemm(before)
    assert torch.equal(ws, ws2) and torch.equal(y, y2)
    assert bool((y[0] == 7).all()) and bool((y[:, :2] == 7).all()) and bool((y[:, 2 + N:] == 7).all())
    assert np.abs(y[1:-1, 2:2 + N].float().cpu().numpy()).max() > 0


@pytest.mark.gpu
def test_output_over_the_input():
    """The two kernels take an output on top of their input; the one kernel, whose CTAs read while others write, leaves it to them."""
    import torch
    from paper_2512_05746_b200 import binding as hq
    M = K = N = 256
    x = torch.randn((M, K), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda").to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 4, 256, hq.WEIGHT_MODES["folded"], hq.HQ_CODES_INT8).to_device()
    ws = torch.empty((hq.hq_workspace_size(M, K, hq.HQ_CODES_INT8),), dtype=torch.uint8, device="cuda")
    want = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    hq.hq_qlinear(x, pw, None, 4, want, ws)
    for _ in range(5):
        y = x.clone()
        hq.hq_qlinear(y, pw, None, 4, y, ws)
        assert torch.equal(y, want)


@pytest.mark.gpu
def test_output_over_the_static_scale():
    """Likewise an output on top of the static scale, which the first of the two kernels has copied by then."""
    import torch
    from paper_2512_05746_b200 import binding as hq
    M = K = N = 256
    x = torch.randn((M, K), generator=torch.Generator(device="cuda").manual_seed(6), device="cuda").to(torch.bfloat16)
    pw = hq.hq_weight_prepare(inputs.weights((N, K), seed=N), 4, 256, hq.WEIGHT_MODES["folded"], hq.HQ_CODES_INT8).to_device()
    ws = torch.empty((hq.hq_workspace_size(M, K, hq.HQ_CODES_INT8),), dtype=torch.uint8, device="cuda")
    want, y = (torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    hq.hq_qlinear(x, pw, None, 4, want, ws, static_scale=torch.tensor([0.3], device="cuda"))
    for i in (0, M * N // 2 - 1):
        inside = y.view(-1).view(torch.float32)[i: i + 1]
        for _ in range(20):
            inside.fill_(0.3)
            hq.hq_qlinear(x, pw, None, 4, y, ws, static_scale=inside)
            assert torch.equal(y, want)

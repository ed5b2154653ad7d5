"""Codes of 4096-channel blocks, which change lanes before they are stored, against the same codes two to a byte, which do not: every
row in its place, nothing beside it, whatever the pitch and the number of rows a CTA leaves empty."""
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("rows,blocks,extra", [(1, 1, 0), (3, 1, 48), (257, 1, 16), (5, 2, 0), (64, 2, 32)])
def test_codes_of_wide_blocks(rows, blocks, extra, static, dt):
    import torch
    from paper_2512_05746_b200 import binding as hq
    cols = 4096 * blocks
    x = torch.randn((rows, cols), generator=torch.Generator(device="cuda").manual_seed(rows + blocks), device="cuda")
    x[:, 5] *= 50
    x = x if dt == "f32" else x.to(torch.bfloat16)
    ss = torch.tensor([0.3], device="cuda") if static else None
    buf = torch.full((rows + 2, cols + extra), 0x5A, dtype=torch.uint8, device="cuda")
    nib = torch.zeros((rows, cols // 2), dtype=torch.uint8, device="cuda")
    s8, s4 = torch.zeros(rows, device="cuda"), torch.zeros(rows, device="cuda")
    for a_bits in (3, 4):
        buf.fill_(0x5A)
        hq.hq_hadamard_quant(x, 4096, a_bits, buf[1:-1], 1, scales=s8, static_scale=ss)
        hq.hq_hadamard_quant(x, 4096, a_bits, nib, 0, scales=s4, static_scale=ss)
        torch.cuda.synchronize()
        want = torch.stack((nib & 15, nib >> 4), dim=-1).view(rows, cols).to(torch.int8)
        want = torch.where(want > 7, want - 16, want)
        assert torch.equal(buf[1:-1, :cols].view(torch.int8), want) and torch.equal(s8, s4)
        assert bool((buf[0] == 0x5A).all()) and bool((buf[-1] == 0x5A).all()) and bool((buf[1:-1, cols:] == 0x5A).all())
        assert want.unique().numel() > 4

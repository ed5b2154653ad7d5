"""GroupNorm statistics by one CTA per run of groups: scales and codes against fp64 over the shapes a run can take (pixels that the
sets of eight do not divide, groups of four channels that share a 16-byte piece, runs of several groups, a concatenated input
whose seam lies inside a run), with the tolerances of the other prologue tests."""
import numpy as np
import pytest

from hq_testutil import check_codes
from paper_2512_05746_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nb,H,W,C,G,n,dt,c1", [
    (2, 32, 32, 512, 32, 256, "bf16", 0),       # one group per CTA, whole sets
    (1, 8, 8, 2048, 32, 256, "bf16", 1024),     # fewer sets than threads of a piece; two tensors
    (3, 4, 24, 256, 64, 256, "bf16", 0),        # groups of four channels: two of them in a piece; 96 pixels = one set and a half
    (1, 4, 8, 384, 32, 128, "f32", 0),          # 12 channels per group in fp32, fewer pixels than a set of every thread
    (40, 8, 8, 1024, 32, 256, "bf16", 0),       # several groups per CTA
    (70, 8, 8, 512, 32, 256, "bf16", 256),      # the seam between two tensors lies between two runs
    (64, 16, 16, 512, 32, 256, "bf16", 0),      # 17 MB
    (2, 64, 64, 256, 32, 256, "bf16", 0),       # a cluster of four CTAs per run of two groups
    (1, 100, 50, 512, 32, 256, "bf16", 256),    # ... of eight, 625 sets over its threads: none left for the last three; two tensors
    (1, 36, 44, 256, 2, 256, "f32", 0),         # ... groups of 128 channels, 196 sets and 16 pixels behind them
    (3, 48, 48, 256, 32, 128, "bf16", 128),     # ... of two per run of two groups; two tensors
    (5, 48, 48, 768, 32, 256, "bf16", 0),       # more runs than SMs: one CTA each, four rounds of sets over 85 threads
    (2, 64, 64, 768, 32, 256, "f32", 0),        # ... of two, where four would share the sets unevenly
    (3, 4, 5, 768, 32, 256, "bf16", 0),         # 20 rows a sample: four to a CTA of the transform, and not eight
    (2, 6, 4, 1536, 32, 256, "f32", 0),         # 24: four and not two
])
def test_gn_statistics_of_a_run_of_groups(oracle, Nb, H, W, C, G, n, dt, c1):
    import torch
    from paper_2512_05746_b200 import binding as hq
    rng = np.random.default_rng(C + H)
    x = inputs.activations((Nb, H, W, C), outlier_count=max(1, C // 100), outlier_scale=8.0, seed=C + G) + np.float32(0.7)
    xt = torch.from_numpy(x).cuda()
    if dt == "bf16":
        xt = xt.to(torch.bfloat16)
        x = xt.float().cpu().numpy()
    e = torch.from_numpy(rng.standard_normal((Nb, C)).astype(np.float32)).cuda().to(torch.bfloat16)
    gamma = (1.0 + 0.2 * rng.standard_normal(C)).astype(np.float32)
    beta = (0.1 * rng.standard_normal(C)).astype(np.float32)
    rows = Nb * H * W
    codes, scales = torch.zeros((rows, C), dtype=torch.uint8, device="cuda"), torch.zeros((rows,), device="cuda")
    scratch = torch.full((Nb * G * 24,), 0xFF, dtype=torch.uint8, device="cuda")
    xa, xb = (xt, None) if c1 == 0 else (xt[..., :c1].contiguous(), xt[..., c1:].contiguous())
    hq.hq_gn_silu_quant(xa, G, torch.from_numpy(gamma).cuda(), torch.from_numpy(beta).cuda(), 1e-5, n, 4, codes, hq.HQ_CODES_INT8,
                        scratch, scales=scales, pre_bias=e, x2=xb)
    torch.cuda.synchronize()
    pick = sorted({0, Nb // 2, Nb - 1})
    xe = x[pick] + e.float().cpu().numpy()[pick][:, None, None, :].astype(np.float64)
    u = oracle.transform(oracle.groupnorm_silu(xe, G, gamma, beta, 1e-5).reshape(-1, C), n)
    q_ref, s_ref, v = oracle.quantize(u, 4, want_v=True)
    q = codes.view(Nb, H * W, C)[pick].reshape(-1, C).cpu().numpy().view(np.int8)
    s = scales.view(Nb, H * W)[pick].reshape(-1).cpu().numpy()
    assert float(np.abs(s / s_ref - 1.0).max()) <= 1e-6
    check_codes(q, q_ref, v, f"groupnorm runs {Nb}x{H}x{W}x{C}", tie_rel=1e-6, mismatch_frac=1e-4)


@pytest.mark.parametrize("Nb,H,W,C,G,slab", [
    (2, 32, 32, 512, 32, True),         # 32 pixel rows on 64 CTAs
    (1, 64, 64, 2048, 32, True),        # long runs, but the one-wave kernel's sums meet at 32 addresses
    (4, 40, 40, 2048, 32, True),        # 26 MB, shared evenly by single CTAs and unevenly by clusters of two
    (2, 64, 64, 1536, 32, True),        # 25 MB: clusters of two, unevenly shared by four
    (1, 256, 256, 128, 32, False),      # 16 CTAs of 65536 pixels each
    (1, 64, 64, 256, 1, False),         # one group: one CTA for the whole image
    (1, 160, 256, 512, 32, False),      # 42 MB on 32 CTAs
])
def test_few_large_samples_are_not_left_to_a_few_ctas(Nb, H, W, C, G, slab):
    """Which kernel took the statistics shows in the scratch: the one with a CTA per run of groups keeps its fp64 sums to itself."""
    import torch
    from paper_2512_05746_b200 import binding as hq
    gen = torch.Generator(device="cuda").manual_seed(C)
    x = (torch.randn((Nb, H, W, C), generator=gen, device="cuda") + 0.5).to(torch.bfloat16)
    gamma, beta = torch.randn((C,), generator=gen, device="cuda"), torch.randn((C,), generator=gen, device="cuda")
    scratch = torch.full((Nb * G * 24,), 0xFF, dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(x)
    hq.hq_groupnorm_act(x, G, gamma, beta, 1e-5, False, out, scratch)
    assert bool((scratch[: Nb * G * 16] == 0xFF).all()) == slab
    v = x.double().view(Nb, H * W, G, C // G)
    want = (v - v.mean(dim=(1, 3), keepdim=True)) * (v.var(dim=(1, 3), unbiased=False, keepdim=True) + 1e-5).rsqrt()
    want = want.view(Nb, H, W, C) * gamma.double() + beta.double()
    # one bf16 rounding (2^-9 relative) of an fp32 value that a few roundings at the size of its terms (at most 6 |gamma|) moved
    assert bool(((out.double() - want).abs() <= want.abs() * 2.0 ** -8 + 6 * gamma.double().abs() * 2.0 ** -20).all())

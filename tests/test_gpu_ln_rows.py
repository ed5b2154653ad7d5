"""The LayerNorm prologue's row statistics over the shapes of a row's threads (3 threads: no two lanes add up by shuffles; 36: runs
of four; 256: whole warps) and with either affine vector absent: scales and codes against fp64, and the same bits on every pass
(a row's parts are added in a fixed order)."""
import numpy as np
import pytest

from hq_testutil import check_codes
from paper_2512_05746_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,n,rpg,dt,with_w,with_b", [
    (321, 96, 32, 0, "f32", True, False),           # three threads a row, ragged rows
    (256, 1152, 128, 64, "bf16", False, True),      # 36 threads a row: nine parts
    (512, 384, 128, 128, "bf16", True, True),       # twelve threads a row: three parts
    (64, 8192, 512, 32, "f32", True, True),         # 256 threads a row
    (64, 16384, 4096, 32, "bf16", True, True),      # 256 threads of 64 values: the largest table
])
def test_ln_row_statistics(oracle, rows, cols, n, rpg, dt, with_w, with_b):
    import torch
    from paper_2512_05746_b200 import binding as hq
    rng = np.random.default_rng(cols)
    x = inputs.activations((rows, cols), outlier_count=max(1, cols // 100), outlier_scale=8.0, seed=cols) + np.float32(0.4)
    xt = torch.from_numpy(x).cuda()
    if dt == "bf16":
        xt = xt.to(torch.bfloat16)
        x = xt.float().cpu().numpy()
    groups = (rows + rpg - 1) // rpg if rpg else 1
    w = (1.0 + 0.3 * rng.standard_normal((groups, cols))).astype(np.float32) if with_w else None
    b = (0.5 * rng.standard_normal((groups, cols))).astype(np.float32) if with_b else None
    wd, bd = (None if v is None else torch.from_numpy(v).cuda() for v in (w, b))
    out = []
    for _ in range(3):
        codes = torch.zeros((rows, cols), dtype=torch.uint8, device="cuda")
        scales = torch.zeros((rows,), device="cuda")
        hq.hq_ln_quant(xt, wd, bd, rpg, 1e-6, n, 4, codes, hq.HQ_CODES_INT8, scales=scales)
        out.append((codes, scales))
    assert all(torch.equal(c, out[0][0]) and torch.equal(s, out[0][1]) for c, s in out[1:])
    ones, zeros = np.ones((groups, cols), np.float32), np.zeros((groups, cols), np.float32)
    u = oracle.transform(oracle.layernorm_affine(x, ones if w is None else w, zeros if b is None else b, rows_per_group=rpg, eps=1e-6), n)
    q_ref, s_ref, v = oracle.quantize(u, 4, want_v=True)
    # the statistics and the transform in fp32 move a scale by a few units of 2^-24, as in the other prologue tests
    assert float(np.abs(out[0][1].cpu().numpy() / s_ref - 1.0).max()) <= 1e-6
    check_codes(out[0][0].cpu().numpy().view(np.int8), q_ref, v, f"layernorm rows {rows}x{cols}", tie_rel=1e-6, mismatch_frac=1e-4)


@pytest.mark.parametrize("rows,cols,n,rpg,dt,with_w,with_b", [
    (1024, 1536, 256, 256, "bf16", True, True),     # two CTAs fewer per SM with a table
    (1024, 4096, 128, 0, "f32", True, True),        # one affine for all rows
    (304, 8192, 4096, 16, "bf16", True, False),     # 64 values a thread, no addend
    (160, 16384, 512 * 8, 0, "f32", False, True),   # the widest row, no factor
    (4096, 1152, 128, 0, "bf16", False, False),     # neither vector
    (321, 96, 32, 0, "f32", False, False),
])
def test_ln_affine_read_where_it_is_used(oracle, rows, cols, n, rpg, dt, with_w, with_b):
    """Rows whose table of affine vectors would cost resident CTAs, and rows without any."""
    test_ln_row_statistics(oracle, rows, cols, n, rpg, dt, with_w, with_b)

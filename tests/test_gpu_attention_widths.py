"""The attention core on tensor-map tiles at head widths of 32, 48 and 96 (lengths that fill their key blocks): one block, several,
a partly filled query tile, the last head's tile that reaches past its channels; element-wise bound of the arithmetic."""
import numpy as np
import pytest

from hq_testutil import attention_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nb,L,heads,dh", [(3, 64, 3, 32), (2, 192, 5, 48), (2, 256, 2, 96), (1, 320, 1, 96)])
def test_attention_on_tensor_map_tiles(oracle, Nb, L, heads, dh):
    import torch
    from paper_2512_05746_b200 import binding as hq
    C = heads * dh
    qkv = torch.from_numpy(np.random.default_rng(L + dh).standard_normal((Nb * L, 3 * C)).astype(np.float32)).cuda().to(torch.bfloat16)
    out = torch.zeros((Nb * L, C), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    hq.hq_attention(qkv, Nb, heads, out, dev_status=status)
    hq.hq_check_status(status)
    qr = qkv.float().cpu().numpy().astype(np.float64)
    want = oracle.attention(qr.reshape(Nb, L, 3 * C), heads).reshape(Nb * L, C)
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - want) <= attention_bound(oracle, qr, Nb, L, C, heads, want))

"""CPU-only checks of the C-ABI library: it loads, exports what include/hq.h declares, validates arguments
before touching the GPU, and its offline weight preparation agrees with the oracle."""
import ctypes as C
import os
import re

import numpy as np
import pytest

from paper_2512_05746_b200 import inputs
from hq_testutil import decode_blob

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def hq():
    from paper_2512_05746_b200 import build
    build.build()
    from paper_2512_05746_b200 import binding
    return binding


def test_library_exports_every_declared_symbol(hq):
    text = open(os.path.join(ROOT, "include", "hq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    declared = set(re.findall(r"\b(hq_[a-z0-9_]+)\s*\(", text))
    assert declared, "no declarations found"
    assert declared == set(hq.EXPORTS)
    for name in declared:
        assert hasattr(hq.lib, name), name
    assert hq.hq_version() >= 100
    assert hq.status_string(0) == "ok" and "overflow" in hq.status_string(6)


def test_check_status_decodes_timeout_word(hq):
    ok = np.zeros(1, np.int32)
    bad = np.array([0x300], np.int32)
    assert hq.lib.hq_check_status(ok.ctypes.data_as(C.c_void_p)) == 0
    assert hq.lib.hq_check_status(bad.ctypes.data_as(C.c_void_p)) == 8
    assert hq.lib.hq_check_status(None) == 1


def test_argument_validation_without_gpu(hq):
    L = hq.lib
    fake = C.c_void_p(0x1000)
    # NULL pointers
    assert L.hq_hadamard_quant(None, 0, 4, 256, 256, 256, 4, 0, None, fake, 0, 128, fake, None) == 1
    # cols not a multiple of the block / block not a power of two
    assert L.hq_hadamard_quant(fake, 0, 4, 384, 384, 256, 4, 0, None, fake, 0, 192, fake, None) == 2
    assert L.hq_hadamard_quant(fake, 0, 4, 384, 384, 96, 4, 0, None, fake, 0, 192, fake, None) == 2
    # bits outside {3,4,8}; 8-bit codes in a nibble container
    assert L.hq_hadamard_quant(fake, 0, 4, 256, 256, 256, 5, 0, None, fake, 0, 128, fake, None) == 1
    assert L.hq_hadamard_quant(fake, 0, 4, 256, 256, 256, 8, 0, None, fake, 0, 128, fake, None) == 2
    # static mode without a scale
    assert L.hq_hadamard_quant(fake, 0, 4, 256, 256, 256, 4, 1, None, fake, 0, 128, fake, None) == 1
    # zero rows is a no-op
    assert L.hq_hadamard_quant(fake, 0, 0, 256, 256, 256, 4, 0, None, fake, 0, 128, fake, None) == 0
    out = C.c_size_t(0)
    assert L.hq_workspace_size(128, 256, 0, C.byref(out)) == 0 and out.value >= 128 * 128 + 128 * 4
    assert L.hq_workspace_size(128, 256, 1, C.byref(out)) == 0 and out.value >= 128 * 256 + 128 * 4
    assert L.hq_workspace_size(128, 0, 0, C.byref(out)) == 2


def test_gemm_validation_without_gpu(hq):
    w = inputs.weights((256, 256), seed=0)
    pw = hq.hq_weight_prepare(w, 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)
    L = hq.lib
    fake = C.c_void_p(0x1000)
    d = C.byref(pw.desc)
    # container mismatch with the blob
    assert L.hq_qgemm(fake, 0, 4, 128, 256, 128, d, fake, fake, 0, fake, None, 1.0, fake, None, 1, 256, None, None) == 2
    # K mismatch
    assert L.hq_qgemm(fake, 1, 4, 128, 512, 512, d, fake, fake, 0, fake, None, 1.0, fake, None, 1, 256, None, None) == 2
    # neither output requested
    assert L.hq_qgemm(fake, 1, 4, 128, 256, 256, d, fake, fake, 0, fake, None, 1.0, None, None, 1, 256, None, None) == 1
    # 8-bit activations against 2-limb folded weights whose integers are large: K * 128 * max|B| >= 2^31
    w8 = np.ones((128, 4096), np.float32)
    pw8 = hq.hq_weight_prepare(w8, 8, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)
    assert L.hq_qgemm(fake, 1, 8, 128, 4096, 4096, C.byref(pw8.desc), fake, fake, 0, fake, None, 1.0, fake, None, 1,
                      128, None, None) == 6
    # conv: unsupported filter size
    wc = inputs.weights((128, 3, 3, 128), seed=2)
    pwc = hq.hq_weight_prepare(wc, 4, 128, hq.HQ_W_PLAIN, hq.HQ_CODES_INT8)
    assert L.hq_qconv2d(fake, 1, 4, 1, 8, 8, 128, C.byref(pwc.desc), fake, 5, 5, 1, 1, fake, 1, fake, None, 1.0, fake,
                        None, 1, None, None) == 3


@pytest.mark.parametrize("mode", ["plain", "folded"])
@pytest.mark.parametrize("container", [0, 1])
@pytest.mark.parametrize("shape,had_block,w_bits", [((40, 256), 256, 4), ((130, 3, 3, 128), 128, 4),
                                                     ((16, 64), 16, 4), ((300, 768), 256, 4), ((8, 512), 512, 8),
                                                     ((5, 1, 1, 24), 8, 4)])
def test_weight_prepare_matches_oracle(hq, oracle, mode, container, shape, had_block, w_bits):
    w = inputs.weights(shape, seed=len(shape) + had_block)
    pw = hq.hq_weight_prepare(w, w_bits, had_block, hq.WEIGHT_MODES[mode], container)
    B_ref, s_ref = oracle.prepare_weights(w.reshape(shape[0], -1, shape[-1]), w_bits, had_block, mode)
    assert np.array_equal(pw.s_w, s_ref)
    assert np.array_equal(decode_blob(pw), B_ref)
    d = pw.desc
    assert d.bytes == hq.hq_weight_blob_bytes(shape[0], d.RS, shape[-1], w_bits, had_block, hq.WEIGHT_MODES[mode])
    assert d.max_abs_b == np.abs(B_ref).max()
    expect_limbs = 2 if (mode == "folded" and had_block * 2 ** (w_bits - 1) > 128) else 1
    assert d.limbs == expect_limbs
    a = 2.0 ** (-0.5 * np.log2(had_block)) if mode == "folded" else 1.0
    assert np.isclose(pw.alpha, a, rtol=1e-7)


def test_weight_prepare_double_close_to_oracle(hq, oracle):
    w = inputs.weights((64, 512), seed=9)
    pw = hq.hq_weight_prepare(w, 4, 512, hq.HQ_W_DOUBLE, hq.HQ_CODES_INT8)
    B_ref, s_ref = oracle.prepare_weights(w.reshape(64, 1, 512), 4, 512, "double")
    assert np.allclose(pw.s_w, s_ref, rtol=1e-6)
    diff = decode_blob(pw) != B_ref          # butterfly vs dense summation order: only exact ties may differ
    assert diff.mean() <= 1e-4
    assert pw.desc.limbs == 1 and pw.alpha == 1.0


def test_weight_prepare_errors(hq):
    w = inputs.weights((8, 48), seed=0)
    with pytest.raises(hq.HqError) as e:
        hq.hq_weight_prepare(w, 4, 32, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)    # 48 % 32 != 0
    assert e.value.status == 2
    with pytest.raises(hq.HqError) as e:
        hq.hq_weight_prepare(w, 5, 16, hq.HQ_W_PLAIN, hq.HQ_CODES_INT8)
    assert e.value.status == 1


def test_unet_layer_list_matches_the_workload_description():
    """Base 256, multipliers (1,2,3,4), 2 residual blocks per level, attention at 32/16/8, batch 64 on a 64x64 latent:
    121 quantized layers of 47 distinct shapes, 16.0 TOP per forward counted with one weight limb."""
    from paper_2512_05746_b200 import unet
    layers = unet.quantized_layers()
    assert len(layers) == 121 and len(unet.distinct_shapes(layers)) == 47
    assert abs(2 * sum(L["macs"] for L in layers) / 1e12 - 16.04) < 0.01
    for L in layers:
        cin = L["C"] if L["kind"] == "conv" else L["K"]
        assert cin % L["had_block"] == 0 and L["had_block"] == 256
    assert sum(1 for L in layers if L["kind"] == "conv" and L["stride"] == 2) == 3
    assert sum(1 for L in layers if L["kind"] == "conv" and L["R"] == 1) == 15
    assert max(L["C"] for L in layers if L["kind"] == "conv") == 2048       # skip concatenation at the deepest level


def test_dit_layer_list():
    """Width 1152 = 9 x 128, depth 28, MLP ratio 4, batch 32 x 256 tokens: 28 x 5 + 3 quantized linears."""
    from paper_2512_05746_b200 import dit
    layers = dit.quantized_layers()
    assert len(layers) == 28 * 5 + 3
    assert all(L["K"] % L["had_block"] == 0 and L["had_block"] == 128 for L in layers)
    big = [L for L in layers if L["M"] == 32 * 256]
    assert len(big) == 28 * 4 and {(L["K"], L["N"]) for L in big} == {(1152, 3456), (1152, 1152), (1152, 4608), (4608, 1152)}


@pytest.mark.parametrize("had_block", [128, 1024])
def test_fused_layers_refuse_null_weights_before_a_launch(hq, had_block):
    """The split fold (blocks of 32 to 512) derives a second address from the weights': a null one has to be refused as it is
    where the layer runs on the weights alone (block 1024)."""
    K, N, M = 1152 if had_block == 128 else 2048, 4608, 8192
    lin = hq.hq_weight_prepare(inputs.weights((N, K), seed=1), 4, had_block, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)
    conv = hq.hq_weight_prepare(inputs.weights((256, 3, 3, 1024), seed=1), 4, had_block, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)
    assert lin.desc.reserved == conv.desc.reserved == (1 if had_block == 128 else 0)
    L, d, dc, fake, big = hq.lib, C.byref(lin.desc), C.byref(conv.desc), C.c_void_p(0x1000), 1 << 30
    assert L.hq_qlinear(fake, 1, M, K, K, d, None, fake, None, 4, 0, None, fake, 1, N, fake, big, None, None) == 1
    assert L.hq_ln_qlinear(fake, 1, M, K, K, None, None, 0, 1e-6, d, None, fake, None, 4, fake, 1, N, fake, big, None, None) == 1
    assert L.hq_gn_qlinear(fake, 1, 8, M // 8, K, 32, fake, fake, 1e-5, 0, d, None, fake, None, 4, fake, 1, N, fake, big, fake,
                           1 << 20, None, None) == 1
    assert L.hq_qconv(fake, 1, 8, 32, 32, 1024, dc, None, 3, 3, 1, 1, fake, None, 4, 1, fake, fake, 1, fake, big, None, None) == 1
    assert L.hq_qconv_cat(fake, fake, 0, 1, 8, 32, 32, 1024, dc, None, 3, 3, 1, 1, fake, None, 4, 1, fake, fake, 1, fake, big,
                          None, None) == 1
    assert L.hq_gn_silu_qconv(fake, 1, 8, 32, 32, 1024, 32, fake, fake, None, 1e-5, dc, None, 3, 3, 1, 1, fake, None, 4, 1, fake,
                              fake, 1, fake, big, fake, 1 << 20, None, None) == 1
    assert L.hq_gn_silu_qconv_cat(fake, fake, 0, 1, 8, 32, 32, 1024, 32, fake, fake, None, 1e-5, dc, None, 3, 3, 1, 1, fake, None, 4,
                                  1, fake, fake, 1, fake, big, fake, 1 << 20, None, None) == 1
    assert L.hq_qlinear_noalloc(fake, 1, 1024, K, K, d, None, fake, None, 4, 0, None, fake, 1, N, None, None) == 1


@pytest.mark.parametrize("rows,cols,n,mode,w_bits,container,a_bits,static,stride,taps,room", [
    (4096, 1152, 128, "folded", 4, 1, 4, False, 1, 1, True),        # 4.5 MiB of codes, runs on one limb
    (4096, 1152, 128, "folded", 4, 0, 3, True, 1, 1, True),         # two codes per byte
    (65536, 1152, 128, "folded", 4, 1, 8, False, 1, 1, False),      # 8-bit codes need two limbs
    (65536, 1024, 1024, "folded", 4, 1, 4, False, 1, 1, False),     # one limb where it is given the room: the query does not ask above 512
    (65536, 1152, 128, "double", 4, 1, 4, False, 1, 1, False),      # one limb anyhow
    (256, 256, 256, "folded", 4, 1, 4, False, 1, 1, False),         # nothing to gain
    (15 * 32 * 32, 512, 256, "folded", 4, 1, 4, True, 1, 9, True),  # 7.6 MiB
    (64 * 32 * 32, 512, 256, "folded", 4, 1, 4, False, 1, 9, False),    # likewise one scale per pixel under a 3x3 window
])
def test_layer_workspace_asks_for_what_the_layer_uses(hq, rows, cols, n, mode, w_bits, container, a_bits, static, stride, taps, room):
    N = {1152: 4608, 256: 256}.get(cols, 1024)
    w = inputs.weights((N, cols) if taps == 1 else (512, 3, 3, cols), seed=0)
    pw = hq.hq_weight_prepare(w, w_bits, n, hq.WEIGHT_MODES[mode], container)
    pitch = (cols // 2 if container == 0 else cols + 15) // 16 * 16
    codes = (rows * pitch + 255) // 256 * 256 + 4 * rows
    want = (codes + 255) // 256 * 256 + rows * cols if room else codes
    assert hq.hq_layer_workspace_size(pw, a_bits, rows, static, stride) == want
    pw.desc.reserved = 0                                            # a blob of the two-limb section alone
    assert hq.hq_layer_workspace_size(pw, a_bits, rows, static, stride) == codes
    out = C.c_size_t(0)
    assert hq.lib.hq_layer_workspace_size(None, a_bits, 0, rows, 1, C.byref(out)) == 1
    assert hq.lib.hq_layer_workspace_size(C.byref(pw.desc), 5, 0, rows, 1, C.byref(out)) == 1
    assert hq.lib.hq_layer_workspace_size(C.byref(pw.desc), a_bits, 0, -1, 1, C.byref(out)) == 2
    assert hq.lib.hq_layer_workspace_size(C.byref(pw.desc), a_bits, 0, rows, 3, C.byref(out)) == 3


@pytest.mark.parametrize("n", [32, 512])
@pytest.mark.parametrize("kind", ["subnormal", "not a number", "all not a number"])
def test_split_section_holds_the_extreme_integers(hq, n, kind):
    """-8 in the quantized weights: the scale of the largest of them is rounded to a subnormal, or they are no numbers."""
    N, rng = 64, np.random.default_rng(n)
    w = rng.choice([-1.0, 1.0], size=(N, n)).astype(np.float32)
    if kind == "subnormal":                 # the absolute maximum, 11 units, over a scale of one and a half, rounded to one or two
        w = (np.where(rng.random((N, n)) < 0.5, -11.0, 7.0) * 2.0 ** -149).astype(np.float32)
    elif kind == "not a number":
        w[rng.random((N, n)) < 0.5] = np.nan
    else:
        w[:] = np.nan
    pw = hq.hq_weight_prepare(w, 4, n, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8)
    d = pw.desc
    assert d.reserved == 1
    B1 = pw.blob[d.N_pad * 2 * d.C_pad:].reshape(d.N_pad, d.C_pad)[:N, :n].astype(np.int64)
    B = decode_blob(pw).reshape(N, n).astype(np.int64)
    # the remaining factors of the folded weights, index bits 2, 3, 4, 1, 0 in this order
    for bit in [2, 3, 4, 1, 0][: n.bit_length() - 5]:
        v = B1.reshape(N, -1, 2, 1 << bit)
        B1 = np.stack([v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]], axis=2).reshape(N, n)
    assert np.array_equal(B1, B)


@pytest.mark.parametrize("n", [1024, 2048, 4096])
@pytest.mark.parametrize("blocks,taps,N", [(1, 1, 130), (2, 1, 64), (1, 9, 8)])
def test_the_size_of_a_buffer_never_says_that_a_section_is_there(hq, n, blocks, taps, N):
    """Above 512 channels the one-limb section is known by desc->bytes alone: a descriptor that was given the size of the buffer
    must not equal one of a blob with a section (its bytes, or halved with 128 further columns and a parity)."""
    C, N_pad = n * blocks, (N + 127) // 128 * 128
    rows = N_pad * taps * C
    section = hq.hq_weight_blob_bytes(N, taps, C, 4, n, hq.HQ_W_FOLDED) - 2 * rows
    halved = N_pad * (C + 129) if blocks == taps == 1 and n > 1024 else 0
    assert section > max(rows, halved) and section % 16 == 0

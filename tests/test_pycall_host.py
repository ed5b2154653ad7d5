"""The native marshalling of the frequent calls hands the entry points what the tensors and arguments say: checked against functions
in their place that keep their arguments."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2512_05746_b200 import inputs

P, I, L, Z, F = C.c_void_p, C.c_int, C.c_int64, C.c_size_t, C.c_float
QLINEAR = [P, I, L, L, L, P, P, P, P, I, I, P, P, I, L, P, Z, P, P]
QCONV = [P, I, L, L, L, L, P, P, I, I, I, I, P, P, I, I, P, P, I, P, Z, P, P]
LN = [P, I, L, L, L, P, P, L, F, P, P, P, P, I, P, I, L, P, Z, P, P]
QUANT = [P, I, L, L, L, I, I, I, P, P, I, L, P, P]


class Stream:
    cuda_stream = 0x7123456789


@pytest.fixture()
def taken():
    from paper_2512_05746_b200 import binding as hq
    seen, status = [], [0]

    def fake(types):
        def keep(*args):
            seen.append(args)
            return status[0]
        return C.CFUNCTYPE(I, *types)(keep)
    fakes = [fake(t) for t in (QLINEAR, QCONV, LN, QUANT)]
    own = [C.cast(getattr(hq.lib, n), P).value for n in ("hq_qlinear", "hq_qconv", "hq_ln_qlinear", "hq_hadamard_quant")]
    hq._hqcall.bind(hq._dtype_code, *(C.cast(f, P).value for f in fakes))
    try:
        yield hq, seen, status
    finally:
        hq._hqcall.bind(hq._dtype_code, *own)


def weights(hq, shape):
    return hq.hq_weight_prepare(inputs.weights(shape, seed=1), 4, 64, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device("cpu")


def plain(args):
    return [0 if v is None else v for v in args]


@pytest.mark.parametrize("xdt,ydt", [(torch.float32, torch.bfloat16), (torch.bfloat16, torch.float32)])
@pytest.mark.parametrize("static", [False, True])
def test_linear(taken, xdt, ydt, static):
    hq, seen, _ = taken
    pw = weights(hq, (48, 64))
    x, y = torch.zeros((5, 96), dtype=xdt)[:, 16:80], torch.zeros((5, 64), dtype=ydt)[:, :48]
    ws, b, st = torch.zeros(77, dtype=torch.int16), torch.zeros(48), torch.zeros(1, dtype=torch.int32)
    ss = torch.zeros(1) if static else None
    hq.hq_qlinear(x, pw, b, np.int64(3), y, ws, static_scale=ss, dev_status=st, stream=Stream)
    code = {torch.float32: 0, torch.bfloat16: 1}
    assert plain(seen[0]) == [x.data_ptr(), code[xdt], 5, 64, 96, C.addressof(pw.desc), pw.blob_dev.data_ptr(), pw.s_w_dev.data_ptr(),
                              b.data_ptr(), 3, int(static), ss.data_ptr() if static else 0, y.data_ptr(), code[ydt], 64, ws.data_ptr(), 154,
                              st.data_ptr(), Stream.cuda_stream]
    hq.hq_qlinear(x, pw, None, 4, y, ws, static_scale=torch.zeros(0), stream=Stream)        # a scale that holds nothing is still a scale
    assert plain(seen[1])[8:12] == [0, 4, 1, 0] and plain(seen[1])[17] == 0


def test_convolution_normalised_linear_and_transform(taken):
    hq, seen, _ = taken
    pw = weights(hq, (48, 3, 3, 64))
    x, y = torch.zeros((2, 6, 4, 64), dtype=torch.bfloat16), torch.zeros((2, 3, 2, 48), dtype=torch.bfloat16)
    ws, b, ss = torch.zeros(77, dtype=torch.uint8), torch.zeros(48), torch.zeros(1)
    hq.hq_qconv(x, pw, 3, 3, 2, 1, b, 4, y, ws, static_scale=ss, stream=Stream)
    w = [C.addressof(pw.desc), pw.blob_dev.data_ptr()]
    assert plain(seen[0]) == [x.data_ptr(), 1, 2, 6, 4, 64, *w, 3, 3, 2, 1, pw.s_w_dev.data_ptr(), b.data_ptr(), 4, 1, ss.data_ptr(), y.data_ptr(),
                              1, ws.data_ptr(), 77, 0, Stream.cuda_stream]
    pw = weights(hq, (48, 64))
    x, y, g = torch.zeros((6, 64)), torch.zeros((6, 48), dtype=torch.bfloat16), torch.zeros((3, 64))
    hq.hq_ln_qlinear(x, g, None, 2, 1e-6, pw, b, 4, y, ws, stream=Stream)
    assert plain(seen[1]) == [x.data_ptr(), 0, 6, 64, 64, g.data_ptr(), 0, 2, np.float32(1e-6), C.addressof(pw.desc), pw.blob_dev.data_ptr(),
                              pw.s_w_dev.data_ptr(), b.data_ptr(), 4, y.data_ptr(), 1, 48, ws.data_ptr(), 77, 0, Stream.cuda_stream]
    codes, sc = torch.zeros((6, 80), dtype=torch.uint8), torch.zeros(6)
    hq.hq_hadamard_quant(x, 64, 8, codes, 1, scales=sc, stream=Stream)
    assert plain(seen[2]) == [x.data_ptr(), 0, 6, 64, 64, 64, 8, 0, 0, codes.data_ptr(), 1, 80, sc.data_ptr(), Stream.cuda_stream]


def test_what_was_refused_is_refused(taken):
    hq, seen, status = taken
    pw, ws = weights(hq, (48, 64)), torch.zeros(77, dtype=torch.uint8)
    x, y = torch.zeros((6, 64)), torch.zeros((6, 48), dtype=torch.bfloat16)
    with pytest.raises(ValueError):
        hq.hq_qlinear(x.view(2, 3, 64), pw, None, 4, y, ws, stream=Stream)
    with pytest.raises(TypeError):
        hq.hq_qlinear(x.double(), pw, None, 4, y, ws, stream=Stream)
    with pytest.raises(AttributeError):
        hq.hq_qlinear(x, pw, 3.0, 4, y, ws, stream=Stream)
    with pytest.raises(AttributeError):
        hq.hq_qlinear(x, object(), None, 4, y, ws, stream=Stream)
    with pytest.raises(TypeError):
        hq.hq_qlinear(x, pw, None, "4", y, ws, stream=Stream)
    assert not seen
    status[0] = 5
    with pytest.raises(hq.HqError) as e:
        hq.hq_qlinear(x, pw, None, 4, y, ws, stream=Stream)
    assert e.value.status == 5


def test_the_module_belongs_to_this_python_and_says_why_it_cannot_be_loaded():
    import os
    import subprocess
    import sys
    import sysconfig

    from paper_2512_05746_b200 import binding, build
    assert os.path.samefile(binding._hqcall.__file__, build.PYCALL) and build.PYCALL.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    r = subprocess.run([sys.executable, "-c", "import sys; sys.modules['paper_2512_05746_b200._hqcall'] = None\n"
                        "import paper_2512_05746_b200.binding"], capture_output=True, text=True, cwd=os.path.dirname(os.path.dirname(build.LIB)))
    assert r.returncode != 0 and "_hqcall cannot be loaded" in r.stderr and "halted" in r.stderr

"""A fused call may be launched while the kernel in front of it on the stream is still running.  What that kernel wrote, it reads as
if the two were synchronised in between: calls chained through an operand, many times over changing values and in a graph, give
what the same calls give one at a time."""
import pytest

from paper_2512_05746_b200 import inputs


def chained(torch, step, values, outputs):
    """`step(value)` for every value: one at a time, back to back, and as one graph; the `outputs` of each must agree."""
    def collect(sync=False):
        out = []
        for v in values:
            step(v)
            if sync:
                torch.cuda.synchronize()
            out.append([t.clone() for t in outputs])
        return out

    apart, together = collect(sync=True), collect()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        graph.capture_begin()
        try:
            captured = collect()
        finally:
            graph.capture_end()
    torch.cuda.current_stream().wait_stream(stream)
    graph.replay()
    torch.cuda.synchronize()
    for i, want in enumerate(apart):
        for a, b, c in zip(want, together[i], captured[i]):
            assert torch.equal(a, b) and torch.equal(a, c), i
    assert any(not torch.equal(a, b) for a, b in zip(apart[0], apart[1])), "the values were meant to matter"


def inputs_of(torch, shape, n, dtype=None):
    gen = torch.Generator(device="cuda").manual_seed(shape[-1])
    x = torch.randn((n, *shape), generator=gen, device="cuda") * torch.rand((n, *[1] * len(shape)), generator=gen, device="cuda").mul(4).exp()
    return list(x if dtype is None else x.to(dtype))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["quantize", "linear", "linear of 2048", "convolution"])
def test_static_scale_from_the_transform_in_front(kind):
    import torch
    from paper_2512_05746_b200 import binding as hq
    K = 2048 if kind == "linear of 2048" else 256
    rows, N = 128, 256
    pw = hq.hq_weight_prepare(inputs.weights((N, 3, 3, K) if kind == "convolution" else (N, K), seed=1), 4, 256, hq.HQ_W_FOLDED,
                              hq.HQ_CODES_INT8).to_device()
    codes, own = (torch.zeros((rows, K), dtype=torch.uint8, device="cuda") for _ in range(2))
    s = torch.ones((rows,), device="cuda")
    ws = torch.zeros((hq.hq_workspace_size(rows, K, hq.HQ_CODES_INT8),), dtype=torch.uint8, device="cuda")
    y = torch.zeros((rows, N), dtype=torch.bfloat16, device="cuda")

    def step(x):
        hq.hq_hadamard_quant(x, 256, 4, codes, hq.HQ_CODES_INT8, scales=s)
        if kind == "quantize":
            hq.hq_hadamard_quant(x, 256, 4, own, hq.HQ_CODES_INT8, static_scale=s[:1])
        elif kind == "convolution":
            hq.hq_qconv(x.view(2, 8, 8, K), pw, 3, 3, 1, 1, None, 4, y.view(2, 8, 8, N), ws, static_scale=s[:1])
        else:
            hq.hq_qlinear(x, pw, None, 4, y, ws, static_scale=s[:1])

    chained(torch, step, inputs_of(torch, (rows, K), 200), [own if kind == "quantize" else y])


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,room", [
    (2, 1024, 1024, False),        # both products divided over clusters, the transform between them a dependent
    (64, 256, 256, False),         # the layer in front is one kernel
    (300, 768, 264, False),
    (4096, 1024, 1024, True),      # pairs of SMs
])
def test_residual_from_the_layer_in_front(M, K, N, room):
    import torch
    from paper_2512_05746_b200 import binding as hq
    first, second = (hq.hq_weight_prepare(inputs.weights((N, K), seed=i), 4, 256, hq.HQ_W_FOLDED, hq.HQ_CODES_INT8).to_device()
                     for i in (1, 2))
    ws1, ws2 = (torch.zeros((max(hq.hq_layer_workspace_size(first, 4, M), hq.hq_workspace_size(M, K, 1)) if room else
                             (M * K + 255) // 256 * 256 + 4 * M,), dtype=torch.uint8, device="cuda") for _ in range(2))
    x2 = inputs_of(torch, (M, K), 1, torch.bfloat16)[0]
    r, y = (torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")

    def step(x):
        hq.hq_qlinear(x, first, None, 4, r, ws1, dev_status=status)
        hq.hq_qlinear(x2, second, None, 4, y, ws2, dev_status=status, residual=r)

    chained(torch, step, inputs_of(torch, (M, K), 200 if M < 1000 else 20, torch.bfloat16), [y])
    hq.hq_check_status(status)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["one kernel", "divided over clusters", "convolution", "resident", "streamed"])
def test_weights_from_the_transform_in_front(kind):
    """Codes are weights as a layer of one limb reads them: the transform's rows of codes are the prepared rows, its scales theirs."""
    import torch
    from paper_2512_05746_b200 import binding as hq
    M, K, taps = {"one kernel": (64, 256, 1), "divided over clusters": (64, 2048, 1), "convolution": (128, 256, 9),
                  "resident": (4096, 256, 1), "streamed": (4096, 768, 1)}[kind]
    N = 256
    pw = hq.hq_weight_prepare(inputs.weights((N, 3, 3, K) if taps == 9 else (N, K), seed=1), 4, 256, hq.HQ_W_PLAIN, hq.HQ_CODES_INT8)
    assert pw.desc.limbs == 1 and pw.desc.N_pad == N and pw.desc.max_abs_b == 7
    pw.blob_dev = torch.zeros((N, taps * K), dtype=torch.uint8, device="cuda")
    pw.s_w_dev = torch.ones((N,), device="cuda")
    x = inputs_of(torch, (M, K), 1, torch.bfloat16)[0]
    ws = torch.zeros((hq.hq_workspace_size(M, K, hq.HQ_CODES_INT8),), dtype=torch.uint8, device="cuda")
    y = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    ss = torch.tensor([0.1], device="cuda")
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")

    def step(w):
        hq.hq_hadamard_quant(w, 256, 4, pw.blob_dev, hq.HQ_CODES_INT8, scales=pw.s_w_dev)
        if taps == 9:
            hq.hq_qconv(x.view(2, 8, 8, K), pw, 3, 3, 1, 1, pw.s_w_dev, 4, y.view(2, 8, 8, N), ws, static_scale=ss, dev_status=status)
        else:
            hq.hq_qlinear(x, pw, pw.s_w_dev, 4, y, ws, dev_status=status)

    chained(torch, step, inputs_of(torch, (N, taps * K), 100, torch.bfloat16), [y])
    hq.hq_check_status(status)

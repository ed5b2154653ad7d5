"""`UNet.forward` keeps its launches as a CUDA graph from the second call on: every call gives what the library calls issued one by
one give for the same inputs, on any stream, after a change of the activations' bit width and inside a caller's own capture."""
import pytest

from paper_2512_05746_b200 import inputs

pytestmark = pytest.mark.gpu


def test_forward_by_graph_is_the_forward_by_calls():
    import torch
    from paper_2512_05746_b200 import binding as hq
    from paper_2512_05746_b200.unet import UNet
    cfg = inputs.unet_config(batch=2, latent=32, base=128, attn_resolutions=(16, 8, 4), had_block=128, classes=10)
    net = UNet(cfg, inputs.unet_params(cfg, seed=0), hq, torch.device("cuda", 0)).build(2)
    I = inputs.unet_inputs(cfg, seed=0)
    net.calibrate(*(torch.from_numpy(I[k]) for k in ("x", "t", "y")))

    def draw(seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        return (torch.randn(tuple(I["x"].shape), generator=g, device="cuda"), torch.rand((2,), generator=g, device="cuda") * 1000,
                torch.randint(0, 10, (2,), generator=g, device="cuda", dtype=torch.int32))

    def by_calls(args):
        return net.forward(*args, record=[]).clone()

    assert net.graph is None
    for seed in range(3):
        got = net.forward(*draw(seed)).clone()
        assert torch.equal(got, by_calls(draw(seed)))
    assert net.graph is not None
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        got = net.forward(*draw(7)).clone()
    side.synchronize()
    assert torch.equal(got, by_calls(draw(7)))
    net.a_bits = 8
    for seed in (3, 4):
        got = net.forward(*draw(seed)).clone()
        assert torch.equal(got, by_calls(draw(seed)))
    args, graph = draw(9), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = net.forward(*args)
    graph.replay()
    torch.cuda.synchronize()
    got = out.clone()
    assert torch.equal(got, by_calls(args))
    hq.hq_check_status(net.status)


def test_forward_follows_replaced_weights_status_and_kernel_choice():
    import torch
    from paper_2512_05746_b200 import binding as hq
    from paper_2512_05746_b200.unet import UNet
    cfg = inputs.unet_config(batch=2, latent=32, base=128, attn_resolutions=(16, 8, 4), had_block=128, classes=10)
    net = UNet(cfg, inputs.unet_params(cfg, seed=0), hq, torch.device("cuda")).build(2)
    I = inputs.unet_inputs(cfg, seed=0)
    args = [torch.from_numpy(I[k]) for k in ("x", "t", "y")]
    net.calibrate(*args)
    for _ in range(3):
        net.forward(*args)
    first = net.forward(*args).clone()
    pw, graph = net.pw["mid.attn.qkv"], net.graph
    assert graph is not None
    kept = pw.blob_dev, pw.s_w_dev, net.status               # their addresses are not handed out again
    pw.to_device()
    pw.blob_dev.zero_()                                      # other weights at another address
    want = net.forward(*args, record=[]).clone()
    assert not torch.equal(want, first)
    for _ in range(3):
        assert torch.equal(net.forward(*args), want)
    assert net.graph is not graph
    net.status = torch.zeros_like(net.status)
    for _ in range(3):
        assert torch.equal(net.forward(*args), want)
    hq.hq_check_status(net.status)
    graph, before = net.graph, hq.hq_set_pair_gemm(0)
    try:
        for _ in range(3):
            assert torch.equal(net.forward(*args), want)
        assert net.graph is not graph
    finally:
        hq.hq_set_pair_gemm(before)
    del kept

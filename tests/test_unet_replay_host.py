"""When `UNet.replay` may reuse a captured forward, on the CPU: a stand-in for the graph keeps the launches of its capture with the
addresses they had, and every forward has to launch what the calls issued one by one would launch now."""
import contextlib
import types

import pytest
import torch

from paper_2512_05746_b200 import unet


class FakeCuda:
    """Launches go to `log`, or to the graph that is being captured; a replay repeats the graph's."""

    def __init__(self):
        self.log, self.capturing, self.device = [], None, 0
        cuda = self

        class CUDAGraph:
            def capture_begin(self, **_):
                self.launches, cuda.capturing = [], self

            def capture_end(self):
                cuda.capturing = None

            def replay(self):
                cuda.log += self.launches

        self.CUDAGraph = CUDAGraph
        self.Stream = self.current_stream = lambda: types.SimpleNamespace(wait_stream=lambda other: None)

    def stream(self, s):
        return contextlib.nullcontext()

    def current_device(self):
        return self.device

    def is_current_stream_capturing(self):
        return False

    def launch(self, what):
        (self.log if self.capturing is None else self.capturing.launches).append(what)


class Workspace(torch.Tensor):
    device = types.SimpleNamespace(index=0)


def make_net():
    from paper_2512_05746_b200 import binding as hq
    cuda, net = FakeCuda(), unet.UNet.__new__(unet.UNet)
    buf = lambda: torch.zeros(8)
    net.torch = types.SimpleNamespace(cuda=cuda, device=torch.device, Tensor=torch.Tensor)
    net.hq, net.dev, net.cfg, net.cont, net.a_bits = hq, torch.device("cuda"), dict(groups=32), 1, 4
    net.calibrating, net.recording, net.graph, net.graph_key = False, None, None, None
    net.pw = {n: hq.PreparedWeight(hq.WeightDesc(N=8), None, None) for n in "ab"}
    for pw in net.pw.values():
        pw.blob_dev, pw.s_w_dev = buf(), buf()
    net.f32, net.bf, net.static = {"a.b": buf()}, {"label_emb": buf()}, {"a": buf()}
    for name in ("scratch", "status", "x_in", "t_in", "y_in", "eps_out"):
        setattr(net, name, buf())
    net.ws = Workspace(torch.zeros(64, dtype=torch.uint8))
    net.layers = list(net.pw.values())
    net.operands = [*net.f32.values(), *net.bf.values(), *net.static.values()]
    bias = net.f32["a.b"]

    def call(pw):
        at = lambda v: 0 if v is None else v.data_ptr()
        cuda.launch((net.a_bits, hq._pair_gemm_mode, bytes(pw.desc), at(pw.blob_dev), at(pw.s_w_dev), bias.data_ptr(), net.ws.data_ptr(),
                     net.ws.nbytes, at(net.scratch), at(net.status), at(net.x_in), at(net.eps_out), cuda.device))

    net.tape = [("q", n, lambda pw=pw: call(pw)) for n, pw in net.pw.items()]
    return net, cuda


def forward(net, cuda):
    cuda.log = []
    net.replay()
    got, cuda.log = cuda.log, []
    net.run()
    assert got == cuda.log


def change(net, cuda, what):
    pw = net.pw["a"]
    if what == "weights":
        pw.blob_dev = torch.zeros(8)
    elif what == "weight scales":
        pw.s_w_dev = torch.zeros(8)
    elif what == "descriptor":
        pw.desc.reserved = 1
    elif what in ("status", "scratch", "x_in", "eps_out"):
        setattr(net, what, torch.zeros(8))
    elif what == "no status":
        net.status = None
    elif what == "storage of a bias":
        net.f32["a.b"].data = torch.zeros(8)
    elif what == "smaller workspace":
        net.ws = Workspace(net.ws[:32])
    elif what == "another call":
        net.tape[1] = ("g", "other", lambda: cuda.launch("other"))
    elif what == "kernel choice":
        net.hq.hq_set_pair_gemm(0)
    elif what == "another device current":
        cuda.device = 1
    else:
        net.a_bits = 8


@pytest.mark.parametrize("what", ["weights", "weight scales", "descriptor", "status", "no status", "scratch", "x_in", "eps_out",
                                  "storage of a bias", "smaller workspace", "another call", "kernel choice",
                                  "another device current", "a_bits"])
def test_a_captured_forward_is_dropped_when_its_calls_would_differ(what):
    net, cuda = make_net()
    for _ in range(3):
        forward(net, cuda)
    assert net.graph is not None
    kept = net.pw["a"].blob_dev, net.status, net.scratch      # their addresses are not handed out again
    before = net.hq.pair_gemm_mode()
    try:
        for _ in range(3):
            change(net, cuda, what)
            forward(net, cuda)
    finally:
        net.hq.hq_set_pair_gemm(before)
    del kept


def test_an_unchanged_forward_keeps_its_graph():
    net, cuda = make_net()
    forward(net, cuda)
    forward(net, cuda)
    graph = net.graph
    for _ in range(3):
        forward(net, cuda)
    assert graph is not None and net.graph is graph

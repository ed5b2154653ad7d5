"""A latent-diffusion UNet on the Hadamard-quantized layers: the layer list (shapes only) and the forward pass.

`quantized_layers` lists the quantized convolutions and linears of the network, for workloads that run them on their
own.  `UNet` runs one denoising step of the whole network: every call below is an entry point of the C library (the
quantized layers with their fused normalisation prologues, and the unquantized operations between them); this module
only decides the order of the calls and owns the buffers.

The noise-prediction network the method is applied to is a UNet over a latent image; every convolution except the
first and the last, and every linear layer, runs as the Hadamard-quantized layer.  This module walks the usual
encoder / middle / decoder structure and emits one record per quantized layer, so that the benchmark can run them
with synthetic activations and random weights:

  level l of the encoder: `res_blocks` residual blocks (3x3 conv, time-embedding linear, 3x3 conv, 1x1 skip conv when
  the channel count changes), each followed by a self-attention block (QKV linear, output projection) at the
  resolutions listed in `attn_resolutions`; a stride-2 3x3 convolution goes down to the next level;
  middle: residual block, attention, residual block;
  decoder: `res_blocks + 1` residual blocks per level, fed with the concatenation of the running tensor and the
  matching encoder output, attention as in the encoder, and a 3x3 convolution after each nearest-neighbour upsampling;
  the time embedding itself is a two-layer MLP.

Normalisation, activation functions, the attention product, up/down-sampling and the first / last convolution are
not quantized layers and are not listed.
"""
from __future__ import annotations


def quantized_layers(batch: int = 64, latent: int = 64, base: int = 256, mults=(1, 2, 3, 4), res_blocks: int = 2,
                     attn_resolutions=(32, 16, 8), had_block: int = 256) -> list[dict]:
    """One dict per quantized layer, in execution order.

    kind 'conv': Nb, H, W (INPUT size), C, Cout, R (1 or 3), stride, pad;  kind 'linear': M, K, N.
    Every record also carries `had_block`, `macs` (multiply-accumulates) and a `name`."""
    layers: list[dict] = []
    temb = 4 * base

    def conv(name, res, cin, cout, R=3, stride=1):
        ho = res // stride
        layers.append(dict(kind="conv", name=name, Nb=batch, H=res, W=res, C=cin, Cout=cout, R=R, stride=stride,
                           pad=R // 2, had_block=had_block, macs=batch * ho * ho * cout * R * R * cin))

    def linear(name, M, K, N):
        layers.append(dict(kind="linear", name=name, M=M, K=K, N=N, had_block=min(had_block, K),
                           macs=M * N * K))

    def resblock(name, res, cin, cout):
        conv(f"{name}.conv1", res, cin, cout)
        linear(f"{name}.emb", batch, temb, cout)
        conv(f"{name}.conv2", res, cout, cout)
        if cin != cout:
            conv(f"{name}.skip", res, cin, cout, R=1)

    def attention(name, res, ch):
        linear(f"{name}.qkv", batch * res * res, ch, 3 * ch)
        linear(f"{name}.proj", batch * res * res, ch, ch)

    linear("time_embed.0", batch, base, temb)
    linear("time_embed.2", batch, temb, temb)

    ch, res = base, latent
    skips = [ch]                                   # output of the (unquantized) first convolution
    for lvl, m in enumerate(mults):
        for b in range(res_blocks):
            resblock(f"down{lvl}.res{b}", res, ch, m * base)
            ch = m * base
            if res in attn_resolutions:
                attention(f"down{lvl}.attn{b}", res, ch)
            skips.append(ch)
        if lvl + 1 < len(mults):
            conv(f"down{lvl}.downsample", res, ch, ch, R=3, stride=2)
            res //= 2
            skips.append(ch)
    resblock("mid.res0", res, ch, ch)
    attention("mid.attn", res, ch)
    resblock("mid.res1", res, ch, ch)
    for lvl in reversed(range(len(mults))):
        m = mults[lvl]
        for b in range(res_blocks + 1):
            resblock(f"up{lvl}.res{b}", res, ch + skips.pop(), m * base)
            ch = m * base
            if res in attn_resolutions:
                attention(f"up{lvl}.attn{b}", res, ch)
        if lvl > 0:
            res *= 2
            conv(f"up{lvl}.upsample", res, ch, ch)
    return layers


def distinct_shapes(layers: list[dict]) -> list[tuple]:
    """The set of distinct layer shapes, as sortable tuples."""
    out = set()
    for L in layers:
        if L["kind"] == "conv":
            out.add(("conv", L["Nb"], L["H"], L["C"], L["Cout"], L["R"], L["stride"]))
        else:
            out.add(("linear", L["M"], L["K"], L["N"]))
    return sorted(out)


class UNet:
    """One denoising step eps = net(x, t, y) of the network `inputs.unet_config` describes.

    Every convolution except the first and the last, and every linear, is a Hadamard-quantized layer (W4, `a_bits`
    activations, folded weights).  3x3 convolutions take one static activation scale each (the per-layer learned scale
    of the method; here calibrated once by `calibrate`), 1x1 convolutions and linears one dynamic scale per row.
    GroupNorm + SiLU in front of a residual block's convolutions and GroupNorm in front of an attention block's QKV
    projection are fused into the quantized layer's transform kernel.  Activations are bf16 NHWC.

    `build(Nb)` allocates every buffer and records the sequence of library calls; `run` replays it.  Calls are tagged
    "q" (a quantized layer, including its fused normalisation) or "g" (everything else), so that the two parts can be
    timed separately on the buffers of a complete forward."""

    EPS = 1e-5

    def __init__(self, cfg: dict, params: dict, hq, device, container: int | None = None, a_bits: int = 4):
        import torch
        self.torch, self.hq, self.cfg, self.dev, self.a_bits = torch, hq, cfg, device, a_bits
        self.cont = hq.HQ_CODES_INT8 if container is None else container
        self.had = cfg["had_block"]
        self.pw, self.f32, self.bf = {}, {}, {}
        for name, arr in params.items():
            stem, leaf = name.rsplit(".", 1) if "." in name else (name, "")
            if name == "label_emb":
                self.bf[name] = torch.from_numpy(arr).to(device).to(torch.bfloat16)
            elif leaf == "w" and stem not in ("in_conv", "out_conv"):
                K = arr.shape[-1]
                hb = self.had if K % self.had == 0 else 1
                self.pw[stem] = hq.hq_weight_prepare(arr, 4, hb, hq.HQ_W_FOLDED, self.cont).to_device(device)
            else:
                self.f32[name] = torch.from_numpy(arr).to(device)
        self.static = {}            # name of a 3x3 convolution -> device tensor [1]
        self.status = torch.zeros((1,), dtype=torch.int32, device=device)
        self.tape = []
        self.calibrating = False
        self.recording = None
        self.graph, self.graph_key = None, None
        self._group_embeddings()

    def _group_embeddings(self):
        """The projections of the step embedding, one per residual block and all of the same input, laid out as one layer: their
        weights, weight scales and biases become views of tensors that hold all of them, so that a forward projects once."""
        self.emb = None
        names = [n for n in self.pw if n.endswith(".emb")]
        shape = lambda d: (d.C, d.C_pad, d.RS, d.w_bits, d.had_block, d.mode, d.limbs, d.container)
        descs = [self.pw[n].desc for n in names]
        if len(names) < 2 or len({shape(d) for d in descs}) > 1 or any(d.N % 128 for d in descs):
            return
        rows = [d.N * d.limbs * d.C_pad for d in descs]                 # whole 128-row groups follow one another in a blob
        cat = self.torch.cat
        whole = self.hq.PreparedWeight(type(descs[0]).from_buffer_copy(descs[0]), None, None)
        whole.blob_dev = cat([self.pw[n].blob_dev[:r] for n, r in zip(names, rows)])
        whole.s_w_dev = cat([self.pw[n].s_w_dev for n in names])
        bias = cat([self.f32[n + ".b"] for n in names])
        whole.desc.N = whole.desc.N_pad = sum(d.N for d in descs)
        whole.desc.bytes, whole.desc.reserved = sum(rows), 0            # without the one-limb section: Nb rows never use it
        whole.desc.max_abs_b = max(d.max_abs_b for d in descs)
        at, byte, start = 0, 0, {}
        for n, d, r in zip(names, descs, rows):
            pw = self.pw[n]
            pw.blob_dev, pw.s_w_dev, self.f32[n + ".b"] = whole.blob_dev[byte:byte + r], whole.s_w_dev[at:at + d.N], bias[at:at + d.N]
            d.bytes, d.reserved = r, 0
            start[n] = at
            at, byte = at + d.N, byte + r
        self.emb = (whole, bias, start)
        self.emb_key = self._emb_operands()

    def _emb_operands(self):
        return [(pw.blob_dev.data_ptr(), pw.s_w_dev.data_ptr(), self.f32[n + ".b"].data_ptr(), bytes(pw.desc))
                for n, pw in ((n, self.pw[n]) for n in self.emb[2])]

    def _emb_together(self):
        """Whether this run projects the step embedding for all blocks at once: not while calls are recorded or calibrated one by
        one, and not once a block has been given operands elsewhere."""
        return self.recording is None and not self.calibrating and self._emb_operands() == self.emb_key

    # ------------------------------------------------------------------ recording helpers
    def _emit(self, tag, name, fn, rec=None):
        """Adds one library call to the tape.  rec: () -> dict of tensors to keep when a recording is requested."""
        def call():
            fn()
            if self.recording is not None and rec is not None:
                self.torch.cuda.synchronize()
                self.recording.append(dict(name=name, **{k: (v.clone() if hasattr(v, "clone") else v) for k, v in rec().items()}))
        self.tape.append((tag, name, call))

    def _new(self, shape, dtype=None):
        return self.torch.empty(shape, dtype=dtype or self.torch.bfloat16, device=self.dev)

    def _need_ws(self, pw, rows, static=False, stride=1):
        # for 4-bit codes too, whose layers use more of it: `a_bits` may be changed after the build
        self._ws_need = max(self._ws_need, *(self.hq.hq_layer_workspace_size(pw, b, rows, static, stride) for b in (self.a_bits, 4)))

    def _ws_views(self, rows, cols):
        row_bytes = cols // 2 if self.cont == self.hq.HQ_CODES_NIBBLE else cols
        pitch = (row_bytes + 15) // 16 * 16
        off = (rows * pitch + 255) // 256 * 256
        return self.ws[: rows * pitch].view(rows, pitch), self.ws[off: off + rows * 4].view(self.torch.float32)

    # ------------------------------------------------------------------ layers
    def _conv3(self, name, x, norm=None, stride=1, pre_bias=None, x2=None, residual=None):
        """x2: the layer's input is the channel concatenation [x | x2], which is read in place and never written.  pre_bias: a
        function that gives the addend in front of the normalisation.  residual: added to the output as it is stored; a recorded forward leaves the addition to `_residual`."""
        hq, t = self.hq, self.torch
        Nb, H, W, Cin = x.shape
        Cin += x2.shape[3] if x2 is not None else 0
        pw = self.pw[name]
        self._need_ws(pw, Nb * H * W, static=True, stride=stride)
        y, plain = self._output((Nb, H // stride, W // stride, pw.desc.N), residual)
        bias = self.f32[name + ".b"]
        ss = self.static.setdefault(name, t.ones((1,), dtype=t.float32, device=self.dev))
        g = (self.f32[norm + ".gamma"], self.f32[norm + ".beta"]) if norm else None
        G = self.cfg["groups"]
        addend = pre_bias or (lambda: None)

        def calibrate():
            if not self.calibrating:
                return
            codes, sc = self._ws_views(Nb * H * W, Cin)
            if g:
                hq.hq_gn_silu_quant(x, G, g[0], g[1], self.EPS, pw.desc.had_block, self.a_bits, codes, self.cont, self.scratch,
                                    scales=sc, pre_bias=addend(), x2=x2)
            else:
                hq.hq_hadamard_quant(x.view(-1, x.shape[3]), pw.desc.had_block, self.a_bits, codes, self.cont, scales=sc,
                                     x2=None if x2 is None else x2.view(-1, x2.shape[3]))
            ss.copy_(sc.max().reshape(1))

        def run():
            calibrate()
            if g:
                fused = residual is not None and self.recording is None
                hq.hq_gn_silu_qconv(x, G, g[0], g[1], self.EPS, pw, 3, 3, stride, 1, bias, self.a_bits, y if fused else plain(), self.ws,
                                    self.scratch, static_scale=ss, dev_status=self.status, pre_bias=addend(), x2=x2,
                                    residual=residual if fused else None)
            else:
                hq.hq_qconv(x, pw, 3, 3, stride, 1, bias, self.a_bits, plain(), self.ws, static_scale=ss, dev_status=self.status,
                            x2=x2)

        self._emit("q", name, run, lambda: dict(op="conv3", x=x, x2=x2, y=plain(), norm=norm, stride=stride, static=ss, pre_bias=addend(),
                                                codes=self._ws_views(Nb * H * W, Cin)[0]))
        return y if residual is None else (y, plain)

    def _conv1(self, name, x, x2=None):
        hq = self.hq
        Nb, H, W, Cin = x.shape
        Cin += x2.shape[3] if x2 is not None else 0
        pw = self.pw[name]
        self._need_ws(pw, Nb * H * W)
        y = self._new((Nb, H, W, pw.desc.N))
        bias = self.f32[name + ".b"]
        self._emit("q", name, lambda: hq.hq_qconv(x, pw, 1, 1, 1, 0, bias, self.a_bits, y, self.ws, dev_status=self.status,
                                                      x2=x2),
                   lambda: dict(op="conv1", x=x, x2=x2, y=y, codes=self._ws_views(Nb * H * W, Cin)[0],
                                scales=self._ws_views(Nb * H * W, Cin)[1]))
        return y

    def _linear(self, name, x, norm=None, Nb=None, residual=None):
        hq = self.hq
        M, K = x.shape
        pw = self.pw[name]
        self._need_ws(pw, M)
        y, plain = self._output((M, pw.desc.N), residual)
        bias = self.f32[name + ".b"]
        if norm:
            gm, bt = self.f32[norm + ".gamma"], self.f32[norm + ".beta"]
            fn = lambda: hq.hq_gn_qlinear(x, Nb, self.cfg["groups"], gm, bt, self.EPS, False, pw, bias, self.a_bits, y, self.ws,
                                          self.scratch, dev_status=self.status)
        else:
            def fn():
                fused = residual is not None and self.recording is None
                hq.hq_qlinear(x, pw, bias, self.a_bits, y if fused else plain(), self.ws, dev_status=self.status,
                              residual=residual if fused else None)
        self._emit("q", name, fn, lambda: dict(op="linear", x=x, y=plain(), norm=norm, Nb=Nb, codes=self._ws_views(M, K)[0],
                                               scales=self._ws_views(M, K)[1]))
        return y if residual is None else (y, plain)

    def _embedding(self, name, x):
        """A block's projection of the step embedding; returns a function that gives its [Nb, C] (rows of a wider tensor where all
        blocks' projections are made at once, by the first of them)."""
        hq = self.hq
        if self.emb is None:
            e = self._linear(name, x)
            return lambda: e
        (whole, bias_all, start), pw, bias = self.emb, self.pw[name], self.f32[name + ".b"]
        M, K = x.shape
        self._need_ws(pw, M)
        first = self.emb_out is None
        if first:
            self._need_ws(whole, M)
            self.emb_out = self._new((M, whole.desc.N))
        out, rows = self.emb_out, self.emb_out[:, start[name]:start[name] + pw.desc.N]
        apart = self._later((M, pw.desc.N))

        def fn():
            if first:                                                   # once for all blocks of a run
                self.emb_joined = self._emb_together()
            if not self.emb_joined:
                hq.hq_qlinear(x, pw, bias, self.a_bits, apart(), self.ws, dev_status=self.status)
            elif first:
                hq.hq_qlinear(x, whole, bias_all, self.a_bits, out, self.ws, dev_status=self.status)
        self._emit("q", name, fn, lambda: dict(op="linear", x=x, y=apart(), norm=None, Nb=None, codes=self._ws_views(M, K)[0],
                                               scales=self._ws_views(M, K)[1]))
        return lambda: rows if self.emb_joined else apart()

    def _output(self, shape, residual):
        """A layer's output, and a function that gives the buffer of its output before the residual is added: the output itself
        without one, else a buffer that only a recorded forward, which takes the two steps apart, makes."""
        y = self._new(shape)
        return y, (lambda: y) if residual is None else self._later(shape)

    def _later(self, shape):
        """A function that gives a buffer and makes it when it is first asked for."""
        made = []

        def buffer():
            if not made:
                made.append(self._new(shape))
            return made[0]
        return buffer

    def _residual(self, name, a, out, plain):
        """The addition out = a + plain(), which the layer that produces the sum has done except in a recorded forward."""
        hq = self.hq

        def fn():
            if self.recording is not None:
                hq.hq_add(a, plain(), out)
        self._emit("g", name, fn, lambda: dict(op="add", a=a, b=plain(), out=out))

    def _glue(self, name, op, fn, **tensors):
        self._emit("g", name, fn, lambda: dict(op=op, **tensors))

    def _resblock(self, name, x, semb, x2=None):
        """x2: the block's input is the channel concatenation [x | x2] (a skip connection joining the up-sampling path);
        its two consumers, the first convolution and the 1x1 skip convolution, read the two tensors in place."""
        cin, cout = x.shape[-1] + (x2.shape[-1] if x2 is not None else 0), self.pw[name + ".conv1"].desc.N
        h = self._conv3(name + ".conv1", x, norm=name + ".norm1", x2=x2)
        e = self._embedding(name + ".emb", semb)
        assert x2 is None or cin != cout       # a concatenated input always changes the channel count here
        xs = x if cin == cout else self._conv1(name + ".skip", x, x2=x2)
        # h + e is never stored: the second convolution's normalisation takes the embedding as a per-sample addend; nor is its own
        # output, to which the block's input (or its 1x1 convolution) is added as it is stored
        out, plain = self._conv3(name + ".conv2", h, norm=name + ".norm2", pre_bias=e, residual=xs)
        self._residual(name + ".residual", xs, out, plain)
        return out

    def _attention(self, name, x):
        hq = self.hq
        Nb, H, W, ch = x.shape
        x2 = x.view(Nb * H * W, ch)
        qkv = self._linear(name + ".qkv", x2, norm=name + ".norm", Nb=Nb)
        a = self._new((Nb * H * W, ch))
        heads = self.cfg["heads"]
        self.attn_flops += 4.0 * Nb * float(H * W) ** 2 * ch
        self._glue(name + ".core", "attention", lambda: hq.hq_attention(qkv, Nb, heads, a, dev_status=self.status),
                   qkv=qkv, out=a, Nb=Nb, heads=heads)
        out, plain = self._linear(name + ".proj", a, residual=x2)
        self._residual(name + ".residual", x2, out, plain)
        return out.view(x.shape)

    # ------------------------------------------------------------------ the network
    def build(self, Nb: int):
        """Allocates the buffers of a forward at batch Nb and records its sequence of library calls."""
        t, hq, cfg = self.torch, self.hq, self.cfg
        S, base, mults, nres = cfg["latent"], cfg["base"], cfg["mults"], cfg["res_blocks"]
        temb = 4 * base
        self.tape = []
        self.graph, self.graph_key = None, None
        self.Nb = Nb
        self.emb_out = None            # [Nb, channels of all blocks]: the projections of the step embedding,
        self.emb_joined = False        # where the running pass made them at once
        self.attn_flops = 0.0          # 4 L^2 C per sample and attention block (QK^T and PV)
        self._ws_need = 256
        self.scratch = t.empty((Nb * cfg["groups"] * 24,), dtype=t.uint8, device=self.dev)
        self.x_in = t.empty((Nb, S, S, cfg["in_ch"]), dtype=t.bfloat16, device=self.dev)
        self.t_in = t.empty((Nb,), dtype=t.float32, device=self.dev)
        self.y_in = t.empty((Nb,), dtype=t.int32, device=self.dev)

        te = self._new((Nb, base))
        self._glue("time_embed.sin", "timestep_embedding", lambda: hq.hq_timestep_embedding(self.t_in, te), t=self.t_in, out=te)
        e1 = self._linear("time_embed.0", te)
        e1s = self._new(e1.shape)
        self._glue("time_embed.act", "silu", lambda: hq.hq_silu(e1, e1s), x=e1, out=e1s)
        emb = self._linear("time_embed.2", e1s)
        table = self.bf["label_emb"]
        self._glue("label_emb.add", "class_embed_add", lambda: hq.hq_class_embed_add(emb, table, self.y_in),
                   labels=self.y_in, out=emb)
        semb = self._new(emb.shape)
        self._glue("emb.act", "silu", lambda: hq.hq_silu(emb, semb), x=emb, out=semb)

        h = self._new((Nb, S, S, base))
        w_in, b_in = self.f32["in_conv.w"], self.f32["in_conv.b"]
        self._glue("in_conv", "conv_float", (lambda o=h: hq.hq_conv2d_direct(self.x_in, w_in, b_in, 3, 1, 1, o)), x=self.x_in,
                   out=h)
        ch, res = base, S
        skips = [h]
        for lvl, m in enumerate(mults):
            for b in range(nres):
                h = self._resblock(f"down{lvl}.res{b}", h, semb)
                if res in cfg["attn_resolutions"]:
                    h = self._attention(f"down{lvl}.attn{b}", h)
                skips.append(h)
            if lvl + 1 < len(mults):
                h = self._conv3(f"down{lvl}.downsample", h, stride=2)
                res //= 2
                skips.append(h)
        h = self._resblock("mid.res0", h, semb)
        h = self._attention("mid.attn", h)
        h = self._resblock("mid.res1", h, semb)
        for lvl in reversed(range(len(mults))):
            for b in range(nres + 1):
                sk = skips.pop()
                h = self._resblock(f"up{lvl}.res{b}", h, semb, x2=sk)         # [h | skip], never written out
                if res in cfg["attn_resolutions"]:
                    h = self._attention(f"up{lvl}.attn{b}", h)
            if lvl > 0:
                up = self._new((Nb, 2 * res, 2 * res, h.shape[3]))
                self._glue(f"up{lvl}.upsample.nearest", "upsample", (lambda a=h, o=up: hq.hq_upsample_nearest2x(a, o)), x=h, out=up)
                res *= 2
                h = self._conv3(f"up{lvl}.upsample", up)
        hn = self._new(h.shape)
        gm, bt = self.f32["out_norm.gamma"], self.f32["out_norm.beta"]
        self._glue("out_norm", "groupnorm_silu", (lambda a=h: hq.hq_groupnorm_act(a, cfg["groups"], gm, bt, self.EPS, True, hn,
                                                                                   self.scratch)), x=h, out=hn)
        self.eps_out = t.empty((Nb, S, S, cfg["in_ch"]), dtype=t.float32, device=self.dev)
        w_o, b_o = self.f32["out_conv.w"], self.f32["out_conv.b"]
        self._glue("out_conv", "conv_float", lambda: hq.hq_conv2d_direct(hn, w_o, b_o, 3, 1, 1, self.eps_out), x=hn,
                   out=self.eps_out)
        # one workspace for the codes and scales of whichever quantized layer is running (sized for the largest)
        self.ws = t.empty((self._ws_need,), dtype=t.uint8, device=self.dev)
        # what the recorded calls read beside the buffers made here: `replay` looks whether it is still what it captured
        self.layers = list(self.pw.values())
        self.operands = [*self.f32.values(), *self.bf.values(), *self.static.values()]
        return self

    def set_inputs(self, x, t, y):
        """x NHWC (any float dtype), t [Nb] denoising steps, y [Nb] class labels (device or host tensors)."""
        self.x_in.copy_(x)
        self.t_in.copy_(t)
        self.y_in.copy_(y)

    def run(self, tags=("q", "g")):
        for tag, _, call in self.tape:
            if tag in tags:
                call()

    def calibrate(self, x, t, y):
        """One forward in which every 3x3 convolution first measures its input: its static activation scale becomes the
        largest per-pixel scale of that input."""
        self.set_inputs(x, t, y)
        self.calibrating = True
        try:
            self.run()
        finally:
            self.calibrating = False
        self.torch.cuda.synchronize()
        self.hq.hq_check_status(self.status)

    def _looked_up(self):
        """Everything the recorded calls look up anew each time they run: a graph of them is what they are as long as this
        compares equal (about 40 us; a weight put on the device again, another status word or another kernel choice differs)."""
        tensors = [self.ws, self.scratch, self.status, self.x_in, self.t_in, self.y_in, self.eps_out, *self.operands]
        for pw in self.layers:
            tensors += (pw.blob_dev, pw.s_w_dev)
        tensors = [v for v in tensors if v is not None]
        return (self.a_bits, self.cont, self.EPS, self.cfg["groups"], self.hq.pair_gemm_mode(), self.ws.nbytes, self.scratch.nbytes,
                tuple(self.tape), b"".join(pw.desc for pw in self.layers), list(map(self.torch.Tensor.data_ptr, tensors)))

    def replay(self):
        """`run()` with its launches kept as a CUDA graph.  The calls of a forward and their buffers are fixed by `build`, and
        at small batches issuing them from the host takes longer than the device needs (2 images: 2.9 ms for 2.4 ms of
        kernels).  The first forward after a build runs the calls themselves, the second one captures them; any change of what
        the calls look up starts over.  Inside a caller's own capture, or with another device current, the calls run as they
        are."""
        t = self.torch
        if self.calibrating or self.ws.device.index != t.cuda.current_device() or t.cuda.is_current_stream_capturing():
            self.run()
            return
        key = self._looked_up()
        if self.graph_key != key:
            self.run()
            self.graph, self.graph_key = None, key
            return
        if self.graph is None:
            graph, stream = t.cuda.CUDAGraph(), t.cuda.Stream()
            stream.wait_stream(t.cuda.current_stream())
            with t.cuda.stream(stream):
                graph.capture_begin(capture_error_mode="thread_local")
                try:
                    self.run()
                finally:
                    graph.capture_end()
            t.cuda.current_stream().wait_stream(stream)
            self.graph = graph
        self.graph.replay()

    def forward(self, x, t, y, record=None):
        """eps [Nb, S, S, in_ch] fp32.  record: a list that receives, per library call, its name and copies of the tensors
        it read and wrote (for layer-by-layer checks)."""
        self.set_inputs(x, t, y)
        if record is None:
            self.replay()
            return self.eps_out
        self.recording = record
        try:
            self.run()
        finally:
            self.recording = None
        return self.eps_out

"""Timed cases of the acoustic-encoder library: what its users call, over the sizes they call it with.

Three kinds of pass, all through the package's Python entry points:

  block   one block forward + backward (sepconv_fwd, sepconv_bwd): a training loop built from single blocks
  train   one training step of the QuartzNet-5x5-style encoder (encoder_fwd_bwd)
  infer   one evaluation-mode pass of that encoder ending in log-probabilities (encoder_infer)

Inputs and upstream gradients are N(0,1), weights Kaiming-uniform, per-sample lengths uniform in [len_lo, T] with the
longest sample filling the batch, as a padded batch does.  Plans (descriptors, layer lists), parameters, workspaces and
gradient buffers are made once in prepare(), as a training or serving program keeps them.
"""
import torch
import torch.nn.functional as F

import paper_1909_09577_b200 as api
import synth_inputs as si

DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
CONV_WEIGHTS = ("wd", "wp", "wr")


# ---- cases ----------------------------------------------------------------------------------------------------------
def _block(dtype, B, C_in, C_out, T, K, len_lo, residual="none", stride=1, dilation=1, full_conv=False):
    return {"kind": "block", "dtype": dtype, "B": B, "C_in": C_in, "C_out": C_out, "T": T, "K": K, "len_lo": len_lo,
            "residual": residual, "stride": stride, "dilation": dilation, "full_conv": full_conv}


def _train(dtype, B, T, len_lo):
    return {"kind": "train", "dtype": dtype, "B": B, "T": T, "len_lo": len_lo}


def _infer(B, T, len_lo):
    return {"kind": "infer", "dtype": "f16", "B": B, "T": T, "len_lo": len_lo}


def listed():
    cases = {
        # a two-sample fp32 block (parity configuration 1): nothing but launches and host work
        "block_f32_small": _block("f32", 2, 64, 64, 128, 33, 128, residual="identity"),
        # an fp16 block of the first encoder stage on a ragged batch (parity configuration 2)
        "block_f16_ragged": _block("f16", 32, 256, 256, 400, 33, 200, residual="identity"),
        # a bf16 block that widens, with the projected residual (parity configuration 3)
        "block_bf16_proj": _block("bf16", 32, 256, 512, 400, 63, 100, residual="proj"),
        # the same kind of block on a batch padded only to its longest utterance: an odd frame count and batch
        "block_bf16_odd": _block("bf16", 23, 384, 384, 797, 39, 200, residual="proj"),
        # the encoder's striding first layer on its own
        "block_bf16_stride2": _block("bf16", 32, 64, 256, 1600, 33, 400, stride=2),
        # the encoder's widest block with dilated taps (the block variant)
        "block_bf16_dilated": _block("bf16", 16, 512, 512, 800, 87, 200, dilation=2),
        # the original Jasper block's dense convolution (the block variant)
        "block_f16_full_conv": _block("f16", 16, 256, 256, 400, 11, 100, full_conv=True),
        # the benchmark's training step: 32 full-length samples of 1600 frames (configuration 4)
        "train_full": _train("bf16", 32, 1600, 1600),
        # the large ragged training step (configuration 5)
        "train_ragged": _train("bf16", 64, 3200, 200),
        # recognising one short command: latency only
        "infer_chunk": _infer(1, 161, 161),
        # one ten-second utterance
        "infer_utterance": _infer(1, 1001, 1001),
        # offline recognition of a ragged batch, padded to its longest utterance
        "infer_batch": _infer(32, 1237, 300),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return min(hi, int(lo * (hi / lo) ** rng.random() + 0.5))


def draw(rng):
    kind = rng.choices(("block16", "block32", "full_conv", "train", "infer"), weights=(8, 2, 2, 3, 5))[0]
    if kind == "block32":
        C, T = rng.choice((32, 64, 96, 128)), _log_int(rng, 64, 320)
        return _block("f32", rng.randint(2, 8), C, C, T, rng.randrange(5, 41, 2), rng.randint(T // 2, T),
                      residual=rng.choice(("none", "identity")))
    if kind == "block16":
        stride, dilation = rng.choices(((1, 1), (2, 1), (1, 2)), weights=(6, 1, 1))[0]
        T = _log_int(rng, 100, 1600)
        widths = (64, 128, 192, 256, 320, 384, 512)
        return _block(rng.choice(("bf16", "f16")), _log_int(rng, 2, 48), rng.choice(widths), rng.choice(widths), T,
                      rng.randrange(11, 89, 2), rng.randint(T // 4, T), stride=stride, dilation=dilation,
                      residual="none" if stride == 2 else rng.choice(("none", "proj")))
    if kind == "full_conv":
        T = _log_int(rng, 100, 600)
        widths = (64, 128, 192, 256)
        return _block(rng.choice(("bf16", "f16")), _log_int(rng, 2, 24), rng.choice(widths), rng.choice(widths), T,
                      rng.randrange(5, 30, 2), rng.randint(T // 4, T), full_conv=True, residual=rng.choice(("none", "proj")))
    if kind == "train":
        B = _log_int(rng, 16, 64)
        T = 16 * _log_int(rng, 25, min(200, 204800 // (16 * B)))     # training batches are padded to a multiple of 16 frames
        return _train(rng.choice(("bf16", "f16")), B, T, rng.choice((T, T // 2, T // 8)))
    B = _log_int(rng, 1, 32)
    T = _log_int(rng, 100, min(3200, 102400 // B))
    return _infer(B, T, T if B == 1 else rng.randint(T // 4, T))


# ---- inputs ---------------------------------------------------------------------------------------------------------
_contexts = {}


def _context():
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = api.Context(dev)
    return _contexts[dev]


def _layers(case):
    if case["kind"] != "block":
        return si.quartznet5x5_layers(log_probs=case["kind"] == "infer")
    return [si.LayerCfg(case["C_in"], case["C_out"], K=case["K"], stride=case["stride"], residual=case["residual"],
                        dilation=case["dilation"], has_dw=not case["full_conv"], full_conv=case["full_conv"])]


def _fan_in(L, name):
    return {"wd": L.K, "wp": L.C_in * (L.K if L.full_conv else 1), "wr": L.C_res}[name]


def _fill(t, L, name, gen, trained):
    """Draws one parameter into the tensor t.  trained: scales around one and mostly positive shifts, as training leaves
    them; otherwise the scales and shifts that training starts from."""
    if name in CONV_WEIGHTS:
        b = (6.0 / _fan_in(L, name)) ** 0.5
        t.copy_((torch.rand(t.shape, generator=gen, device="cuda") * 2 - 1) * b)
    elif name in ("gamma", "gamma_r"):
        t.copy_(torch.rand(t.shape, generator=gen, device="cuda") + 0.5 if trained else torch.ones_like(t))
    else:
        t.copy_(torch.rand(t.shape, generator=gen, device="cuda") if trained else torch.zeros_like(t))


def _lengths(case, gen):
    n = torch.randint(case["len_lo"], case["T"] + 1, (case["B"],), generator=gen, device="cuda", dtype=torch.int32)
    n[0] = case["T"]
    return n


def _normal(shape, dtype, gen):
    return torch.randn(shape, generator=gen, device="cuda").to(dtype)


def _running_statistics(layers, param, gen):
    """The batch statistics that a network with these parameters shows on inputs of the expected kind: what the running
    averages of a trained network hold.  Plain float32 torch on a small batch."""
    stats, inputs = [], []
    y = torch.randn((2, layers[0].C_in, 256), generator=gen, device="cuda")
    for i, L in enumerate(layers):
        inputs.append(y)
        p = lambda n: param(i, n).float()
        u = F.conv1d(y, p("wd")[:, None], stride=L.stride, padding=(L.K - 1) // 2, groups=L.C_in) if L.has_dw else y
        v = torch.matmul(p("wp"), u)
        if not L.has_bn:
            stats.append(None)
            continue
        z, s = 0.0, {}
        for r, q in (("", v),) + ((("_r", torch.matmul(p("wr"), inputs[L.res_from])),) if L.residual == "proj" else ()):
            mean, var = q.mean((0, 2)), q.var((0, 2), unbiased=False)
            s["mean" + r], s["var" + r] = mean.cpu().numpy(), var.cpu().numpy()
            z = z + (p("gamma" + r) / (var + L.eps).sqrt())[:, None] * (q - mean[:, None]) + p("beta" + r)[:, None]
        stats.append(s)
        y = torch.relu(z)
    return stats


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    td, B, T, layers = DTYPE[case["dtype"]], case["B"], case["T"], _layers(case)
    s = {"kind": case["kind"], "ctx": _context(), "lengths": _lengths(case, gen),
         "x": _normal((B, layers[0].C_in, T), td, gen)}
    if case["kind"] == "block":
        L = layers[0]
        params = {}
        for name, shape in L.param_shapes().items():
            params[name] = torch.empty(shape, dtype=td if name in CONV_WEIGHTS else torch.float32, device="cuda")
            _fill(params[name], L, name, gen, trained=False)
        desc = api.block_desc(L, B, T, case["dtype"])
        fwd, bwd = api.sepconv_workspace_bytes(desc)
        s.update(desc=desc, params=params, dy=_normal((B, L.C_out, desc.T_out), td, gen),
                 running_mean=torch.zeros(L.C_out, device="cuda"), running_var=torch.ones(L.C_out, device="cuda"),
                 grads={"d" + n: torch.zeros(t.shape, device="cuda") for n, t in params.items()},
                 fwd_workspace=torch.empty(fwd, dtype=torch.uint8, device="cuda"),
                 bwd_workspace=torch.empty(bwd, dtype=torch.uint8, device="cuda"))
        return s
    spec = api.EncoderSpec(layers, B, T, case["dtype"])
    blob = torch.zeros(spec.param_bytes, dtype=torch.uint8, device="cuda")
    for i, L in enumerate(layers):
        for name in L.param_shapes():
            _fill(spec.param_view(blob, i, name), L, name, gen, trained=case["kind"] == "infer")
    s.update(spec=spec, blob=blob,
             workspace=torch.empty(api.encoder_workspace_bytes(spec), dtype=torch.uint8, device="cuda"))
    if case["kind"] == "train":
        s.update(dlogits=_normal((B, spec.C_out, spec.T_out), td, gen),
                 logits=torch.empty((B, spec.C_out, spec.T_out), dtype=td, device="cuda"),
                 grads=torch.zeros(spec.grad_bytes, dtype=torch.uint8, device="cuda"))
    else:
        running = _running_statistics(layers, lambda i, n: spec.param_view(blob, i, n), gen)
        s["running"], s["running_offsets"] = spec.pack_running(running, "cuda")
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    if s["kind"] == "block":
        y, out_len, saved = api.sepconv_fwd(s["ctx"], s["desc"], s["x"], s["lengths"], s["params"],
                                            running_mean=s["running_mean"], running_var=s["running_var"],
                                            workspace=s["fwd_workspace"])
        dx, _, grads = api.sepconv_bwd(s["ctx"], s["desc"], s["dy"], s["x"], y, s["lengths"], s["params"], saved,
                                       grads=s["grads"], workspace=s["bwd_workspace"])
        return {"y": y, "out_len": out_len, "dx": dx, "grads": grads, "running_mean": s["running_mean"],
                "running_var": s["running_var"]}
    if s["kind"] == "train":
        logits, out_len, grads, _ = api.encoder_fwd_bwd(s["ctx"], s["spec"], s["x"], s["lengths"], s["blob"], s["dlogits"],
                                                        grads_blob=s["grads"], workspace=s["workspace"], logits=s["logits"])
        return {"logits": logits, "out_len": out_len, "grads": grads.view(torch.float32)}
    out, out_len = api.encoder_infer(s["ctx"], s["spec"], s["x"], s["lengths"], s["blob"], s["running"],
                                     s["running_offsets"], workspace=s["workspace"])
    return {"log_probs": out, "out_len": out_len}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    """Bytes: activations, upstream gradients, results, parameters and their gradients, once each.  Flops: the
    contractions on the frames that hold data (lengths at the mean of their range), forward once and, in a training
    pass, twice more for the two gradients."""
    layers, B, T = _layers(case), case["B"], case["T"]
    e = 4 if case["dtype"] == "f32" else 2
    frac = (case["len_lo"] + T) / 2.0 / T
    train = case["kind"] != "infer"
    flops, pbytes, gbytes, t = 0.0, 0, 0, T
    for L in layers:
        t = (t - 1) // (L.stride if (L.has_dw or L.full_conv) else 1) + 1
        per_frame = 0
        for name, shape in L.param_shapes().items():
            n = 1
            for d in shape:
                n *= d
            pbytes += n * (e if name in CONV_WEIGHTS else 4)
            gbytes += n * 4
            if name in CONV_WEIGHTS:
                per_frame += 2 * n
        flops += per_frame * B * t * frac * (3 if train else 1)
    x, y = e * B * layers[0].C_in * T, e * B * layers[-1].C_out * t
    if case["kind"] == "block":
        return {"bytes": 2 * x + 2 * y + pbytes + gbytes, "flops": flops}      # x, dx; y, dy
    if case["kind"] == "train":
        return {"bytes": x + 2 * y + pbytes + gbytes, "flops": flops}          # x; logits, dlogits
    return {"bytes": x + y + pbytes, "flops": flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 2e-5}                   # float32 sums of up to some thousand terms, through one normalisation
    if case["kind"] == "block":
        # 16-bit results and operands; a pre-activation within a rounding of zero may fall on the other side of the
        # ReLU, which moves single gradient elements by their own size
        return {"rel": 1e-2, "max": 0.5}
    if case["kind"] == "infer":
        return {"rel": 1e-2, "max": 0.3}       # 29 layers of float16 activations
    # the gradient is rounded to 16 bits twice in each of 29 layers
    return {"rel": 2e-2, "max": 0.5}

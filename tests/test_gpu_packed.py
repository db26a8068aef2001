"""Blocks and encoders whose row length is not a multiple of 8 frames, or whose taps are two frames apart: these run on
packed copies through the tensor-core kernels.  Sizes at the edges: one frame, rows shorter than a vector, a row that ends
one frame short of or past a vector, batches on both sides of the 16-sample kernels."""
import pytest
import torch

import synth_inputs as si
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import paper_1909_09577_b200 as api
    return api


@pytest.fixture(scope="module")
def ctx(api):
    c = api.Context(0)
    yield c
    c.close()


CASES = [
    # (layer kwargs, B, T, shortest length)
    (dict(C_in=16, C_out=24, K=5, residual="proj"), 3, 9, 5),
    (dict(C_in=64, C_out=72, K=33, residual="proj"), 17, 271, 60),
    (dict(C_in=72, C_out=64, K=39), 16, 129, 1),
    (dict(C_in=32, C_out=32, K=11, residual="identity"), 18, 257, 100),
    (dict(C_in=40, C_out=136, K=15, stride=2), 5, 333, 90),
    (dict(C_in=16, C_out=16, K=9, stride=2), 33, 136, 30),                      # T a multiple of 8, T / 2 not
    (dict(C_in=64, C_out=48, K=1, has_dw=False), 4, 203, 50),
    (dict(C_in=64, C_out=64, K=87, dilation=2), 17, 400, 60),
    (dict(C_in=24, C_out=40, K=11, dilation=2, residual="proj"), 8, 161, 1),    # a length of one: an empty second phase
    (dict(C_in=32, C_out=32, K=7, dilation=2, residual="identity"), 20, 262, 31),
]


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_packed_blocks(api, ctx, dtype, case):
    kw, B, T, lo = CASES[case]
    L = si.LayerCfg(**kw)
    d = si.draw(si.Workload("packed", dtype, B, T, [L], 500 + case, len_lo=lo, len_hi=T, affine="random"))
    d.lengths[0], d.lengths[-1] = T, lo
    rep = U.run_block(ctx, api, L, dtype, d.x, d.lengths, d.params[0], d.g)
    print(f"\npacked case {case} {dtype}: {rep}")
    rep.check()


def compare_with_chain(spec, w, d, logits, out_len, grads, dx, chain):
    """Every result of a padded encoder against the chain of packed block calls.  The two differ where a layer without batch
    norm takes another kernel (its sums in another order), which moves an element of its bf16 input gradient by at most one
    unit, 2^-8 of it; that difference re-rounds once in every layer before it."""
    got = {"logits": (logits, chain["logits"]), "dx": (dx, chain["dx"])}
    for i in range(len(w.layers)):
        for name in d.params[i]:
            got[f"{i}.{name}"] = (spec.grad_view(grads, i, name), chain["grads"][i]["d" + name])
    err = {k: ((a.float() - b.float()).norm() / b.float().norm()).item() for k, (a, b) in got.items()}
    print("\npadded encoder against the chain:", {k: f"{e:.1e}" for k, e in err.items()})
    assert (out_len.cpu().numpy() == chain["out_len"]).all()
    assert max(err.values()) <= 2.0 ** -8 * len(w.layers) ** 0.5, err


@pytest.mark.parametrize("T", [497, 500])
def test_padded_encoder_equals_chain(api, ctx, T):
    """A whole encoder on rows that are no multiple of 8 frames against the chain of (packed) block calls."""
    w = si.tiny_encoder(dtype="bf16", B=18, T=T, ragged=True, width=32)
    d = si.draw(w)
    d.lengths[3] = T
    reports, chain = U.run_chain(ctx, api, w, d)
    spec = api.EncoderSpec(w.layers, w.B, w.T, w.dtype)
    blob = spec.pack_params(d.params, "cuda")
    logits, out_len, grads, dx = api.encoder_fwd_bwd(ctx, spec, U.dev(d.x, w.dtype), torch.from_numpy(d.lengths).cuda(), blob,
                                                     U.dev(d.g, w.dtype), want_dx=True)
    assert ctx.last_status() == 0
    scale = torch.as_tensor(chain["logits"]).float().pow(2).mean().sqrt()
    assert (logits.float() - chain["logits"].float()).abs().max() <= 0.1 * scale
    assert logits.shape[2] == spec.T_out and (out_len.cpu().numpy() == chain["out_len"]).all()
    assert (dx.float() - chain["dx"].float()).norm() <= 0.05 * chain["dx"].float().norm()
    compare_with_chain(spec, w, d, logits, out_len, grads, dx, chain)


def test_padded_encoder_starting_without_depthwise(api, ctx):
    """Padded rows into a first layer whose contraction follows the copies directly: its block offsets must be settled.  The
    workspace starts as zeros (an empty block list: nothing out of range is reachable, and the results would be zero)."""
    layers = [si.LayerCfg(16, 32, K=1, has_dw=False), si.LayerCfg(32, 32, K=7, stride=2),
              si.LayerCfg(32, 29, K=1, has_dw=False, has_bn=False, has_relu=False, has_bias=True)]
    w = si.Workload("padded_pointwise_first", "bf16", 18, 497, layers, 31, len_lo=120, len_hi=497, affine="random")
    d = si.draw(w)
    reports, chain = U.run_chain(ctx, api, w, d)
    spec = api.EncoderSpec(layers, w.B, w.T, w.dtype)
    blob, x, g = spec.pack_params(d.params, "cuda"), U.dev(d.x, w.dtype), U.dev(d.g, w.dtype)
    lens, ws = torch.from_numpy(d.lengths).cuda(), torch.empty(api.encoder_workspace_bytes(spec), dtype=torch.uint8, device="cuda")
    for call in range(2):
        ws.zero_()
        logits, out_len, grads, dx = api.encoder_fwd_bwd(ctx, spec, x, lens, blob, g, want_dx=True, workspace=ws)
        assert ctx.last_status() == 0
        compare_with_chain(spec, w, d, logits, out_len, grads, dx, chain)


@pytest.mark.parametrize("B,C,T,dilation", [(17, 24, 271, 1), (16, 150, 272, 1), (17, 24, 270, 2), (15, 256, 801, 1), (3, 24, 129, 1)])
def test_input_gradient_keeps_the_bits_of_its_taps(api, ctx, B, C, T, dilation):
    """bfloat16 taps of any magnitude: scaling them by a power of two scales the input gradient by exactly that (the kernels
    that take float16 operands must not round taps below 2^-14 or overflow above 65504)."""
    L = si.LayerCfg(C, 16, K=33, dilation=dilation)
    d = si.draw(si.Workload("taps", "bf16", B, T, [L], 77, len_lo=T // 2, len_hi=T))
    desc, x, g = api.block_desc(L, B, T, "bf16"), U.dev(d.x, "bf16"), U.dev(d.g, "bf16")
    lens, p = torch.from_numpy(d.lengths).cuda(), U.params_dev(d.params[0], "bf16")
    y, _, saved = api.sepconv_fwd(ctx, desc, x, lens, p)
    dx = api.sepconv_bwd(ctx, desc, g, x, y, lens, p, saved)[0]
    assert dx.float().abs().max() > 0
    for e in (-16, -24, 20):
        q = dict(p, wd=p["wd"] * 2.0 ** e)
        dq = api.sepconv_bwd(ctx, desc, g, x, y, lens, q, saved)[0]
        assert ctx.last_status() == 0
        assert torch.equal(dq.float() * 2.0 ** -e, dx.float()), e


@pytest.mark.parametrize("K,B,T", [(1, 3, 16), (3, 2, 1040), (7, 9, 528), (35, 4, 512), (87, 2, 4112), (95, 5, 304)])
def test_stride_two_depthwise(api, ctx, K, B, T):
    """The stride-2 depthwise kernels: both parities of the padding, one tap to the most they take, rows around their tiles."""
    L = si.LayerCfg(C_in=24, C_out=16, K=K, stride=2)
    d = si.draw(si.Workload("s2", "bf16", B, T, [L], 700 + K, len_lo=max(1, T // 5), len_hi=T, affine="random"))
    d.lengths[0], d.lengths[-1] = T, T // 5
    rep = U.run_block(ctx, api, L, "bf16", d.x, d.lengths, d.params[0], d.g)
    print(f"\nstride 2 K={K}: {rep}")
    rep.check()

"""sepconv_fwd_static -- the forward block call for callers that may not allocate device memory
(fixed-memory real-time pipelines, plugins under a framework that owns the device heap).  It must
give exactly what sepconv_fwd gives, call after call, although all calls share one built-in scratch
array that still holds the previous call's data."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from oracle import sepconv_oracle as O
from tests import parity_util as U

pytestmark = pytest.mark.gpu


def _run_pair(api, ctx, L, B, T, dtype, seed, first_call_on_device=False):
    w = si.Workload("static", dtype, B, T, [L], seed, len_lo=T // 3, len_hi=T, affine="random")
    d = si.draw(w)
    desc = api.block_desc(L, B, T, dtype)
    xd, pd = U.dev(d.x, dtype), U.params_dev(d.params[0], dtype)
    ld = torch.from_numpy(d.lengths).cuda()
    y_ref, len_ref, saved_ref = api.sepconv_fwd(ctx, desc, xd, ld, pd)
    # caller-owned outputs, allocated before the call under test
    y = torch.full_like(y_ref, float("nan"))
    out_len = torch.zeros_like(len_ref)
    saved = {k: torch.full_like(v, float("nan")) for k, v in saved_ref.items()}
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    free_before = torch.cuda.mem_get_info()[0]          # the driver's view: sees any allocation, not only torch's
    api.sepconv_fwd_static(ctx, desc, xd, ld, pd, y, out_len, saved)
    assert ctx.last_status() == 0
    assert torch.cuda.memory_allocated() == before
    if not first_call_on_device:                        # the first call loads the module that holds the array
        assert torch.cuda.mem_get_info()[0] == free_before
    rep = U.Report(dtype)
    rep.add("y", U.host(y), U.host(y_ref))
    # frames at and beyond a sample's output length are unspecified in the saved pointwise results
    valid = (torch.arange(y.shape[2], device="cuda")[None, None, :] < len_ref[:, None, None]).cpu().numpy()
    for k in saved_ref:
        if k in ("v", "vr"):
            rep.add(k, U.masked(saved[k], valid), U.masked(saved_ref[k], valid))
        else:
            rep.add(k, U.host(saved[k]), U.host(saved_ref[k]))
    rep.check()
    assert torch.equal(out_len, len_ref)
    assert torch.equal(y, y_ref)          # same kernels, same order: identical bits


def test_static_scratch_forward_matches_twice():
    import paper_1909_09577_b200 as api
    ctx = api.Context(0)
    try:
        # two calls in a row with different shapes and types: the second starts from the first one's leftovers
        _run_pair(api, ctx, si.LayerCfg(48, 64, K=33, residual="proj"), 4, 200, "bf16", seed=31, first_call_on_device=True)
        _run_pair(api, ctx, si.LayerCfg(32, 32, K=9, residual="identity"), 3, 120, "f32", seed=32)
        _run_pair(api, ctx, si.LayerCfg(48, 64, K=33, residual="proj"), 4, 200, "bf16", seed=33)
    finally:
        ctx.close()


def test_static_scratch_rejects_large_blocks():
    import paper_1909_09577_b200 as api
    ctx = api.Context(0)
    try:
        L = si.config(3).layers[0]                  # at B = 64 it needs more scratch than the built-in array holds
        desc = api.block_desc(L, 64, 400, "bf16")
        assert api.sepconv_workspace_bytes(desc)[0] > api.binding.STATIC_SCRATCH_BYTES
        x = torch.zeros((64, 256, 400), dtype=torch.bfloat16, device="cuda")
        y = torch.zeros((64, 512, 400), dtype=torch.bfloat16, device="cuda")
        lens = torch.full((64,), 400, dtype=torch.int32, device="cuda")
        with pytest.raises(api.SepconvError) as e:
            api.sepconv_fwd_static(ctx, desc, x, lens, {"wd": x, "wp": x, "gamma": x, "beta": x, "wr": x,
                                                        "gamma_r": x, "beta_r": x}, y, lens, {"u": x})
        assert e.value.code == -7
    finally:
        ctx.close()


DENSE = [
    # blocks whose operand copies exceed the built-in array while the scratch of the dense form does not
    (dict(C_in=256, C_out=256, K=33), 32, 397, "bf16"),
    (dict(C_in=512, C_out=512, K=33, dilation=2), 8, 400, "bf16"),
    (dict(C_in=256, C_out=256, K=11, has_dw=False, full_conv=True), 32, 800, "f16"),
    (dict(C_in=64, C_out=64, K=33), 32, 797, "f16"),
]


@pytest.mark.parametrize("case", range(len(DENSE)))
def test_static_scratch_without_room_for_copies(case):
    import paper_1909_09577_b200 as api
    kw, B, T, dtype = DENSE[case]
    L = si.LayerCfg(**kw)
    d = si.draw(si.Workload("static", dtype, B, T, [L], 40 + case, len_lo=T // 3, len_hi=T, affine="random"))
    desc = api.block_desc(L, B, T, dtype)
    assert api.sepconv_workspace_bytes(desc)[0] > api.binding.STATIC_SCRATCH_BYTES
    new = lambda shape, dt: torch.full(shape, float("nan"), dtype=dt, device="cuda")
    y, out_len = new((B, L.C_out, T), U.TD[dtype]), torch.zeros(B, dtype=torch.int32, device="cuda")
    saved = {"u": new((B, L.C_in, T), torch.float16), "v": new((B, L.C_out, T), torch.float16),
             "mean": new((L.C_out,), torch.float32), "invstd": new((L.C_out,), torch.float32)}
    ctx = api.Context(0)
    try:
        api.sepconv_fwd_static(ctx, desc, U.dev(d.x, dtype), torch.from_numpy(d.lengths).cuda(), U.params_dev(d.params[0], dtype),
                               y, out_len, saved)
        assert ctx.last_status() == 0
    finally:
        ctx.close()
    S = O.block_fwd(L, d.x, d.lengths, d.params[0])
    vm = S["valid"]
    rep = U.Report(dtype)
    if L.has_dw:
        rep.add("u", U.host(saved["u"]), S["u"], vm)
    rep.add("v", U.masked(saved["v"], vm), np.where(vm, S["v"], 0.0), vm)
    rep.add("mean", U.host(saved["mean"]), S["mean"])
    rep.add("invstd", U.host(saved["invstd"]), S["invstd"])
    rep.add("y", U.host(y), S["y"], vm, stored=True)
    rep.check()
    np.testing.assert_array_equal(out_len.cpu().numpy(), S["out_len"])

"""Calls repeated with the same arguments are replayed as CUDA graphs: the replays read the buffers anew, give the bits of
the direct calls, count their launches, and step aside when the caller is capturing."""
import pytest
import torch

import synth_inputs as si
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [128, 77])
def test_replays_equal_direct_calls(T):
    import paper_1909_09577_b200 as api
    L = si.LayerCfg(32, 48, K=9, residual="proj")
    ctx, ref = api.Context(0), api.Context(0)
    desc = api.block_desc(L, 17, T, "bf16")
    ws, wb = (torch.empty(n, dtype=torch.uint8, device="cuda") for n in api.sepconv_workspace_bytes(desc))
    x, dy = torch.empty((17, 32, T), dtype=torch.bfloat16, device="cuda"), torch.empty((17, 48, T), dtype=torch.bfloat16, device="cuda")
    lens = torch.empty(17, dtype=torch.int32, device="cuda")
    y, saved, params, counts = None, None, None, []
    for call in range(6):                  # the same buffers with new contents every time: two direct calls, then graphs
        d = si.draw(si.Workload("replay", "bf16", 17, T, [L], 70 + call, len_lo=T // 2, len_hi=T, affine="random"))
        x.copy_(U.dev(d.x, "bf16")), dy.copy_(U.dev(d.g, "bf16")), lens.copy_(torch.from_numpy(d.lengths))
        new = U.params_dev(d.params[0], "bf16")
        if params is None:
            params, grads = new, {"d" + n: torch.zeros_like(t, dtype=torch.float32) for n, t in new.items()}
        for n in params:
            params[n].copy_(new[n])
        n0 = ctx.launch_count()
        y, _, saved = api.sepconv_fwd(ctx, desc, x, lens, params, workspace=ws, y=y, saved=saved)
        dx, _, _ = api.sepconv_bwd(ctx, desc, dy, x, y, lens, params, saved, grads=grads, workspace=wb)
        counts.append(ctx.launch_count() - n0)
        ry, _, rs = api.sepconv_fwd(ref, desc, x, lens, params)
        rdx, _, rg = api.sepconv_bwd(ref, desc, dy, x, ry, lens, params, rs)
        assert torch.equal(y, ry) and torch.equal(dx, rdx) and all(torch.equal(grads[k], rg[k]) for k in rg)
    assert len(set(counts)) == 1 and ctx.last_status() == 0
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=s):
        api.sepconv_fwd(ctx, desc, x, lens, params, workspace=ws, y=y, saved=saved, stream=s)
    y.zero_()
    g.replay()
    assert torch.equal(y, ry)
    ctx.close(), ref.close()

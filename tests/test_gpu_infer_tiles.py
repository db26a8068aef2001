"""Evaluation-mode blocks through each tile shape of the contraction that ends with batch norm, residual and ReLU: few units
(128 x 64), many with up to 128 or with more output channels, more samples than the small and the wide tile's tables hold, and
the forms of the layer's tail."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from oracle import sepconv_oracle as O
from tests import parity_util as U

pytestmark = pytest.mark.gpu

CASES = [
    (dict(C_in=64, C_out=136, K=11, residual="proj"), 1, 72),
    (dict(C_in=40, C_out=128, K=5, residual="proj"), 20, 1040),                                  # 340 units, one row tile
    (dict(C_in=264, C_out=264, K=9, residual="identity"), 9, 776),                               # 351 units, three row tiles
    (dict(C_in=16, C_out=24, K=5), 260, 72),
    (dict(C_in=24, C_out=264, K=5, residual="proj"), 260, 40),
    (dict(C_in=32, C_out=32, K=7, residual="identity", res_before_relu=False), 3, 200),
    (dict(C_in=32, C_out=48, K=7, has_relu=False), 3, 200),
]


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_infer_tiles(dtype, case):
    import paper_1909_09577_b200 as api
    kw, B, T = CASES[case]
    L = si.LayerCfg(**kw)
    d = si.draw(si.Workload("infer", dtype, B, T, [L], 980 + case, len_lo=max(1, T // 4), len_hi=T, affine="random"))
    d.lengths[0] = T
    rng = np.random.default_rng(70 + case)
    run = {"mean": 0.3 * rng.standard_normal(L.C_out), "var": rng.uniform(0.5, 2.0, L.C_out)}
    if L.residual == "proj":
        run.update(mean_r=0.3 * rng.standard_normal(L.C_out), var_r=rng.uniform(0.5, 2.0, L.C_out))
    run = {k: v.astype(np.float32) for k, v in run.items()}
    ctx = api.Context(0)
    y, out_len = api.sepconv_infer(ctx, api.block_desc(L, B, T, dtype), U.dev(d.x, dtype), torch.from_numpy(d.lengths).cuda(),
                                   U.params_dev(d.params[0], dtype), {k: torch.from_numpy(v).cuda() for k, v in run.items()},
                                   x_res=U.dev(d.x, dtype) if L.residual != "none" else None)
    assert ctx.last_status() == 0
    ctx.close()
    S = O.block_infer(L, d.x, d.lengths, d.params[0], run)
    np.testing.assert_array_equal(out_len.cpu().numpy(), S["out_len"])
    rep = U.Report(dtype)
    rep.add("y", U.host(y), S["y"], S["valid"], stored=True)
    print(f"\ninfer tiles {case} {dtype}: {rep}")
    rep.check()
    assert np.all(U.host(y)[~np.broadcast_to(S["valid"], y.shape)] == 0)

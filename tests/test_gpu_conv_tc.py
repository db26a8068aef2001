"""The non-separable convolution on the tensor cores: channel tails below and above a tile, frame counts around a 64-frame
block, taps that reach past both ends of the rows, one tap, dilation, both tile heights, rows of any length."""
import pytest

import synth_inputs as si
from tests import parity_util as U

pytestmark = pytest.mark.gpu

CASES = [
    # (layer kwargs, B, T, shortest length)
    (dict(C_in=8, C_out=8, K=1), 2, 64, 20),
    (dict(C_in=24, C_out=40, K=5, residual="proj"), 3, 72, 1),
    (dict(C_in=136, C_out=72, K=11), 5, 128, 40),
    (dict(C_in=64, C_out=320, K=3, residual="proj"), 20, 520, 100),          # 256-row tiles
    (dict(C_in=256, C_out=256, K=4), 9, 200, 50),                            # even K
    (dict(C_in=32, C_out=32, K=29, residual="identity"), 4, 56, 9),          # taps wider than some samples
    (dict(C_in=48, C_out=64, K=7, dilation=3), 6, 136, 33),
    (dict(C_in=72, C_out=136, K=35, residual="proj"), 2, 301, 70),           # odd rows; more taps than one reduction chunk
]


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_conv_on_tensor_cores(dtype, case):
    import paper_1909_09577_b200 as api
    kw, B, T, lo = CASES[case]
    L = si.LayerCfg(has_dw=False, full_conv=True, **kw)
    d = si.draw(si.Workload("conv", dtype, B, T, [L], 600 + case, len_lo=lo, len_hi=T, affine="random"))
    d.lengths[0], d.lengths[-1] = T, lo
    ctx = api.Context(0)
    rep = U.run_block(ctx, api, L, dtype, d.x, d.lengths, d.params[0], d.g)
    ctx.close()
    print(f"\nconv case {case} {dtype}: {rep}")
    rep.check()

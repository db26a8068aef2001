"""Small float32 blocks, whose batch norm is one kernel per direction with a CTA per channel: channels of one frame, of as
many eight-frame chunks as the kernel takes and of one more, rows that are no whole number of chunks, and each form of the
layer's tail."""
import pytest

import synth_inputs as si
from tests import parity_util as U

pytestmark = pytest.mark.gpu

CASES = [
    # (layer kwargs, B, T, shortest length)
    (dict(C_in=20, C_out=12, K=3), 2, 1, 1),
    (dict(C_in=16, C_out=16, K=5, residual="identity"), 8, 1024, 300),                   # 1024 chunks
    (dict(C_in=16, C_out=24, K=5), 5, 1633, 700),                                        # 1025
    (dict(C_in=8, C_out=40, K=9, residual="proj"), 7, 61, 5),
    (dict(C_in=24, C_out=24, K=7, residual="identity", res_before_relu=False), 3, 130, 64),
    (dict(C_in=16, C_out=8, K=1, has_dw=False, has_bn=False, has_bias=True, has_relu=False), 4, 50, 9),
    (dict(C_in=16, C_out=12, K=5, has_dw=False, full_conv=True), 3, 77, 20),
    # rows that are no whole number of chunks: at the limit for eight samples, at that for more and past it
    (dict(C_in=24, C_out=24, K=5, residual="identity"), 8, 1021, 300),
    (dict(C_in=16, C_out=24, K=5), 9, 221, 90),
    (dict(C_in=16, C_out=24, K=5, residual="proj"), 9, 253, 90),
    (dict(C_in=8, C_out=264, K=3), 16, 125, 60),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_small_channels(case):
    import paper_1909_09577_b200 as api
    kw, B, T, lo = CASES[case]
    L = si.LayerCfg(**kw)
    d = si.draw(si.Workload("bn_small", "f32", B, T, [L], 900 + case, len_lo=lo, len_hi=T, affine="random"))
    d.lengths[0] = T
    ctx = api.Context(0)
    rep = U.run_block(ctx, api, L, "f32", d.x, d.lengths, d.params[0], d.g)
    ctx.close()
    print(f"\nsmall case {case}: {rep}")
    rep.check()

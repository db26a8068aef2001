"""16-bit blocks whose statistics merge and apply step are one kernel with a CTA per channel, and whose backward reduction has a
CTA per channel too: one vector per channel, the most vectors and channels the kernel takes and one more of each, samples that
leave most CTAs of the contraction without a unit, and each residual form."""
import pytest

import synth_inputs as si
from tests import parity_util as U

pytestmark = pytest.mark.gpu

CASES = [
    # (layer kwargs, B, T, shortest length)
    (dict(C_in=24, C_out=40, K=5, residual="proj"), 1, 8, 8),
    (dict(C_in=296, C_out=296, K=9, residual="identity"), 16, 512, 130),          # 1024 vectors, 296 channels
    (dict(C_in=16, C_out=304, K=9, residual="proj"), 4, 264, 1),                  # too many channels
    (dict(C_in=16, C_out=24, K=11), 5, 1640, 300),                                # 1025 vectors
    (dict(C_in=64, C_out=136, K=5, has_dw=False, full_conv=True), 3, 264, 20),
    # the row-mapped reduction: few channels with more than 4096 vectors, in its shortest rows and in rows that end inside a warp
    (dict(C_in=8, C_out=16, K=5), 17, 2048, 100),
    (dict(C_in=16, C_out=63, K=5, residual="proj"), 16, 2056, 900),
    (dict(C_in=24, C_out=24, K=5, residual="identity"), 9, 3648, 1200),
    (dict(C_in=8, C_out=8, K=3), 16, 2048, 700),                                  # 4096 vectors: not yet
    (dict(C_in=8, C_out=8, K=3), 17, 2040, 100),                                  # rows too short for it
]


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_apply_per_channel(dtype, case):
    import paper_1909_09577_b200 as api
    kw, B, T, lo = CASES[case]
    L = si.LayerCfg(**kw)
    d = si.draw(si.Workload("apply_ch", dtype, B, T, [L], 960 + case, len_lo=lo, len_hi=T, affine="random"))
    d.lengths[0] = T
    ctx = api.Context(0)
    rep = U.run_block(ctx, api, L, dtype, d.x, d.lengths, d.params[0], d.g)
    ctx.close()
    print(f"\napply case {case} {dtype}: {rep}")
    rep.check()

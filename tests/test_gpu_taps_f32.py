"""Float32 tap gradients of rows that are no multiple of 8 frames (their last chunk is filled up with zeros in shared memory):
one frame past a chunk and one short of it, rows shorter than the taps, the fewest and the most taps the kernel takes."""
import pytest

import synth_inputs as si
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,B,T,lo", [(3, 4, 50, 7), (7, 6, 195, 90), (9, 3, 7, 2), (15, 2, 129, 60), (33, 7, 228, 150), (87, 5, 71, 30), (95, 9, 303, 64)])
def test_tap_gradients(K, B, T, lo):
    import paper_1909_09577_b200 as api
    L = si.LayerCfg(C_in=24, C_out=16, K=K)
    d = si.draw(si.Workload("taps", "f32", B, T, [L], 940 + K, len_lo=lo, len_hi=T, affine="random"))
    d.lengths[0] = T
    ctx = api.Context(0)
    rep = U.run_block(ctx, api, L, "f32", d.x, d.lengths, d.params[0], d.g)
    ctx.close()
    print(f"\ntaps {K} T={T}: {rep}")
    rep.check()

"""GPU parity of the pooling kernels: every number of taps, units of one to sixteen partial rows, segments that end
off a multiple of four and start off a 16-byte boundary, segments shorter than the halo and longer than a warp's
120 tokens."""
import pytest
import torch

from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import assert_scores_close, make_path, oracle_layer, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,S,Hq,Hk,w", [
    (I.POOL_AVG, 1, 2, 2, 32), (I.POOL_AVG, 3, 4, 1, 32), (I.POOL_AVG, 5, 16, 2, 64), (I.POOL_AVG, 7, 32, 2, 64),
    (I.POOL_AVG, 9, 32, 1, 128), (I.POOL_AVG, 11, 4, 2, 32), (I.POOL_AVG, 33, 4, 2, 32), (I.POOL_AVG, 7, 14, 2, 64),
    (I.POOL_MAX, 1, 2, 2, 32), (I.POOL_MAX, 5, 6, 2, 64), (I.POOL_MAX, 7, 4, 1, 256), (I.POOL_MAX, 9, 8, 1, 128),
    (I.POOL_MAX, 15, 4, 2, 32),
    # rows that are no multiple of those in flight: 3 kv heads of 8 and of 16, heads of 2, 4, 8 and 16
    (I.POOL_AVG, 7, 24, 3, 128), (I.POOL_AVG, 5, 48, 3, 128), (I.POOL_AVG, 9, 8, 1, 128), (I.POOL_MAX, 5, 3, 3, 200),
    (I.POOL_MAX, 7, 3, 1, 512), (I.POOL_MAX, 9, 3, 3, 1024), (I.POOL_MAX, 3, 3, 1, 2048),
])
def test_pooling_of_ragged_segments(mode, S, Hq, Hk, w):
    seqlens = tuple(w + t for t in (1, 3, 121, 120, 479, 962))
    wl = I.workload("C3", n_q_heads=Hq, n_kv_heads=Hk, window=w, pool_kernel=S, pool_mode=mode, seqlens=seqlens,
                    budgets=tuple(w for _ in seqlens), layers=1, l_min=1, l_obs=2, distractors=0)
    x = I.layer_inputs(wl, 0, seed=S)
    path = make_path(wl)
    B.asl_score_layer(path.ctx, to_dev(x["q_obs"]), to_dev(x["k"]), path.scores_kv, path.scores_agg, path.workspace, path.ws_bytes)
    torch.cuda.synchronize()
    P_ref, agg_ref = oracle_layer(wl, x)
    assert_scores_close(path.scores_kv.cpu().numpy(), P_ref, "scores_kv")
    assert_scores_close(path.scores_agg.cpu().numpy(), agg_ref, "scores_agg")
    path.close()

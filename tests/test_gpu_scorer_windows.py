"""GPU parity of the scorer where its chunks of query rows are not whole: windows off a multiple of 32, halves that
are not full, heads padded under max pooling, windows cut into pieces, single-tile and single-key segments, and a
batch whose segments fall into several groups."""
import numpy as np
import pytest
import torch

from oracle import asl_oracle as O
from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import assert_scores_close, make_path, oracle_layer, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [I.POOL_AVG, I.POOL_MAX])
@pytest.mark.parametrize("Hq,Hk,w,seqlens", [
    (4, 1, 1, (2, 130)),             # one row per head; one past token, one key past a tile
    (6, 2, 33, (34, 161 + 33)),      # padded heads under max pooling
    (8, 1, 20, (500,)),              # 160 rows: two halves of 96
    (14, 2, 24, (385, 128 + 24)),    # seven heads per kv head
    (8, 2, 100, (700,)),             # two heads per chunk
    (4, 2, 130, (300,)),             # a head over both halves
    (2, 1, 256, (600,)),
    (2, 1, 300, (900, 301)),         # a head in two pieces
])
def test_windows_of_any_length(mode, Hq, Hk, w, seqlens):
    wl = I.workload("C3", n_q_heads=Hq, n_kv_heads=Hk, window=w, pool_mode=mode, seqlens=seqlens,
                    budgets=tuple(w for _ in seqlens), layers=1, l_min=1, l_obs=2, distractors=0)
    x = I.layer_inputs(wl, 0, seed=17)
    path = make_path(wl)
    q, k = to_dev(x["q_obs"]), to_dev(x["k"])
    P_ref, agg_ref = oracle_layer(wl, x)
    B.asl_score_layer(path.ctx, q, k, path.scores_kv, path.scores_agg, path.workspace, path.ws_bytes)
    lse = torch.empty((wl.batch, Hq, w), dtype=torch.float32, device="cuda")
    B.asl_window_lse(path.ctx, path.workspace, path.ws_bytes, lse)
    torch.cuda.synchronize()
    assert_scores_close(path.scores_kv.cpu().numpy(), P_ref, "scores_kv")
    assert_scores_close(path.scores_agg.cpu().numpy(), agg_ref, "scores_agg")
    cu = wl.cu_seqlens()
    for b in range(wl.batch):
        ref = O.window_lse(O.widen_bf16(x["q_obs"][b]), O.widen_bf16(x["k"][cu[b]:cu[b + 1]]), wl.group)
        assert np.abs(lse[b].cpu().numpy().astype(np.float64) - ref).max() <= 2e-4
    B.asl_score_layer_lse(path.ctx, q, k, lse, path.scores_kv, path.scores_agg, path.workspace, path.ws_bytes)
    torch.cuda.synchronize()
    assert_scores_close(path.scores_kv.cpu().numpy(), P_ref, "one-pass scores_kv")
    assert B.asl_device_status(path.ctx) == (B.ASL_OK, 0)
    path.close()


@pytest.mark.parametrize("ctas", [0, 5])
def test_many_requests_in_several_groups(ctas):
    """Forty requests of one to three tiles: more segments than CTAs, runs that end inside segments."""
    seqlens = tuple(33 + 37 * i % 350 for i in range(40))
    wl = I.workload("C1", seqlens=seqlens, budgets=tuple(32 for _ in seqlens), layers=1, l_min=1, l_obs=2)
    x = I.layer_inputs(wl, 0, seed=18)
    path = make_path(wl, score_ctas=ctas)
    for _ in range(2):
        B.asl_score_layer(path.ctx, to_dev(x["q_obs"]), to_dev(x["k"]), path.scores_kv, path.scores_agg, path.workspace, path.ws_bytes)
    torch.cuda.synchronize()
    P_ref, _ = oracle_layer(wl, x)
    assert_scores_close(path.scores_kv.cpu().numpy(), P_ref, "scores_kv")
    assert B.asl_device_status(path.ctx) == (B.ASL_OK, 0)
    path.close()


@pytest.mark.parametrize("ctas,n", [(8, 512), (8, 513), (0, 7424), (0, 7425), (0, 33)])
def test_one_group_of_segments_where_a_cta_has_one_tile(ctas, n):
    """The last length with a single group and the first with two (two kv heads: 8 tiles for 8 CTAs, 116 for the smallest
    grid of a B200).  Other inputs in every call: an offset of the call before last, in whose set a call counts, shows."""
    wl = I.workload("C1", seqlens=(n,), budgets=(32,), layers=1, l_min=1, l_obs=2)
    path = make_path(wl, score_ctas=ctas)
    for seed in range(5):
        x = I.layer_inputs(wl, 0, seed=seed)
        q, k = to_dev(x["q_obs"]), to_dev(x["k"])
        if seed & 1:
            B.asl_score_columns(path.ctx, q, k, None, path.workspace, path.ws_bytes, 0)
            B.asl_pool_scores(path.ctx, path.workspace, path.ws_bytes, 0, path.scores_kv, path.scores_agg)
        else:
            B.asl_score_layer(path.ctx, q, k, path.scores_kv, path.scores_agg, path.workspace, path.ws_bytes)
        torch.cuda.synchronize()
        P_ref, _ = oracle_layer(wl, x)
        assert_scores_close(path.scores_kv.cpu().numpy(), P_ref, f"scores_kv, inputs {seed}")
    assert B.asl_device_status(path.ctx) == (B.ASL_OK, 0)
    path.close()

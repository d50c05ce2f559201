"""GPU parity of the two-pass scorer where one key's logit lies above the fp32 range of its row's reference (the first
logit that a CTA meets of the row): every column of a tile's accumulator, whichever unit takes its exponential."""
import numpy as np
import pytest
import torch

from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import assert_scores_close, make_path, oracle_layer, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("ctas", [0, 3])                  # 3: runs of several tiles, the sums of earlier ones are kept
@pytest.mark.parametrize("powers", [120.0, 300.0])        # of two, for the smallest row; the largest has half as many again
@pytest.mark.parametrize("block", [32, 96])               # amid a tile; its last 32 keys (the last 16 are redone from registers)
def test_one_key_far_above_the_first_of_its_row(block, powers, ctas, fp8):
    """4 requests x 8 kv heads, in each one heavy key and no other: its column is the block's first plus 0 .. 31.  The rows
    of a head have different lengths, so that their logits cover [powers, 1.5 powers] in steps of about one."""
    Hq, Hk, w, n, d = 32, 8, 64, 700, 128
    wl = I.workload("C3", n_q_heads=Hq, n_kv_heads=Hk, window=w, seqlens=(n,) * 4, budgets=(w + 100,) * 4, layers=1,
                    l_min=1, l_obs=2)
    g = np.random.default_rng(12)
    q = np.ones((4, Hq, w, d), np.float32) * (1.0 + np.arange(w, dtype=np.float32) / 128)[None, None, :, None]
    k = g.normal(0.0, 0.25, size=(4, n, Hk, d)).astype(np.float32)
    a = powers * np.log(2.0) / np.sqrt(d)                 # logit a * sqrt(d) nats
    heavy = np.array([[128 * 2 + block + 8 * b + h for h in range(Hk)] for b in range(4)])
    for b in range(4):
        for h in range(Hk):
            k[b, heavy[b, h], h] = a
    x = {"q_obs": I.f32_to_bf16_bits(q), "k": I.f32_to_bf16_bits(k.reshape(4 * n, Hk, d))}
    launch = {"score_ctas": ctas}
    if fp8:
        x["k"], x["k_scale"] = I.keys_to_fp8(x["k"])
        launch.update(k_dtype=B.ASL_K_FP8_E4M3, k_scale=[float(s) for s in x["k_scale"]])
    path = make_path(wl, **launch)
    B.asl_score_layer(path.ctx, to_dev(x["q_obs"]), to_dev(x["k"]), path.scores_kv, path.scores_agg, path.workspace,
                      path.ws_bytes)
    torch.cuda.synchronize()
    assert B.asl_device_status(path.ctx)[0] == B.ASL_OK
    P_ref, agg_ref = oracle_layer(wl, x)
    kv = path.scores_kv.cpu().numpy()
    for b in range(4):                                    # the heavy key has all of the rows' mass: G * W, pooled over 7
        for h in range(Hk):
            assert P_ref[h, b * (n - w) + heavy[b, h]] == pytest.approx(wl.group * w / 7, rel=1e-6)
    assert np.isfinite(kv).all()
    assert_scores_close(kv, P_ref, "scores_kv")
    assert_scores_close(path.scores_agg.cpu().numpy(), agg_ref, "scores_agg")
    path.close()

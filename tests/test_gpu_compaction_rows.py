"""GPU parity of K/V compaction at row counts around a block's 64, bf16 and FP8 keys, and of the row gather."""
import numpy as np
import pytest
import torch

from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import bits_of, make_path, to_dev, with_fp8_keys

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp8", [False, True])
def test_compaction_of_any_number_of_rows(fp8):
    w = 64
    seqlens, kept = (65, 80, 200, 200, 200, 300, 500), (64, 65, 127, 128, 129, 193, 500)
    wl = I.workload("C3", n_q_heads=32, n_kv_heads=8, window=w, seqlens=seqlens, budgets=kept, layers=1, l_min=1, l_obs=2)
    x = I.layer_inputs(wl, 0, seed=3)
    launch = {}
    if fp8:
        x = with_fp8_keys(x)
        launch = dict(k_dtype=B.ASL_K_FP8_E4M3, k_scale=[float(s) for s in x["k_scale"]])
    path = make_path(wl, **launch)
    rng, cu = np.random.default_rng(4), wl.cu_seqlens()
    idx = np.stack([np.concatenate([np.sort(rng.choice(n, m, replace=False)) for n, m in zip(seqlens, kept)]) for _ in range(wl.n_kv_heads)])
    idx_dev = torch.from_numpy(idx.astype(np.int32)).cuda()
    path.k_out.zero_(), path.v_out.zero_()
    B.asl_compact_kv(path.ctx, to_dev(x["k"]), to_dev(x["v"]), idx_dev, path.k_out, path.v_out)
    torch.cuda.synchronize()
    k_out, v_out, at = bits_of(path.k_out), bits_of(path.v_out), 0
    for b, m in enumerate(kept):
        for h in range(wl.n_kv_heads):
            rows = cu[b] + idx[h, at:at + m]
            assert (k_out[h, at:at + m] == x["k"][rows, h]).all() and (v_out[h, at:at + m] == x["v"][rows, h]).all(), (b, h)
        at += m
    path.close()


@pytest.mark.parametrize("row_bytes", [16, 400, 496, 512, 528, 1008, 1024, 1040, 2032, 2048, 2064, 4080, 4096, 4112, 4608, 7168, 8192])
def test_row_gather_of_rows_around_a_warps_loads(row_bytes):
    """A warp has one, two, four or eight loads of 512 bytes in flight: rows below, at and above each of them."""
    w, seqlens, kept = 32, (40, 700, 90), (33, 321, 90)
    wl = I.workload("C1", window=w, seqlens=seqlens, budgets=kept, layers=1, l_min=1, l_obs=2)
    path = make_path(wl)
    rng, cu = np.random.default_rng(row_bytes), wl.cu_seqlens()
    x = rng.integers(-2**31, 2**31, (wl.total_tokens, row_bytes // 4), dtype=np.int64).astype(np.int32)
    ids = [np.sort(rng.permutation(n)[:wl.kept(b)]) for b, n in enumerate(seqlens)]
    out = torch.full((path.sum_kept + 1, row_bytes // 4), 7, dtype=torch.int32, device="cuda")
    B.asl_compact_rows(path.ctx, torch.from_numpy(x).cuda(), torch.from_numpy(np.concatenate(ids).astype(np.int32)).cuda(), out, row_bytes)
    got = out.cpu().numpy()
    assert (got[:-1] == np.concatenate([x[int(cu[b]) + i] for b, i in enumerate(ids)])).all()
    assert (got[-1] == 7).all()
    path.close()

"""GPU parity of rank rows and their statistic where tiles of 1024, 2048 and 4096 scores begin and end, one per segment
or several, up to the line where the radix passes take over: ties within and across tiles, both signs, equal scores
only, and tiles whose scores do not overlap."""
import numpy as np
import pytest
import torch

from oracle import asl_oracle as O
from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import make_path

pytestmark = pytest.mark.gpu


def _scores(T, kind, rng):
    if kind == 0:
        return rng.standard_normal(T).astype(np.float32)
    if kind == 1:                                       # ties everywhere, both zeros, both signs
        return (np.round(rng.standard_normal(T) * 2) / 2 * np.where(rng.random(T) < 0.5, -1.0, 1.0)).astype(np.float32)
    if kind == 2:
        return np.full(T, 0.25, np.float32)
    return (np.exp(rng.normal(-9, 1.5, T)) * 10.0 ** (np.arange(T) // 2048)).astype(np.float32)


@pytest.mark.parametrize("lengths", [
    (1, 1023, 1024), (1025, 2047, 2048), (2049, 5, 4096), (4097, 2050, 1), (8191, 8193, 3), (16384, 4095), (16385, 4097, 12289),
    (65536,), (65535, 8193), (65537,),
])
def test_rank_rows_and_statistic(lengths):
    w = 32
    wl = I.workload("C1", seqlens=tuple(T + w for T in lengths), budgets=tuple(w + (T + 9) // 10 for T in lengths), l_min=1, l_obs=3)
    path = make_path(wl)
    rng = np.random.default_rng(sum(lengths))
    rows = []
    for layer in range(4):
        s = np.concatenate([_scores(T, layer % 4 if layer else 3, rng) for T in lengths])
        path.scores_agg.copy_(torch.from_numpy(s))
        n_rows = min(layer + 1, 3)
        B.asl_rank_stat(path.ctx, path.scores_agg, layer, n_rows, path.rank_ring, path.stat, path.workspace, path.ws_bytes)
        torch.cuda.synchronize()
        stat, got, at, ranks = path.read_stat(), path.rank_ring[layer % 3].cpu().numpy(), 0, []
        for b, T in enumerate(lengths):
            ranks.append(O.rank_desc(s[at:at + T].astype(np.float64)))
            assert (got[at:at + T] == ranks[b]).all(), (layer, b)
            at += T
        rows.append(ranks)
        for b in range(len(lengths)):
            assert stat[b]["evaluated"] == (1 if layer >= 1 else 0)
            if layer >= 1:
                num, m, var = O.rank_statistic(np.stack([r[b] for r in rows[-n_rows:]]), int((lengths[b] + 9) // 10))
                assert (stat[b]["num"], stat[b]["m"]) == (num, m) and stat[b]["var_top"] == pytest.approx(var, rel=1e-14)
    path.close()
    for T in lengths:                                    # the same kernels without a plan
        for kind in range(4):
            s = _scores(T, kind, rng)
            out = torch.full((T,), -1, dtype=torch.int32, device="cuda")
            B.asl_rank_desc_static(torch.from_numpy(s).cuda(), T, out)
            assert (out.cpu().numpy() == O.rank_desc(s.astype(np.float64))).all(), (T, kind)

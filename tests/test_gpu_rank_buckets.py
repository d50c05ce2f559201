"""GPU parity of rank rows where their kernels begin and end: the counted segments' last length and the first split one,
every change of the sample's size, the last split length and the first of the radix passes.  Scores: smooth, heavy tailed,
ties in runs, equal only, and a row that puts all but the sampled tokens into one bucket, too large for a block."""
import numpy as np
import pytest
import torch

from oracle import asl_oracle as O
from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import make_path

pytestmark = pytest.mark.gpu


def _sampled(T):
    """The tokens at which the split samples a segment of T tokens."""
    S = 256 if T <= 32768 else 512 if T <= 131072 else 1024
    s = np.arange(S, dtype=np.int64)
    lo, hi = s * T // S, (s + 1) * T // S
    return np.minimum(T - 1, lo + ((s * 2654435761) % 2**32 >> 8) % np.maximum(1, hi - lo))


def _scores(T, kind, rng):
    if kind == "normal":
        return rng.standard_normal(T).astype(np.float32)
    if kind == "tail":
        return np.exp(rng.normal(-9, 4, T)).astype(np.float32)
    if kind == "ties":
        return np.repeat(np.round(rng.standard_normal(T // 7 + 1) * 2) / 2, 7)[:T].astype(np.float32)
    if kind == "equal":
        return np.full(T, 0.25, np.float32)
    s = rng.random(T) if kind == "one bucket" else np.full(T, 0.5)      # "one bucket, equal"
    s[_sampled(T)] = 2.0 + rng.random(_sampled(T).size)
    return s.astype(np.float32)


KINDS = ("normal", "tail", "ties", "equal", "one bucket", "one bucket, equal")


@pytest.mark.parametrize("T", [1, 31, 33, 127, 129, 4095, 4096, 4097, 5119, 32768, 32769, 131072, 131073, 262144])
def test_rank_row_at_the_edges_of_its_kernels(T):
    rng = np.random.default_rng(T)
    for kind in KINDS:
        s = _scores(T, kind, rng)
        out = torch.full((T,), -1, dtype=torch.int32, device="cuda")
        B.asl_rank_desc_static(torch.from_numpy(s).cuda(), T, out)
        assert (out.cpu().numpy() == O.rank_desc(s.astype(np.float64))).all(), kind


@pytest.mark.parametrize("lengths", [(33,), (4096,), (4097,), (70001, 40000, 3), (131073, 200), (262144,), (262145, 5000)])
def test_row_and_statistic_of_a_plan(lengths):
    w, rows, ranks = 32, 4, []
    wl = I.workload("C1", seqlens=tuple(T + w for T in lengths), budgets=tuple(w + T // 9 for T in lengths), l_min=1, l_obs=rows)
    path = make_path(wl)
    rng = np.random.default_rng(sum(lengths))
    for layer in range(rows + 1):
        per = [_scores(T, KINDS[layer % 6], rng) for T in lengths]
        path.scores_agg.copy_(torch.from_numpy(np.concatenate(per)))
        B.asl_rank_stat(path.ctx, path.scores_agg, layer, min(layer + 1, rows), path.rank_ring, path.stat, path.workspace, path.ws_bytes)
        ranks.append([O.rank_desc(s.astype(np.float64)) for s in per])
        got, at, stat = path.rank_ring[layer % rows].cpu().numpy(), 0, path.read_stat()
        for b, T in enumerate(lengths):
            assert (got[at:at + T] == ranks[-1][b]).all(), (layer, b)
            at += T
            assert stat[b]["evaluated"] == (layer >= 1) and stat[b]["layer_idx"] == layer
            if layer >= 1:
                num, m, _ = O.rank_statistic(np.stack([r[b] for r in ranks[-min(layer + 1, rows):]]), T // 9)
                assert (stat[b]["num"], stat[b]["m"]) == (num, m)
    path.close()


@pytest.mark.parametrize("kind", ["one bucket", "one bucket, equal", "across zero"])
def test_blocks_whose_pairs_crowd_into_one_bin(kind):
    """Requests whose tokens, but for the 512 sampled ones, fall into one bucket: around the most pairs that a bin compares
    with one another (512), the pairs of a step of the passes that sort longer ones (2048) and those that a block holds (4096)."""
    lengths = (960, 1023, 1024, 1025, 1087, 2495, 2496, 2559, 2560, 2561, 4544, 4607, 4608, 4609, 4700, 40000)
    w, S, rng = 32, 512, np.random.default_rng(5)
    wl = I.workload("C1", seqlens=tuple(T + w for T in lengths), budgets=tuple(w + T // 9 for T in lengths), l_min=1, l_obs=2)
    path = make_path(wl)
    scores = []
    for T in lengths:
        i = np.arange(S, dtype=np.int64)
        lo, hi = i * T // S, (i + 1) * T // S
        at = np.minimum(T - 1, lo + ((i * 2654435761) % 2**32 >> 8) % np.maximum(1, hi - lo))
        s = {"one bucket": rng.random(T), "one bucket, equal": np.full(T, 0.5), "across zero": 1e-30 * rng.standard_normal(T)}[kind]
        s[at] = np.where(rng.random(S) < 0.5, 2.0, -2.0 if kind == "across zero" else 2.0) * (1 + rng.random(S))
        scores.append(s.astype(np.float32))
    path.scores_agg.copy_(torch.from_numpy(np.concatenate(scores)))
    for layer in range(2):
        B.asl_rank_stat(path.ctx, path.scores_agg, layer, layer + 1, path.rank_ring, path.stat, path.workspace, path.ws_bytes)
    got, at, stat = path.rank_ring.cpu().numpy(), 0, path.read_stat()
    for b, T in enumerate(lengths):
        row = O.rank_desc(scores[b].astype(np.float64))
        assert (got[:, at:at + T] == row).all(), b
        num, m, _ = O.rank_statistic(np.stack([row, row]), T // 9)
        assert (stat[b]["num"], stat[b]["m"]) == (num, m)
        at += T
    path.close()


@pytest.mark.parametrize("T", [5119, 32768, 131072, 262144])
def test_time_of_a_row_in_one_bucket_grows_with_its_length(T):
    """At most 300 us and 30 ns a token, two to three times what one block's passes take (9 to 13 ns a token); comparing a
    bucket's pairs with one another took 0.9 ms at 5000 tokens of one value and 1.6 s at 131072, 5.6 ms of random ones."""
    rng = np.random.default_rng(T)
    for kind in ("one bucket", "one bucket, equal"):
        s, out = torch.from_numpy(_scores(T, kind, rng)).cuda(), torch.empty(T, dtype=torch.int32, device="cuda")
        B.asl_rank_desc_static(s, T, out)
        begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        begin.record()
        B.asl_rank_desc_static(s, T, out)
        end.record()
        torch.cuda.synchronize()
        assert begin.elapsed_time(end) < 0.3 + 30e-6 * T, kind


@pytest.mark.parametrize("lengths,launches", [
    ((1, 33), 1), ((500, 97) * 4, 1), ((129, 1, 128, 127, 900), 1), ((1023, 1024), 1), ((32,) * 300, 1), ((1100, 1024), 3),
    ((1025,) * 63, 1), ((2048, 2047) * 30, 3), ((2048, 2047) * 33, 1), ((4096, 2049) * 48, 3), ((4096, 4095) * 48, 1)])
def test_short_requests_of_a_batch(lengths, launches):
    """Up to 1024 tokens, and for many requests up to 4096, a block sorts a request and takes its statistic: one launch; three
    for the split row.  Infinities and zeros of both signs; a request whose selection is final keeps its rank row and record."""
    w, rows, n = 32, 3, len(lengths)
    wl = I.workload("C1", seqlens=tuple(T + w for T in lengths), budgets=tuple(w + T // 9 for T in lengths), l_min=1, l_obs=rows)
    path = make_path(wl)
    path.set_controller(B.ASL_CONTROLLER_LATCH)
    rng, ranks = np.random.default_rng(sum(lengths)), []
    selected_word = B.STAT_DTYPE.fields["selected"][1] // 4
    for layer in range(rows + 1):
        per = [_scores(T, KINDS[layer % 4], rng) for T in lengths]
        for s in per[:2]:
            s[::5], s[1::7], s[2::9], s[3::9] = np.inf, -np.inf, 0.0, -0.0
        path.scores_agg.copy_(torch.from_numpy(np.concatenate(per)))
        if layer == rows:
            path.stat.view(torch.int32)[n - 1, selected_word] = 1
        before, ring, count = path.read_stat().copy(), path.rank_ring[layer % rows].cpu().numpy(), B.asl_launch_count(path.ctx)
        B.asl_rank_stat(path.ctx, path.scores_agg, layer, min(layer + 1, rows), path.rank_ring, path.stat, path.workspace, path.ws_bytes)
        assert B.asl_launch_count(path.ctx) - count == launches
        ranks.append([O.rank_desc(s.astype(np.float64)) for s in per])
        got, at, stat = path.rank_ring[layer % rows].cpu().numpy(), 0, path.read_stat()
        for b, T in enumerate(lengths):
            here = slice(at, at + T)
            at += T
            if before[b]["selected"]:
                ranks[-1][b] = ring[here]
                assert (got[here] == ring[here]).all() and stat[b].tobytes() == before[b].tobytes()
                continue
            assert (got[here] == ranks[-1][b]).all(), (layer, b)
            if layer >= 1:
                num, m, _ = O.rank_statistic(np.stack([r[b] for r in ranks[-min(layer + 1, rows):]]), T // 9)
                assert (stat[b]["num"], stat[b]["m"], stat[b]["layer_idx"]) == (num, m, layer)
    path.close()

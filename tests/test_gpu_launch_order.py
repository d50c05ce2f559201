"""Calls issued back to back, each on the results of the one before it, while inputs are overwritten in between: kernels
that become resident before their predecessor has ended must still see all of its work, on one stream, behind an event of
another stream, and in a captured graph."""
import numpy as np
import pytest
import torch

from oracle import asl_oracle as O
from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import inputs as I

from asl_check import make_path

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("how", ["one stream", "events", "graph"])
@pytest.mark.parametrize("T", [3000, 40000])
def test_select_compact_and_rank_chains(T, how):
    w, rounds = 32, 6
    wl = I.workload("C1", seqlens=(T + w,), budgets=(w + T // 5,), l_min=0, l_obs=rounds)
    path = make_path(wl)
    H, d = wl.n_kv_heads, 128
    g = torch.Generator(device="cuda").manual_seed(T)
    scores = torch.rand((rounds, H, T), generator=g, device="cuda")
    keys = torch.randint(-30000, 30000, (rounds, T + w, H, d), generator=g, device="cuda", dtype=torch.int16)
    kv, agg = torch.empty((H, T), device="cuda"), torch.empty(T, device="cuda")
    k, v = torch.empty_like(keys[0]), torch.empty_like(keys[0])
    outs = [(torch.empty_like(path.idx), torch.empty_like(path.k_out), torch.empty_like(path.v_out), torch.empty_like(path.rank_ring[0]))
            for _ in range(rounds)]
    side = torch.cuda.Stream()

    def chain():
        main = torch.cuda.current_stream()
        for r, (idx, k_out, v_out, row) in enumerate(outs):
            kv.copy_(scores[r])
            agg.copy_(scores[r, 0])
            if how == "one stream":
                k.copy_(keys[r])
                v.copy_(keys[r])
            else:                                             # the keys come from another stream
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    k.copy_(keys[r])
                    v.copy_(keys[r])
            B.asl_select_topk(path.ctx, kv, H, path.idx, path.workspace, path.ws_bytes)
            if how != "one stream":
                main.wait_stream(side)
            B.asl_compact_kv(path.ctx, k, v, path.idx, path.k_out, path.v_out)
            idx.copy_(path.idx)
            k_out.copy_(path.k_out)
            v_out.copy_(path.v_out)
            B.asl_rank_stat(path.ctx, agg, r, r + 1, path.rank_ring, path.stat, path.workspace, path.ws_bytes)
            row.copy_(path.rank_ring[r])

    chain()                                                   # (once before a capture)
    if how == "graph":
        torch.cuda.synchronize()
        for o in outs:
            for t in o:
                t.zero_()
        path.stat.zero_()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        graph.replay()
    torch.cuda.synchronize()
    s, kk, ranks = scores.cpu().numpy(), keys.cpu().numpy(), []
    for r, (idx, k_out, v_out, row) in enumerate(outs):
        got_k = k_out.view(torch.int16).cpu().numpy()
        for h in range(H):
            ref = O.select_topk(s[r, h].astype(np.float64), T // 5, T + w, w)
            assert (idx[h].cpu().numpy() == ref).all(), (r, h)
            assert (got_k[h] == kk[r, ref, h]).all(), (r, h)
        assert torch.equal(k_out.view(torch.int16), v_out.view(torch.int16))
        ranks.append(O.rank_desc(s[r, 0].astype(np.float64)))
        assert (row.cpu().numpy() == ranks[-1]).all(), r
    num, m, _ = O.rank_statistic(np.stack(ranks), T // 5)
    stat = path.read_stat()[0]
    assert (stat["num"], stat["m"]) == (num, m)
    path.close()


@pytest.mark.parametrize("how", ["calls", "graph"])
@pytest.mark.parametrize("lengths", [(300,), (500, 33, 499), (40000, 700), (262145, 5000), (300000, 262200)])
def test_rank_rows_with_nothing_in_between(lengths, how):
    """Rank rows of several layers issued back to back over scores that lie ready, so that every kernel of the row follows
    another of the library's: counted, split and radix rows (whose passes read what the kernel just before has written)."""
    w, rounds = 32, 5
    wl = I.workload("C1", seqlens=tuple(T + w for T in lengths), budgets=tuple(w + T // 9 for T in lengths), l_min=0, l_obs=rounds)
    path = make_path(wl)
    g = torch.Generator(device="cuda").manual_seed(len(lengths) + lengths[0])
    scores = torch.randn((rounds, path.sum_T), generator=g, device="cuda")

    def chain():
        for r in range(rounds):
            B.asl_rank_stat(path.ctx, scores[r], r, r + 1, path.rank_ring, path.stat, path.workspace, path.ws_bytes)

    chain()
    if how == "graph":
        torch.cuda.synchronize()
        path.rank_ring.fill_(-1)
        path.stat.zero_()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        graph.replay()
    got, s, stat, at = path.rank_ring.cpu().numpy(), scores.cpu().numpy().astype(np.float64), path.read_stat(), 0
    for b, T in enumerate(lengths):
        ranks = np.stack([O.rank_desc(s[r, at:at + T]) for r in range(rounds)])
        assert (got[:, at:at + T] == ranks).all(), b
        num, m, _ = O.rank_statistic(ranks, T // 9)
        assert (stat[b]["num"], stat[b]["m"]) == (num, m)
        at += T
    path.close()


def _score(path, x, lse, out):
    if lse is None:
        B.asl_score_layer(path.ctx, x[0], x[1], *out, path.workspace, path.ws_bytes)
    else:
        B.asl_score_layer_lse(path.ctx, x[0], x[1], lse, *out, path.workspace, path.ws_bytes)


@pytest.mark.parametrize("how", ["calls", "graph"])
@pytest.mark.parametrize("mode,seqlens", [(I.POOL_AVG, (2900,)), (I.POOL_AVG, (40001, 3000)), (I.POOL_MAX, (9000, 20011))])
def test_layers_on_one_stream_with_nothing_in_between(mode, seqlens, how):
    """Scorer, pooling, rank row, top-k and both gathers, six layers of other inputs in a row, every call right behind the one
    whose results it reads and into buffers of its own; one-pass scoring in turn with two-pass, whose offsets are kept in two
    sets.  The same, bit for bit, as with a synchronize after every call."""
    w, rounds = 32, 6
    wl = I.workload("C3", n_q_heads=8, n_kv_heads=2, window=w, pool_mode=mode, pool_kernel=5, seqlens=seqlens,
                    budgets=tuple(w + n // 6 for n in seqlens), layers=1, l_min=1, l_obs=rounds, distractors=0)
    path = make_path(wl)
    H, d, n = wl.n_kv_heads, wl.head_dim, path.sum_tokens
    g = torch.Generator(device="cuda").manual_seed(n)
    rand = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
    inputs = [(rand(len(seqlens), wl.n_q_heads, w, d), rand(n, H, d), rand(n, H, d), rand(n, 2112)) for _ in range(rounds)]
    lses = [None] * rounds
    for r in range(1, rounds, 2):                              # every second layer in one pass over K
        _score(path, inputs[r], None, (path.scores_kv, path.scores_agg))
        lses[r] = torch.empty((len(seqlens), wl.n_q_heads, w), device="cuda")
        B.asl_window_lse(path.ctx, path.workspace, path.ws_bytes, lses[r])
    torch.cuda.synchronize()

    def buffers():
        return [(torch.zeros((H, path.sum_T), device="cuda"), torch.zeros(path.sum_T, device="cuda"), torch.zeros_like(path.idx),
                 torch.zeros_like(path.k_out), torch.zeros_like(path.v_out), torch.zeros((path.sum_kept,), dtype=torch.int32, device="cuda"),
                 torch.zeros((path.sum_kept, 2112), dtype=torch.bfloat16, device="cuda")) for _ in range(rounds)]

    def chain(outs, between=lambda: None):
        for r, (x, (kv, agg, idx, k_out, v_out, one, rows)) in enumerate(zip(inputs, outs)):
            for call in (lambda: _score(path, x, lses[r], (kv, agg)),
                         lambda: B.asl_rank_stat(path.ctx, agg, r, r + 1, path.rank_ring, path.stat, path.workspace, path.ws_bytes),
                         lambda: B.asl_select_topk(path.ctx, kv, H, idx, path.workspace, path.ws_bytes),
                         lambda: B.asl_compact_kv(path.ctx, x[1], x[2], idx, k_out, v_out),
                         lambda: B.asl_select_topk(path.ctx, agg, 1, one, path.workspace, path.ws_bytes),
                         lambda: B.asl_compact_rows(path.ctx, x[3], one, rows, 4224)):
                call()
                between()

    def state():
        path.stat.zero_()
        path.rank_ring.zero_()
        torch.cuda.synchronize()

    alone, outs = buffers(), buffers()
    state()
    chain(alone, torch.cuda.synchronize)
    ring, stat = path.rank_ring.clone(), path.read_stat().copy()
    state()
    if how == "graph":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain(outs)
        for _ in range(2):                                     # replays follow one another as calls do
            graph.replay()
        path.stat.zero_()
        graph.replay()
    else:
        chain(outs)
    torch.cuda.synchronize()
    for r, (a, o) in enumerate(zip(alone, outs)):
        for i, (x, y) in enumerate(zip(a, o)):
            assert torch.equal(x, y), (r, i)
    assert torch.equal(ring, path.rank_ring) and path.read_stat().tobytes() == stat.tobytes()
    assert B.asl_device_status(path.ctx)[0] == 0
    at = 0
    for b, n_b in enumerate(seqlens):                          # and right: lists, rows and ranks of the scores, by the oracle
        T, kept, s = n_b - w, w + n_b // 6, alone[-1][1].cpu().numpy().astype(np.float64)
        here, k0 = slice(int(path.t_off[b]), int(path.t_off[b]) + T), int(path.kept_off[b])
        assert (ring[rounds - 1, here].cpu().numpy() == O.rank_desc(s[here])).all()
        ref = O.select_topk(s[here], kept - w, n_b, w)
        assert (alone[-1][5][k0:k0 + kept].cpu().numpy() == ref).all()
        assert torch.equal(alone[-1][6][k0:k0 + kept], inputs[-1][3][at + torch.from_numpy(ref).cuda()])
        at += n_b
    path.close()

"""The one-CTA top-k where the last digits of the k-th key are settled by comparing the few keys of one bin (128 at most: bins
of 127, 128 and 129 keys, and some that are split further), where all keys equal to it are kept or some of them, and where the
kept tokens come in passages (words of the bitmap that a whole warp writes: none, a few, all of a warp's)."""
import numpy as np
import pytest

from paper_2601_07667_b200 import inputs as I

from test_gpu_parity import _topk_against_the_oracle

pytestmark = pytest.mark.gpu


def _row(T, k, kind, rng):
    s = np.exp(rng.normal(-9.0, 1.5, size=T))
    if kind[0] in ("equal", "apart"):                    # `more` + 1 tokens share the k-th score, one or all of them kept
        more, one = kind[1:]
        order = np.argsort(-s, kind="stable")
        first = k - 1 if one else max(0, k - 1 - more)
        s[order[first:first + 1 + more]] = s[order[first]]
        if kind[0] == "apart":                           # and have their bin to themselves
            s[order[:first]] *= 1.25
            s[order[first + 1 + more:]] /= 1.25
    elif kind[0] == "passages":                          # runs of `length` tokens far above the rest
        length = kind[1]
        for f in rng.permutation(T // length)[:max(1, k // length)]:
            s[f * length:(f + 1) * length] += 1.0
    return s.astype(np.float32)


@pytest.mark.parametrize("kind", [("smooth",), ("equal", 5, True), ("equal", 5, False), ("equal", 511, True), ("equal", 511, False),
                                  ("equal", 700, True), ("equal", 700, False), ("apart", 126, True), ("apart", 127, True),
                                  ("apart", 127, False), ("apart", 128, True), ("apart", 128, False), ("passages", 17), ("passages", 128), ("passages", 1500)])
@pytest.mark.parametrize("T,k", [(900, 800), (4097, 1000), (12288, 3000), (12289, 3000), (33001, 4000), (66003, 9000)])
def test_topk(T, k, kind):
    w, heads = 32, 3
    wl = I.workload("C1", n_q_heads=heads, n_kv_heads=heads, seqlens=(T + w, 40 + w), budgets=(k + w, 20 + w))
    rng = np.random.default_rng(T + k)
    rows = [np.concatenate([_row(T, k, kind, rng), rng.random(40).astype(np.float32)]) for _ in range(heads)]
    _topk_against_the_oracle(wl, np.stack(rows))

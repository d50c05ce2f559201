"""GPU parity of the one-CTA top-k where its list, its two sampled bounds and its staged output begin and end."""
import numpy as np
import pytest

from paper_2601_07667_b200 import inputs as I

from test_gpu_parity import _topk_against_the_oracle

pytestmark = pytest.mark.gpu
CAP = 12288                                              # scores the kernel lists


@pytest.mark.parametrize("kind", ["smooth", "signed", "ties", "steps"])
@pytest.mark.parametrize("T,k,heads", [                  # many heads: one CTA per segment whatever k; few: large k is tiled
    (1, 1, 2), (31, 30, 2), (1025, 1, 2), (CAP - 1, 700, 2), (CAP, CAP - 1, 2), (CAP + 1, 12, 2), (24577, 24576, 32),
    (30001, 15000, 2), (30001, 15000, 16), (70003, 24576, 32), (70003, 24577, 32), (70003, 69999, 2), (131071, 2 * CAP + 5, 32),
    (131071, 2 * CAP + 5, 2), (262144, 5000, 16), (262144, 131072, 2), (262145, 4000, 2),
])
def test_topk(T, k, heads, kind):
    w = 32
    wl = I.workload("C1", n_q_heads=heads, n_kv_heads=heads, seqlens=(T + w, 77 + w), budgets=(k + w, 20 + w))     # odd heads start off 16 bytes
    rng = np.random.default_rng(T + k)
    s = rng.normal(-9.0, 1.5, size=(wl.n_kv_heads, T + 77))
    if kind == "smooth":
        s = np.exp(s)
    elif kind == "ties":                                 # a step at the k-th score: equal scores fill the list and more
        s = np.where(rng.random(s.shape) < 0.7 * k / T, 1.0 + np.round(rng.random(s.shape), 2), np.round(rng.random(s.shape)) / 2)
    elif kind == "steps":                                # large scores only where the sample does not look, or only there
        s = np.exp(s)
        at = (np.arange(2048, dtype=np.int64) * T) // 2048
        s[0, at] += 1.0
        s[1, :T] += 1.0
        s[1, at] -= 1.0
    _topk_against_the_oracle(wl, s.astype(np.float32))

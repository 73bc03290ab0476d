"""The top-k of given scores at the edges of the select's shapes (candidates a
CTA and a cluster hold) and for the scores its histogram handles worst: the
k-th largest in a range of more keys than are ranked directly, outliers that
stretch the first histogram, ties at the cut, infinities."""
import numpy as np
import pytest
import torch

from paper_2609_06663_gb300 import ecokv as E

pytestmark = pytest.mark.gpu

# 8 / 16 / 32 candidates a thread, one CTA and several, the last one ragged
SIZES = [1, 255, 2048, 2049, 8192, 8193, 16384, 16385, 32768, 32769, 131072]


def scores(kind, t, g):
    if kind == "spread":      # over thirty binades, both signs
        x = torch.randn(t, generator=g) * torch.exp2(torch.randint(-20, 11, (t,), generator=g).float())
    elif kind == "narrow":    # neighbouring floats, two outliers that set the first range
        x = 1.0 + torch.randint(0, 3 * t, (t,), generator=g).float() * 2.0 ** -23
        x[:1] = 3e38
        x[-1:] = -3e38
    elif kind == "ties":      # most scores equal, the cut among them
        x = torch.where(torch.rand(t, generator=g) < 0.9, torch.tensor(0.25), torch.rand(t, generator=g))
    elif kind == "equal":
        x = torch.zeros(t)
        x[::3] = -0.0
    else:                     # infinities on both sides
        x = torch.randn(t, generator=g)
        x[torch.rand(t, generator=g) < 0.2] = float("inf")
        x[torch.rand(t, generator=g) < 0.2] = float("-inf")
    return x


@pytest.mark.parametrize("kind", ["spread", "narrow", "ties", "equal", "inf"])
@pytest.mark.parametrize("t", SIZES)
def test_select_at_shape_edges(t, kind):
    g = torch.Generator().manual_seed(t)
    window = 4
    S = torch.stack([scores(kind, t, g) for _ in range(2)])[None]
    for k in sorted({1, max(1, t // 10), max(1, t // 2), t}):
        if k + window >= t + window:  # a budget of n or more keeps every row
            continue
        p = E.make_params(n_layers=1, h_kv=2, h_q=2, n=t + window, window=window, budget=k + window)
        idx = E.select(p, S.cuda()).cpu().numpy()
        for h in range(2):
            x = S[0, h].double().numpy()
            want = np.sort(np.lexsort((np.arange(t), -x))[:k])
            assert (idx[0, h, :k] == want).all(), f"t={t} k={k} {kind} head {h}"
            assert (idx[0, h, k:] == np.arange(t, t + window)).all()


@pytest.mark.parametrize("t,heads", [(12000, 120), (16384, 120), (20001, 110), (32768, 114), (2048, 700), (9000, 300)])
def test_select_many_heads(t, heads):
    # so many heads that their CTAs take the shapes of 16 and 32 candidates a
    # thread, or (too many for one wave in any shape) clusters of at most four
    g = torch.Generator().manual_seed(t)
    window, k = 4, t // 10
    S = torch.randn(1, heads, t, generator=g)
    S[0, ::3] = (S[0, ::3] * 8).round() / 8  # ties
    p = E.make_params(n_layers=1, h_kv=heads, h_q=heads, n=t + window, window=window, budget=k + window)
    idx = E.select(p, S.cuda()).cpu().numpy()
    for h in [0, 1, 2, heads // 2, heads - 1]:
        x = S[0, h].double().numpy()
        want = np.sort(np.lexsort((np.arange(t), -x))[:k])
        assert (idx[0, h, :k] == want).all(), f"t={t} head {h} of {heads}"

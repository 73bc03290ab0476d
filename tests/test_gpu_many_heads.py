"""More heads than are resident at once: the finalisation in clusters of one to
four small CTAs, and the shapes past them, at the edges of a CTA's candidates."""
import numpy as np
import pytest
import torch

from paper_2609_06663_gb300 import ecokv as E

pytestmark = pytest.mark.gpu
W = 4


@pytest.mark.parametrize("t", [1, 127, 2047, 2048, 2049, 4097, 6145, 8191, 8192, 8193])
def test_select_of_many_heads(t):
    heads, g = 1100, torch.Generator().manual_seed(t)
    S = torch.randn(1, heads, t, generator=g)
    S[:, ::3] = torch.round(4 * S[:, ::3]) / 4  # ties at the cut
    k = max(0, min(t - 1, t // 3))
    p = E.make_params(n_layers=1, h_kv=heads, h_q=heads, n=t + W, window=W, budget=k + W)
    idx = E.select(p, S.cuda()).cpu().numpy()[0]
    x = S[0].numpy()
    for h in range(0, heads, 7):
        assert (idx[h, :k] == np.sort(np.argsort(-x[h], kind="stable")[:k])).all()
        assert (idx[h, k:] == np.arange(t, t + W)).all()


@pytest.mark.parametrize("n,flags", [(300, 0), (2048 + W, 0), (2049 + W, 0), (4100, E.ECOKV_FLAG_MAD), (8192 + W, 0),
                                     (3000, E.ECOKV_FLAG_WINSOR_5)])
def test_scores_of_many_heads(n, flags):
    # The same heads scored a layer at a time, where other shapes take them:
    # every sum runs over the same terms in fp32 groups and, across threads, in
    # another order, in the passes too; the error of a sum of m terms in groups
    # is a few times 2^-24, and S is formed from four such sums and their
    # ratios: 2^-17 of the largest score.  The rows kept differ only where
    # scores are that close, so they are checked against this call's scores.
    layers, heads = 24, 32
    g = torch.Generator(device="cuda").manual_seed(n)
    K = torch.randn(layers, heads, n, 128, device="cuda", generator=g).to(torch.bfloat16)
    Q = torch.randn(layers, heads, W, 128, device="cuda", generator=g).to(torch.bfloat16)
    budget = W + (n - W) // 4
    kw = dict(h_kv=heads, h_q=heads, n=n, window=W, budget=budget, flags=flags, sched_wave=0)
    p = E.make_params(n_layers=layers, **kw)
    idx, Ko, _, S, lam = E.evict(p, K, K, Q, want_scores=True)
    one = E.make_params(n_layers=1, **kw)
    for l in (0, 11, 23):
        S1, lam1, _ = E.score(one, K[l:l + 1], Q[l:l + 1])
        top = S1.abs().amax(-1, keepdim=True)
        assert ((S[l:l + 1] - S1).abs() <= 2.0 ** -17 * top).all()
        assert (lam[l] - lam1[0]).abs().max() <= 1e-5
        x = S[l].cpu().numpy()
        got = idx[l].cpu().numpy()
        for h in range(0, heads, 5):
            k = budget - W
            assert (got[h, :k] == np.sort(np.argsort(-x[h], kind="stable")[:k])).all()
            assert torch.equal(Ko[l, h], K[l, h][idx[l, h].long()])

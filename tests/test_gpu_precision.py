"""What single precision may cost where a sum or a reference was split otherwise:
errors against 64 bits, bounded by the roundings of the path."""
import pytest
import torch

from paper_2609_06663_gb300 import ecokv as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sched_wave", [0, 32], ids=["short_units", "streaming"])
def test_vote_of_rows_whose_first_keys_lie_far_below_the_maximum(sched_wave):
    """The keys that a warp's partial sums are taken against (the first of every 32)
    have logits 50 binary orders below the others', so that a row's sum is about
    2^50 of its reference while its log-sum-exp is near 0.  The error that a
    head's votes share is the row's: at most the approximate exponentials of one
    term (pass 1, two folds, pass 2; 2^-22 each), 2^-20 in all (measured: 4.6e-7).
    A log2 of the sum rounded at its own size of 50 alone may add 1.3e-6."""
    g = torch.Generator(device="cuda").manual_seed(3)
    h, n = 32, 1000
    K = torch.randn(1, h, n, 128, device="cuda", generator=g)
    K[..., 0] = -6 + 2 * torch.rand(1, h, n, device="cuda", generator=g)
    K[:, :, ::32, 0] = -25 - torch.rand(1, h, (n + 31) // 32, device="cuda", generator=g)
    K = K.bfloat16()
    Q = torch.zeros(1, h, 1, 128, device="cuda")
    Q[..., 0] = 16
    p = E.make_params(n_layers=1, h_kv=h, h_q=h, n=n, window=1, budget=100, sched_wave=sched_wave)
    _, _, dbg = E.score(p, K, Q.bfloat16(), dbg=True)
    vote = torch.softmax(K[0, :, :, 0].double() * 16 / 128 ** 0.5, dim=1)[:, :-1]
    others = torch.arange(n - 1, device="cuda") % 32 != 0
    shared = (dbg[0, :, 0].double() / vote - 1)[:, others].mean(1)
    assert float(shared.abs().max()) <= 2.0 ** -20, shared


@pytest.mark.parametrize("heads,n", [(152, 640), (76, 1280), (15, 5120)], ids=lambda v: str(v))
def test_mean_direction_of_short_units_of_five_tiles_a_cta(heads, n):
    """With beta = 0 lambda is r_C = (n ||mu||^2 - 1) / (n - 1).  The tensor core
    accumulates towards zero: each of a tile's eight steps loses up to 2^-23 of
    the sum so far, half of it in the mean, so a tile's sum is short by at most
    4.5 * 2^-24 and ||mu||^2 by twice that, however many tiles a CTA holds.  A
    sum that runs on over five tiles is short by five times as much."""
    g = torch.Generator(device="cuda").manual_seed(5)
    u = torch.randn(heads, 1, 128, device="cuda", generator=g)
    u = u / torch.linalg.vector_norm(u, dim=2, keepdim=True)
    K = (6 * u + 0.6 * torch.randn(heads, n, 128, device="cuda", generator=g)).bfloat16()[None]
    Q = torch.randn(1, heads, 1, 128, device="cuda", generator=g).bfloat16()
    p = E.make_params(n_layers=1, h_kv=heads, h_q=heads, n=n, window=1, budget=n // 4, beta=0.0)
    _, lam, _ = E.score(p, K, Q)
    k = K[0].double()
    mu = (k / torch.linalg.vector_norm(k, dim=2, keepdim=True)).mean(1)
    r_c = (n * (mu * mu).sum(1) - 1) / (n - 1)
    bias = float(((lam[0].double() - r_c) / r_c).mean())
    assert abs(bias) <= 2 * 4.5 * 2.0 ** -24, bias

"""The short-unit kernel (one cluster per head, both passes, scores and selection
in one launch) against the oracle, at the edges of what it takes and of how it
splits a head: one tile to eighty, one CTA a head to sixteen, one to five tiles
a CTA, a ragged last tile, each instance by window rows; and against the
persistent kernel, which an explicit schedule selects."""
import pytest
import torch

from paper_2609_06663_gb300 import ecokv as E
from paper_2609_06663_gb300.workloads import make_inputs, small_workload
from tests.test_gpu_parity import params_of, run_and_compare

pytestmark = pytest.mark.gpu


# n, heads: tiles a head and CTAs a head follow (at most tiles, eight, and as many
# as leave every head's cluster on the device at once, or sixteen for a few heads
# of more than sixteen tiles)
@pytest.mark.parametrize("n,h_kv,group,window", [
    (128, 1, 1, 1), (129, 2, 1, 8), (255, 3, 2, 8), (640, 1, 4, 4), (1024, 8, 4, 4), (1025, 8, 7, 8),
    (640, 100, 1, 8), (1280, 75, 1, 4), (1281, 50, 2, 8), (2560, 38, 1, 4), (3001, 8, 8, 8), (5003, 4, 7, 8),
    (5120, 19, 2, 16), (5120, 1, 4, 16),
    (2049, 7, 4, 8), (6000, 3, 8, 8), (8200, 7, 1, 8), (10240, 2, 7, 8),
    # the most heads that clusters of eight, six, five, four, three and two CTAs hold at
    # once, of the most tiles, and one head more
    (5120, 15, 1, 8), (5120, 16, 1, 8), (3840, 23, 1, 8), (3200, 24, 1, 8), (3200, 28, 1, 8), (2560, 36, 1, 8),
    (1920, 46, 1, 8), (1280, 47, 1, 8), (1280, 76, 1, 8), (640, 77, 1, 8)], ids=lambda v: str(v))
def test_short_unit_shapes(n, h_kv, group, window):
    units = None if h_kv <= 8 else [(0, 0), (0, h_kv // 2), (0, h_kv - 1)]
    run_and_compare(small_workload(n, h_kv=h_kv, group=group, window=window, budget=max(window, n // 10), dtype="bf16",
                                   seed=n, clustered=True), units=units)


@pytest.mark.parametrize("kw", [dict(pool_kernel=1), dict(pool_kernel=33), dict(pool_kernel=41)], ids=str)
def test_short_unit_pooling(kw):
    # halos across the cluster's CTAs, and pooling wider than the staged halo
    run_and_compare(small_workload(3000, h_kv=2, group=4, window=8, budget=300, dtype="bf16", clustered=True, **kw))


def test_short_unit_options():
    w = small_workload(2000, h_kv=2, group=2, window=8, budget=2100, dtype="bf16", n_layers=2)   # B >= N
    run_and_compare(w)
    w = small_workload(2000, h_kv=2, group=2, window=8, budget=8, dtype="bf16", n_layers=2)      # B == W
    run_and_compare(w)
    w = small_workload(2000, h_kv=2, group=2, window=8, budget=200, dtype="bf16", n_layers=2)
    run_and_compare(w, flags=E.ECOKV_FLAG_CENTROID_NONWIN)
    run_and_compare(w, flags=E.ECOKV_FLAG_SC_MIXKV_SIGN)
    run_and_compare(w, flags=E.ECOKV_FLAG_LAMBDA_OVERRIDE, lambda_override=0.25)


def test_short_unit_per_layer_budgets():
    w = small_workload(3000, h_kv=2, group=4, window=8, budget=600, dtype="bf16", n_layers=3)
    K, V, Q = (t.cuda() for t in make_inputs(w))
    p = params_of(w)
    budgets = [600, 8, 300]
    idx, Ko, Vo, S, _ = E.evict_layered(p, K, V, Q, budgets, want_scores=True)
    for l, b in enumerate(budgets):
        pl = params_of(w)
        pl.n_layers, pl.budget = 1, b
        want = E.select(pl, S[l:l + 1].contiguous())[0]
        assert torch.equal(idx[l, :, :b], want) and bool((idx[l, :, b:] == -1).all())
        for h in range(w.h_kv):
            rows = want[h].long()
            assert torch.equal(Ko[l, h, :b], K[l, h][rows]) and torch.equal(Vo[l, h, :b], V[l, h][rows])


@pytest.mark.parametrize("n", [300, 3000])
def test_short_unit_matches_the_persistent_kernel(n):
    """The same scores as the persistent kernel to the rounding of sums taken
    in another order: about 2^-20 of the largest score for each of a few
    thousand single-precision terms, the selection exact on its own scores."""
    w = small_workload(n, h_kv=4, group=4, window=8, budget=n // 5, dtype="bf16", seed=9, clustered=True)
    K, V, Q = (t.cuda() for t in make_inputs(w))
    p = params_of(w)
    idx, _, _, S, lam = E.evict(p, K, V, Q, want_scores=True)
    _, _, _, S2, lam2 = E.evict(params_of(w, sched_wave=4), K, V, Q, want_scores=True)
    assert float((S - S2).abs().max()) <= 2.0 ** -17 * float(S2.abs().max())
    assert float((lam - lam2).abs().max()) <= 2.0 ** -17
    assert torch.equal(idx, E.select(p, S))


@pytest.mark.parametrize("heads,tiles", [(15, 8), (23, 6), (28, 5), (36, 4), (46, 3)], ids=lambda v: str(v))
def test_one_head_more_takes_no_second_wave(heads, tiles):
    """The most heads whose clusters of seven or eight, six, five, four or three
    CTAs are on a GB300 at once, and one head more, which fewer CTAs a head
    keep there: a cluster that waits for the first ones to end makes a call
    1.5 times as long, the smaller clusters at most 1.1 times."""
    n, times = 128 * tiles, []
    for h in (heads, heads + 1):
        K = torch.randn(1, h, n, 128, device="cuda").bfloat16()
        Q = torch.randn(1, h, 8, 128, device="cuda").bfloat16()
        p = E.make_params(n_layers=1, h_kv=h, h_q=h, n=n, window=8, budget=n // 10)
        ws = E.alloc_workspace(p)
        S, lam = torch.empty(1, h, n - 8, device="cuda"), torch.empty(1, h, device="cuda")

        def batch():
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(100):
                assert E.ecokv_score(p, E.ECOKV_BF16, K, Q, S, lam, None, ws, ws.numel(),
                                     torch.cuda.current_stream()) == 0
            b.record()
            b.synchronize()
            return a.elapsed_time(b)

        batch()
        times.append(min(batch() for _ in range(8)))
    assert times[1] <= 1.3 * times[0], times

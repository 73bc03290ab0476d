"""The tensor-core kernel's instances by window rows: the smallest and largest
row count of each (its padding rows, the columns read at once, two or three
tile groups), over slices of several tiles with a ragged end, against the fp64
oracle."""
import pytest
import torch

from oracle import ecokv_oracle as O
from paper_2609_06663_gb300 import ecokv as E
from paper_2609_06663_gb300.workloads import make_inputs, small_workload
from tests.parity import TOL, check_scores, check_selection, oracle_params
from tests.test_gpu_parity import params_of, run_and_compare

pytestmark = pytest.mark.gpu


# g x W window rows: instances of 8, 16, 32, 56, 64, 112 and 128 rows
@pytest.mark.parametrize("group,window", [(1, 1), (1, 8), (3, 3), (2, 8), (1, 17), (4, 8), (3, 11), (7, 8), (3, 19),
                                          (8, 8), (5, 13), (7, 16), (1, 113), (8, 15)],
                         ids=lambda v: str(v))
def test_window_row_instances(group, window):
    # 470 tiles of one head: three or four a CTA, so that every tile group
    # works and pass 2 walks back over more than one tile
    run_and_compare(small_workload(60001, h_kv=1, group=group, window=window, budget=6000, dtype="bf16", seed=2))


@pytest.mark.parametrize("group,window", [(1, 8), (7, 8), (7, 16)], ids=lambda v: str(v))
def test_logits_that_outgrow_their_reference(group, window):
    """Keys that grow along the sequence: the logits of a slice's later tiles
    exceed the first key's by far more than 2^6, so that the reference of the
    partial sums has to be raised, several times over."""
    w = small_workload(60000, h_kv=1, group=group, window=window, budget=6000, dtype="bf16", seed=4)
    K, V, Q = make_inputs(w)
    ramp = torch.linspace(0.2, 30.0, 128).repeat((w.n + 127) // 128)[:w.n]
    tile = torch.arange(w.n) // 128 % 4
    K = (K.float() * (ramp * (1.0 + tile))[None, None, :, None]).to(torch.bfloat16)
    p = params_of(w)
    op = oracle_params(p)
    idx, _, _, S, lam = E.evict(p, K.cuda(), V.cuda(), Q.cuda(), want_scores=True)
    r = O.evict(K, V, Q, op)[(0, 0)]
    check_scores(S[0, 0].cpu().double().numpy(), r, TOL["bf16"], "growing keys")
    check_selection(idx[0, 0].cpu().numpy(), r, op, TOL["bf16"], "growing keys")
    assert abs(float(lam[0, 0]) - r["lam"]) <= TOL["bf16"]


@pytest.mark.parametrize("group,window", [(4, 32), (8, 16), (8, 32)], ids=lambda v: str(v))
def test_128_rows_in_one_launch(group, window):
    # more than 64 MB of keys: up to 128 window rows a launch (256 rows: two),
    # the odd last tile with keys that not every row sees
    run_and_compare(small_workload(33001, h_kv=8, group=group, window=window, budget=3300, dtype="bf16", seed=6),
                    units=[(0, 0), (0, 7)])


# waves of few heads past 64 window rows, where the warps that fold the
# statistics also compute pass 1's norms: their wait for a key tile that follows
# tiles of pass 2 in the ring (slices of one to three tiles, and of more tiles
# than the ring has stages)
@pytest.mark.parametrize("n,wave,lag", [(5000, 1, 1), (5000, 1, 2), (5000, 2, 1), (5000, 5, 1), (19500, 1, 1),
                                        (19500, 5, 1), (40001, 3, 1)], ids=lambda v: str(v))
def test_schedules_of_112_rows(n, wave, lag):
    run_and_compare(small_workload(n, h_kv=2, group=7, window=16, budget=500, dtype="bf16", n_layers=3, seed=8,
                                   clustered=True),
                    units=[(0, 0), (1, 1), (2, 1)], sched_wave=wave, sched_lag=lag, timeout_us=200000)


@pytest.mark.parametrize("wave,lag", [(1, 1), (2, 1), (5, 1), (3, 2)], ids=lambda v: str(v))
def test_schedules_of_128_rows_in_one_launch(wave, lag):
    run_and_compare(small_workload(33001, h_kv=8, group=8, window=16, budget=3300, dtype="bf16", seed=6),
                    units=[(0, 0), (0, 7)], sched_wave=wave, sched_lag=lag, timeout_us=200000)

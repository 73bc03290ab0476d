"""Bounded device-side waits, made to run out on purpose without faulting the
GPU: with ECOKV_FLAG_TEST_STALL the statistics of the first unit never
complete (the streaming kernel expects one more pass-1 arrival than there are
pass-1 items; the short-unit kernel, which takes this shape unless a schedule
is asked for, leaves out the product of one CTA's keys with the statistics), so
the wait of its pass 2 gives up after timeout_us.  The call
must report ECOKV_ERR_TIMEOUT through ecokv_device_status, return well before
the default 2 s limit, and leave the context and the workspace usable: the
next call on the same workspace is bit for bit the call on a fresh one, and
matches the oracle."""
import time

import pytest
import torch

from oracle import ecokv_oracle as O
from paper_2609_06663_gb300 import ecokv as E
from paper_2609_06663_gb300.workloads import make_inputs, small_workload
from tests.parity import TOL, check_rows, check_scores, check_selection, oracle_params

pytestmark = pytest.mark.gpu
DEV = "cuda"


def params_of(w, **kw):
    return E.make_params(n_layers=w.n_layers, h_kv=w.h_kv, h_q=w.h_q, n=w.n, d=w.d, window=w.window,
                         budget=w.budget, pool_kernel=w.pool_kernel, **kw)


@pytest.mark.parametrize("sched_wave", [0, 4], ids=["short_units", "streaming"])
def test_stalled_statistics_time_out_and_the_workspace_recovers(sched_wave):
    w = small_workload(3000, h_kv=2, group=4, window=8, budget=300, dtype="bf16", n_layers=2, clustered=True)
    K, V, Q = make_inputs(w)
    Kd, Vd, Qd = K.to(DEV), V.to(DEV), Q.to(DEV)
    p_stall = params_of(w, flags=E.ECOKV_FLAG_TEST_STALL, timeout_us=20000, sched_wave=sched_wave)
    p = params_of(w, sched_wave=sched_wave)
    assert E.ecokv_workspace_size(p_stall) == E.ecokv_workspace_size(p)
    ws = E.alloc_workspace(p, DEV)
    torch.cuda.synchronize()

    t0 = time.perf_counter()
    E.evict(p_stall, Kd, Vd, Qd, ws=ws)  # enqueued; the failure shows on the device only
    status = E.ecokv_device_status(ws)   # synchronises
    elapsed = time.perf_counter() - t0
    assert status == E.ECOKV_ERR_TIMEOUT, E.STATUS.get(status, status)
    assert elapsed < 1.0, f"the 20 ms limit took {elapsed:.3f} s to fire"
    assert E.ecokv_device_status(ws) == 0  # reading the status cleared it

    # the same workspace right after the aborted call, and a fresh one
    idx, Ko, Vo, S, lam = E.evict(p, Kd, Vd, Qd, ws=ws, want_scores=True)
    idx2, Ko2, Vo2, S2, lam2 = E.evict(p, Kd, Vd, Qd, want_scores=True)
    torch.cuda.synchronize()
    assert E.ecokv_device_status(ws) == 0
    assert torch.equal(S, S2) and torch.equal(lam, lam2) and torch.equal(idx, idx2)
    assert torch.equal(Ko, Ko2) and torch.equal(Vo, Vo2)

    op = oracle_params(p)
    ref = O.evict(K, V, Q, op)
    S_np = S.cpu().double().numpy()
    for (l, h), r in ref.items():
        what = f"unit ({l},{h}) after a timed-out call"
        check_scores(S_np[l, h], r, TOL["bf16"], what)
        check_selection(idx[l, h].cpu().numpy(), r, op, TOL["bf16"], what)
        check_rows(Kd[l, h], idx[l, h], Ko[l, h], what)
        check_rows(Vd[l, h], idx[l, h], Vo[l, h], what)


def test_a_unit_that_gave_up_is_not_finalised():
    """Short units: where one CTA of a cluster gave up none of them goes on to
    the scores (their memory may still be the target of copies, and the counts
    they exchange would be those of no selection); the other units' results
    are those of an undisturbed call."""
    w = small_workload(3000, h_kv=2, group=4, window=8, budget=300, dtype="bf16", n_layers=2, clustered=True)
    K, V, Q = (t.to(DEV) for t in make_inputs(w))
    p_stall = params_of(w, flags=E.ECOKV_FLAG_TEST_STALL, timeout_us=20000)
    want = E.evict(params_of(w), K, V, Q, want_scores=True)
    ws = E.alloc_workspace(p_stall, DEV)
    idx, Ko, Vo, S, lam = (torch.full_like(t, -7) for t in want)
    assert E.ecokv_evict(p_stall, E.dtype_code(K), K, V, Q, idx, Ko, Vo, S, lam, ws, ws.numel()) == 0
    assert E.ecokv_device_status(ws) == E.ECOKV_ERR_TIMEOUT
    for t in (S, lam, idx):
        assert bool((t[0, 0] == -7).all())
    for got, ref in zip((idx, Ko, Vo, S, lam), want):
        assert torch.equal(got[0, 1], ref[0, 1]) and torch.equal(got[1], ref[1])


@pytest.mark.parametrize("window", [8, 28], ids=["32_rows", "112_rows"])
@pytest.mark.parametrize("sched_wave", [0, 4], ids=["default", "schedule"])
def test_a_limit_shorter_than_a_copy(sched_wave, window):
    """A limit of a microsecond may run out while the call's own copies and
    MMAs are in flight; they are waited for with a limit of their own before
    the memory they land in is given back.  Whether the call makes it or
    reports the timeout, the calls after it are undisturbed."""
    w = small_workload(9000, h_kv=2, group=4, window=window, budget=900, dtype="bf16", n_layers=2, clustered=True)
    K, V, Q = (t.to(DEV) for t in make_inputs(w))
    p, p_short = (params_of(w, sched_wave=sched_wave, timeout_us=us) for us in (0, 1))
    want = E.evict(p, K, V, Q, want_scores=True)
    ws = E.alloc_workspace(p, DEV)
    for _ in range(10):
        got = E.evict(p_short, K, V, Q, ws=ws, want_scores=True)
        status = E.ecokv_device_status(ws)
        assert status in (E.ECOKV_OK, E.ECOKV_ERR_TIMEOUT)
        if status == E.ECOKV_OK:
            assert all(torch.equal(a, b) for a, b in zip(got, want))
        got = E.evict(p, K, V, Q, ws=ws, want_scores=True)
        assert E.ecokv_device_status(ws) == E.ECOKV_OK
        assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_stall_flag_needs_the_tensor_core_path():
    """The injected stall exists only in the tensor-core kernel; elsewhere the
    flag is refused before anything is launched."""
    w = small_workload(1000, h_kv=2, group=1, window=8, budget=100, dtype="f32")
    K, V, Q = (t.to(DEV) for t in make_inputs(w))
    p = params_of(w, flags=E.ECOKV_FLAG_TEST_STALL, timeout_us=20000)
    with pytest.raises(E.EcokvError) as e:
        E.evict(p, K, V, Q)
    assert e.value.code == E.ECOKV_ERR_UNSUPPORTED

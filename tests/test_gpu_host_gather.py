"""The gather of a cache in host memory at the edges of a block's 64 rows, and
with the caller's index array off a 4-byte boundary (the indices then come by a
copy): identical to the pass on device copies."""
import pytest

torch = pytest.importorskip("torch")
from paper_2609_06663_gb300 import ecokv as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("budget,dtype,odd", [
    (9, "bf16", False), (63, "bf16", False), (64, "f32", False), (65, "bf16", False), (65, "bf16", True),
    (128, "bf16", False), (129, "f32", True), (400, "bf16", False)])
def test_host_gather_matches_device(budget, dtype, odd):
    n, W, h_kv, layers = 400, 8, 3, 2
    g = torch.Generator().manual_seed(budget)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    K, V = (torch.randn(layers, h_kv, n, 128, generator=g).to(dt) for _ in range(2))
    Q = torch.randn(layers, h_kv, W, 128, generator=g).to(dt)
    p = E.make_params(n_layers=layers, h_kv=h_kv, h_q=h_kv, n=n, window=W, budget=budget)
    n_keep = min(budget, n)
    count = layers * h_kv * n_keep
    raw = torch.full((4 * count + 16,), 0x55, dtype=torch.uint8).pin_memory()
    at = 2 if odd else 0
    Ko = torch.empty(layers, h_kv, n_keep, 128, dtype=dt).pin_memory()
    Vo = torch.empty_like(Ko).pin_memory()
    code = E.dtype_code(K)
    ws = E.alloc_workspace_host(p, code).zero_()
    hK, hV, hQ = K.pin_memory(), V.pin_memory(), Q.pin_memory()
    assert E.ecokv_evict_host(p, code, hK, hV, hQ, raw.data_ptr() + at, Ko, Vo, None, ws, ws.numel()) == 0
    torch.cuda.synchronize()
    assert E.ecokv_device_status(ws) == 0
    idx_r, Ko_r, Vo_r, _, _ = E.evict(p, K.cuda(), V.cuda(), Q.cuda())
    idx = raw[at:at + 4 * count].clone().view(torch.int32).view(layers, h_kv, n_keep)
    assert torch.equal(idx, idx_r.cpu())
    assert torch.equal(Ko, Ko_r.cpu()) and torch.equal(Vo, Vo_r.cpu())
    guard = torch.cat([raw[:at], raw[at + 4 * count:]])
    assert (guard == 0x55).all()  # nothing beside the indices is written

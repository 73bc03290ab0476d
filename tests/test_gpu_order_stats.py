"""The order statistics of the robust forms of Eq. 2 at the edges of a block's
share: rows of a few keys, rows whose 16-byte groups leave a remainder, rows
that start off a 16-byte boundary (an odd candidate count, second head), rows
that fill every slot, and the first ones that are read from L2.

The S_div that the kernels return is compared with one formed in double from
their own single-precision distances and numpy's order statistics of these; the
kernels form s_E, its weighting and the cosine term in single precision, a
handful of roundings of values up to 1, hence 2e-6 (a rank off by one moves s_E
by more than that except where the two neighbours agree)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2609_06663_gb300 import ecokv as E

pytestmark = pytest.mark.gpu
W = 8


@pytest.mark.parametrize("flags", [E.ECOKV_FLAG_WINSOR_1, E.ECOKV_FLAG_MAD], ids=["winsor1", "mad"])
@pytest.mark.parametrize("cand", [1, 3, 1027, 4095, 4097, 12273, 32767, 32768, 32769, 33001])
def test_order_statistics_at_block_edges(cand, flags):
    n, h_kv = cand + W, 2
    g = torch.Generator(device="cuda").manual_seed(cand)
    K = torch.randn(1, h_kv, n, 128, device="cuda", generator=g).to(torch.bfloat16)
    Q = torch.randn(1, h_kv, W, 128, device="cuda", generator=g).to(torch.bfloat16)
    p = E.make_params(n_layers=1, h_kv=h_kv, h_q=h_kv, n=n, window=W, budget=W + 1, flags=flags)
    ws = E.alloc_workspace(p, "cuda")
    _, _, dbg = E.score(p, K, Q, ws=ws, dbg=True)
    torch.cuda.synchronize()
    assert E.ecokv_device_status(ws) == 0
    dbg = dbg.cpu().numpy()
    for h in range(h_kv):
        dE, c = dbg[0, h, 2].astype(np.float32), dbg[0, h, 3].astype(np.float64)
        assert dE.size == cand
        srt, d = np.sort(dE), dE.astype(np.float64)
        if flags & E.ECOKV_FLAG_MAD:
            half = np.float32(0.5)
            med = half * (srt[(cand - 1) // 2] + srt[cand // 2])
            dev = np.sort(np.abs(dE - med))
            mad = half * (dev[(cand - 1) // 2] + dev[cand // 2])
            sE = 1.0 / (1.0 + np.exp(-(d - float(med)) / (float(mad) + float(p.eps))))
        else:
            lo = float(srt[int(np.floor(0.01 * (cand - 1)))])
            hi = float(srt[int(np.ceil(0.99 * (cand - 1)))])
            sE = (np.clip(d, lo, hi) - lo) / (hi - lo + float(p.eps))
        sdiv = float(p.alpha) * sE + (1.0 - float(p.alpha)) * (1.0 - c) / 2.0
        assert np.abs(dbg[0, h, 4].astype(np.float64) - sdiv).max() <= 2e-6

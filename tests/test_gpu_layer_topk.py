"""The layer-wide budget's top-k on both of its paths: layers of up to 131072
concatenated scores (one cluster) and longer ones (the layer select), with
heads whose share of the budget is uneven, checked against a sort of the
layer's own scores."""
import numpy as np
import pytest
import torch

from paper_2609_06663_gb300 import ecokv as E
from paper_2609_06663_gb300.workloads import make_inputs, small_workload
from tests.test_gpu_parity import params_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h_kv,layers", [(300, 3, 2), (4104, 4, 2), (16392, 8, 1), (16393, 8, 1), (33000, 4, 2)],
                         ids=lambda v: str(v))
def test_layer_budget_on_both_paths(n, h_kv, layers):
    w = small_workload(n, h_kv=h_kv, group=2, window=8, budget=n // 8, dtype="bf16", n_layers=layers, seed=5)
    K, V, Q = (t.cuda() for t in make_inputs(w))
    K[:, 0] *= 3.0  # one head unlike the others: its scores, and its share, differ
    p = params_of(w)
    S, _, _ = E.score(p, K, Q)
    idx, off, Ko, Vo, _ = E.evict_adaptive(p, K, V, Q)
    tv, k = n - 8, h_kv * (p.budget - 8)
    for l in range(layers):
        x = S[l].reshape(-1).double().cpu().numpy()
        chosen = np.sort(np.lexsort((np.arange(x.size), -x))[:k])
        want, at = [], [0]
        for h in range(h_kv):
            mine = chosen[(chosen >= h * tv) & (chosen < (h + 1) * tv)] - h * tv
            want += [mine, np.arange(tv, n)]
            at.append(at[-1] + mine.size + 8)
        want = np.concatenate(want)
        assert (idx[l].cpu().numpy() == want).all() and (off[l].cpu().numpy() == np.array(at)).all()
        for h in range(h_kv):
            rows = idx[l, at[h]:at[h + 1]].long()
            assert torch.equal(Ko[l, at[h]:at[h + 1]], K[l, h][rows])
            assert torch.equal(Vo[l, at[h]:at[h + 1]], V[l, h][rows])

"""The calls that are timed, with their inputs, their work and their tolerances.

A prefill engine calls the library either once per layer, as each layer's
keys become available, or once for the whole prompt over all layers; the cases
below are such calls through the C ABI's names in
paper_2609_06663_gb300.ecokv, with the workspace and the output buffers kept
between calls as an engine keeps them.  Shapes are those of the repository's
workloads: LLaVA-1.5 (MHA, 32 x 32 heads), Qwen2.5-VL (28 layers, 28/4 heads),
the one-layer bandwidth sweep (32/8 heads) and the fp32 8-head layer.

Inputs are seeded and synthetic: text keys in a narrow cone around a direction
per head, images as 16-token clusters of near-duplicates, video as frames that
drift slowly, values N(0, 1), window queries around the head's direction.

Which tokens are kept is a cut through a ranking of real numbers: where two
candidates on either side of the cut have scores closer than single precision
resolves, both answers are right and every row after the swap moves by one
place.  So that outputs can be compared row by row, prepare() draws a head (for
a layer-wide budget a layer) again when the 64-bit scores next to its cut are
closer than GAP relative to the score there.
"""
import math

import torch

from paper_2609_06663_gb300 import ecokv as E

GAP = 4e-5
D = 128
VNORM, CENTROID, WINSOR1, WINSOR5, MAD = 0x4, 0x8, 0x10, 0x20, 0x40


def _case(name, entry, layers, h_kv, h_q, n, window, budget, content, dtype="bf16", pool=5, flags=0):
    return dict(name=name, entry=entry, layers=layers, h_kv=h_kv, h_q=h_q, n=n, window=window, budget=budget,
                content=content, dtype=dtype, pool=pool, flags=flags)


def listed():
    return [
        # one layer of a short chat prompt, layer by layer: latency alone
        _case("layer_1k", "evict", 1, 8, 32, 1024, 4, 102, "mixed"),
        # the fp32 layer (CUDA-core passes)
        _case("layer_1k_f32", "evict", 1, 8, 8, 1024, 8, 128, "text", dtype="f32", pool=7),
        # one layer of a prompt of odd length with an image in it
        _case("layer_5003", "evict", 1, 4, 28, 5003, 8, 501, "mixed"),
        # one layer of a long video prompt
        _case("layer_32k", "evict", 1, 4, 28, 32768, 8, 3277, "video"),
        # one layer of the longest prompt, with the widest window of the sweep
        _case("layer_128k_w32", "evict", 1, 8, 32, 131072, 32, 13107, "mixed"),
        # a whole prompt at once: image and question (MHA: many short heads)
        _case("prompt_mha_2k", "evict", 32, 32, 32, 2048, 8, 205, "mixed"),
        # four images and text
        _case("prompt_gqa_8k", "evict", 28, 4, 28, 8192, 4, 1024, "mixed"),
        # a video (the benchmark's workload)
        _case("prompt_gqa_32k", "evict", 28, 4, 28, 32768, 8, 3277, "video"),
        # the layer-wide budget (AdaKV)
        _case("adaptive_8k", "adaptive", 28, 4, 28, 8192, 8, 819, "mixed"),
        # per-layer budgets (PyramidKV) over a prompt of odd length
        _case("pyramid_16411", "layered", 28, 4, 28, 16411, 8, 1641, "mixed"),
        # scores alone with a robust normalisation, as an outside selection policy reads them
        _case("score_12289_winsor", "score", 28, 4, 28, 12289, 16, 1229, "mixed", flags=WINSOR5),
        # layers offloaded to pinned host memory
        _case("host_8k", "host", 4, 4, 28, 8192, 4, 1024, "mixed"),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "prompt", "prompt", "prompt", "adaptive", "layered", "score", "f32",
                       "host"])
    h_kv, h_q = rng.choice([(8, 32), (4, 28), (32, 32), (8, 8), (8, 64), (4, 28)])
    window = rng.choice([1, 4, 8, 8, 16, 32])
    while (h_q // h_kv) * window > 256:
        window //= 2
    frac = rng.uniform(0.05, 0.2)
    content = rng.choice(["text", "mixed", "mixed", "video"])
    flags, dtype, pool, entry, layers = 0, "bf16", 5, "evict", 1
    if kind == "layer":
        n = _logu(rng, 100, 131072 if h_kv <= 8 else 32768)
        flags = rng.choice([0, 0, 0, VNORM, CENTROID])
    elif kind == "f32":
        dtype, pool, n, layers = "f32", 7, _logu(rng, 100, 8192), rng.choice([1, 2])
        h_kv, h_q = 8, 8
    else:
        layers = rng.choice([28, 32])
        entry = {"prompt": "evict"}.get(kind, kind)
        most = {"host": 16384, "score": 32768}.get(kind, 32768) * 112 // (layers * h_kv)
        if kind == "host":
            layers, most = 4, min(16384, 16384 * 4 // h_kv)
        n = _logu(rng, 512, most)
        if kind == "score":
            flags = rng.choice([0, WINSOR1, WINSOR5, MAD])
    if rng.random() < 0.5:  # half of the lengths as a server pads them
        n = max(128, n // 128 * 128) if n >= 128 else n
    window = min(window, max(1, n // 16))
    budget = max(window + 1, int(frac * n + 0.5))
    c = _case("", entry, layers, h_kv, h_q, n, window, budget, content, dtype, pool, flags)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _cone(u, m, g):
    """m keys per head around the head's direction: s (4 u + z)."""
    H = u.shape[0]
    s = torch.exp(0.5 * torch.randn(H, m, 1, generator=g, device=u.device))
    return s * (4.0 * u[:, None, :] + torch.randn(H, m, D, generator=g, device=u.device))


def _clusters(u, count, g):
    x = _cone(u, count, g).repeat_interleave(16, dim=1)
    return x + 0.1 * torch.randn(x.shape, generator=g, device=u.device)


def _keys(case, u, g):
    n, content = case["n"], case["content"]
    pre = n // 32
    if content == "video" and n >= 2560:
        frames = (n - 2 * pre) // 1280
        first = _clusters(u, 80, g)
        steps = 0.2 * torch.randn(u.shape[0], frames, 1280, D, generator=g, device=u.device)
        steps[:, 0] = first
        parts = [_cone(u, pre, g), steps.cumsum(1).flatten(1, 2)]
    elif content != "text" and n >= 64:
        parts = [_cone(u, pre, g), _clusters(u, int(0.28125 * n) // 16, g)]
    else:
        parts = []
    rest = n - sum(p.shape[1] for p in parts)
    return torch.cat(parts + [_cone(u, rest, g)], dim=1)


def _draw_layer(case, seed, layer, attempt, dev):
    """K [h_kv, n, D], Q [h_q, W, D] of one layer in the case's dtype."""
    g = torch.Generator(device=dev)
    g.manual_seed((seed * 1009 + layer) * 64 + attempt)
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    H, G = case["h_kv"], case["h_q"] // case["h_kv"]
    u = torch.randn(H, D, generator=g, device=dev)
    u = u / torch.linalg.vector_norm(u, dim=1, keepdim=True)
    K = _keys(case, u, g).to(dt)
    q = 4.0 * u[:, None, None, :] + torch.randn(H, G, case["window"], D, generator=g, device=dev)
    return K, q.reshape(H * G, case["window"], D).to(dt)


def _budgets(case):
    """Rows every head of each layer keeps."""
    if case["entry"] == "layered":
        L, B = case["layers"], case["budget"]
        last = B / 20.0  # a steep pyramid: from about twice the mean down to a twentieth of it
        first = 2.0 * B - last
        return [max(case["window"], int(first - (first - last) / max(1, L - 1) * i + 0.5)) for i in range(L)]
    return [case["budget"]] * case["layers"]


def _scores64(case, K, V, Q):
    """S [H, n - W] and lambda [H] of one layer, in 64 bits."""
    n, W, H = case["n"], case["window"], case["h_kv"]
    T, f = n - W, case["flags"]
    k = K.double()
    q = Q.double().reshape(H, -1, D)
    R = q.shape[1]
    x = torch.bmm(q, k.transpose(1, 2)) / math.sqrt(D)
    first_hidden = (n - W + 1 + torch.arange(R, device=x.device) % W)[:, None]
    x.masked_fill_(torch.arange(n, device=x.device)[None, :] >= first_hidden, -math.inf)
    raw = torch.softmax(x, dim=2).sum(1)[:, :T]
    del x
    pool = case["pool"]
    imp = torch.nn.functional.avg_pool1d(raw[:, None], pool, 1, pool // 2, count_include_pad=True)[:, 0]
    if f & VNORM:
        imp = imp * torch.linalg.vector_norm(V[:, :T].double(), dim=2)
    kbar = (k[:, :T] if f & CENTROID else k).mean(1, keepdim=True)
    dist = torch.linalg.vector_norm(k - kbar, dim=2)
    k /= torch.linalg.vector_norm(k, dim=2, keepdim=True).clamp_min(1e-12)
    mu = k.mean(1)
    cos = torch.bmm(k, mu[:, :, None])[:, :T, 0]
    r_e = 2.0 - 2.0 * torch.sigmoid(dist.mean(1) / math.sqrt(D))
    r_c = (n * (mu * mu).sum(1) - 1.0) / (n - 1.0)
    lam = _BETA * r_e + (1.0 - _BETA) * r_c
    d = dist[:, :T]
    if f & (WINSOR1 | WINSOR5):
        p, srt = (0.01 if f & WINSOR1 else 0.05), d.sort(1).values
        lo, hi = srt[:, math.floor(p * (T - 1))][:, None], srt[:, math.ceil((1 - p) * (T - 1))][:, None]
        s_e = (d.clamp(lo, hi) - lo) / (hi - lo + _EPS)
    elif f & MAD:
        def med(y):
            srt = y.sort(1).values
            return 0.5 * (srt[:, (T - 1) // 2] + srt[:, T // 2])[:, None]
        m = med(d)
        s_e = torch.sigmoid((d - m) / (med((d - m).abs()) + _EPS))
    else:
        lo, hi = d.amin(1, True), d.amax(1, True)
        s_e = (d - lo) / (hi - lo + _EPS)
    div = _ALPHA * s_e + (1.0 - _ALPHA) * (1.0 - cos) / 2.0
    lo, hi = div.amin(1, True), div.amax(1, True)
    bar = (div - lo) / (hi - lo + _EPS)
    tilde = bar * (imp.mean(1, keepdim=True) / bar.mean(1, keepdim=True))
    return lam[:, None] * tilde + (1.0 - lam[:, None]) * imp, lam


# the library's defaults as the single-precision values its parameter block holds
_ALPHA, _BETA, _EPS = (float(torch.tensor(v, dtype=torch.float32)) for v in (0.8, 0.6, 1e-6))


def _clear_cut(case, S, budget):
    """Per head (one value for a layer-wide budget): whether the scores on either side of the cut are GAP apart."""
    if case["entry"] == "score" or budget >= case["n"]:
        return torch.ones(S.shape[0], dtype=torch.bool, device=S.device)
    k = budget - case["window"]
    if case["entry"] == "adaptive":
        S, k = S.reshape(1, -1), k * S.shape[0]
    if k <= 0:
        return torch.ones(S.shape[0], dtype=torch.bool, device=S.device)
    v = S.topk(k + 1, dim=1).values
    ok = (v[:, k - 1] - v[:, k]) > GAP * v[:, k - 1].abs()
    return ok


def _inputs(case, seed):
    """K, V, Q of every layer on the GPU, with clear cuts; and S, lambda in 64 bits."""
    dev = torch.device("cuda")
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    L, H, n, G = case["layers"], case["h_kv"], case["n"], case["h_q"] // case["h_kv"]
    budgets = _budgets(case)
    K = torch.empty(L, H, n, D, dtype=dt, device=dev)
    V = torch.empty_like(K)
    Q = torch.empty(L, case["h_q"], case["window"], D, dtype=dt, device=dev)
    S = torch.empty(L, H, n - case["window"], dtype=torch.float64, device=dev)
    lam = torch.empty(L, H, dtype=torch.float64, device=dev)
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 1009 + 911)
    for l in range(L):
        V[l].copy_(torch.randn(H, n, D, generator=g, device=dev))
        K[l], Q[l] = _draw_layer(case, seed, l, 0, dev)
        S[l], lam[l] = _scores64(case, K[l], V[l], Q[l])
    for attempt in range(1, 64):
        clear = torch.stack([_clear_cut(case, S[l], budgets[l]) for l in range(L)]).cpu()
        if bool(clear.all()):
            break
        for l in range(L):
            if bool(clear[l].all()):
                continue
            k, q = _draw_layer(case, seed, l, attempt, dev)
            heads = range(H) if clear[l].numel() < H else (~clear[l]).nonzero()[:, 0].tolist()
            for h in heads:
                K[l, h], Q[l, h * G:(h + 1) * G] = k[h], q[h * G:(h + 1) * G]
            S[l], lam[l] = _scores64(case, K[l], V[l], Q[l])
    return K, V, Q, S, lam


def prepare(case, seed):
    K, V, Q, _, _ = _inputs(case, seed)
    L, H, n, d = K.shape
    host = case["entry"] == "host"
    p = E.make_params(n_layers=L, h_kv=H, h_q=case["h_q"], n=n, window=case["window"], budget=case["budget"],
                      pool_kernel=case["pool"], flags=case["flags"])
    s = {"case": case, "dtype": E.dtype_code(K)}
    if case["entry"] == "layered":
        s["budgets"] = torch.tensor(_budgets(case), dtype=torch.int32)
        p.budget = int(s["budgets"].max())
    keep = min(p.budget, n)
    dev = "cpu" if host else "cuda"

    def out(*shape, dt):
        t = torch.zeros(*shape, dtype=dt, device=dev)
        return t.pin_memory() if host else t

    if case["entry"] == "score":
        s["S"] = out(L, H, n - case["window"], dt=torch.float32)
    else:
        rows = (L, H * keep) if case["entry"] == "adaptive" else (L, H, keep)
        s["idx"] = out(*rows, dt=torch.int32)
        s["K_out"], s["V_out"] = out(*rows, d, dt=K.dtype), out(*rows, d, dt=K.dtype)
        if case["entry"] == "adaptive":
            s["head_off"] = out(L, H + 1, dt=torch.int32)
    s["lam"] = out(L, H, dt=torch.float32)
    if host:
        K, V, Q = (t.cpu().pin_memory() for t in (K, V, Q))
    s["ws"] = E.alloc_workspace_host(p, s["dtype"]) if host else E.alloc_workspace(p)
    s.update(p=p, K=K, V=V, Q=Q)
    return s


def run(s):
    p, dt, ws, stream = s["p"], s["dtype"], s["ws"], torch.cuda.current_stream()
    entry = s["case"]["entry"]
    if entry == "score":
        code = E.ecokv_score(p, dt, s["K"], s["Q"], s["S"], s["lam"], None, ws, ws.numel(), stream)
        got = {"S": s["S"], "lam": s["lam"]}
    else:
        got = {k: s[k] for k in ("idx", "head_off", "K_out", "V_out", "lam") if k in s}
        if entry == "adaptive":
            code = E.ecokv_evict_adaptive(p, dt, s["K"], s["V"], s["Q"], s["idx"], s["head_off"], s["K_out"],
                                          s["V_out"], s["lam"], ws, ws.numel(), stream)
        elif entry == "layered":
            code = E.ecokv_evict_layered(p, dt, s["K"], s["V"], s["Q"], s["budgets"], s["idx"], s["K_out"],
                                         s["V_out"], None, s["lam"], ws, ws.numel(), stream)
        elif entry == "host":
            code = E.ecokv_evict_host(p, dt, s["K"], s["V"], s["Q"], s["idx"], s["K_out"], s["V_out"], s["lam"], ws,
                                      ws.numel(), stream)
        else:
            code = E.ecokv_evict(p, dt, s["K"], s["V"], s["Q"], s["idx"], s["K_out"], s["V_out"], None, s["lam"], ws,
                                 ws.numel(), stream)
    if code != E.ECOKV_OK:
        raise E.EcokvError(code, entry)
    return got


def work(case):
    """Keys and window queries read once; kept value rows read, kept rows and
    indices written (scores instead for the score entry); value norms read
    every value row."""
    e = 4 if case["dtype"] == "f32" else 2
    units, n, W = case["layers"] * case["h_kv"], case["n"], case["window"]
    row = D * e
    total = units * n * row + case["layers"] * case["h_q"] * W * row + units * 4
    if case["entry"] == "score":
        total += units * (n - W) * 4
    else:
        kept = sum(min(b, n) for b in _budgets(case)) * case["h_kv"]
        total += 2 * kept * row + kept * 4
        total += units * n * row if case["flags"] & VNORM else kept * row
    # per key: the window logits, and the norm, the two sums and the two products with them
    return {"bytes": total, "flops": units * n * (2.0 * D * (case["h_q"] // case["h_kv"]) * W + 10.0 * D)}


def tolerance(case):
    # Four times what the outputs are from 64 bits at the start.  bf16: lambda
    # up to 8e-6 (sums of 32k keys accumulated on the tensor cores), the scores
    # 3e-6 in norm and 5e-6 at most; fp32: 5e-7 in norm, 2e-6 at most.  Kept
    # rows are copies and indices whole numbers: those are the same.
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 1e-5, "differ": 0.0}
    return {"rel": 3.5e-5, "max": 1e-4, "differ": 0.0}


def exact(case, seed):
    K, V, Q, S, lam = _inputs(case, seed)
    if case["entry"] == "score":
        return {"S": S, "lam": lam}
    n, W, H = case["n"], case["window"], case["h_kv"]
    T, keep_all = n - W, case["budget"] >= n
    budgets = _budgets(case)
    stride = min(max(budgets), n)
    idx, off, Ko, Vo = [], [], [], []
    for l, b in enumerate(budgets):
        keep = torch.zeros(H, n, dtype=torch.bool, device=K.device)
        keep[:, T:] = True
        if b >= n:
            keep[:] = True
        elif b > W and case["entry"] == "adaptive":
            top = S[l].reshape(-1).topk(H * (b - W)).indices
            keep[top // T, top % T] = True
        elif b > W:
            keep.scatter_(1, S[l].topk(b - W, dim=1).indices, True)
        h, i = keep.nonzero(as_tuple=True)
        if case["entry"] == "adaptive":
            idx.append(i.int())
            off.append(torch.cat([torch.zeros(1, device=K.device), keep.sum(1).cumsum(0)]).int())
            Ko.append(K[l, h, i].double())
            Vo.append(V[l, h, i].double())
        else:
            rows, pad = i.reshape(H, -1), stride - min(b, n)
            fill = torch.nn.functional.pad
            idx.append(fill(rows, (0, pad), value=-1).int())
            Ko.append(fill(K[l, h, i].double().reshape(H, -1, D), (0, 0, 0, pad)))
            Vo.append(fill(V[l, h, i].double().reshape(H, -1, D), (0, 0, 0, pad)))
    got = {"idx": torch.stack(idx), "K_out": torch.stack(Ko), "V_out": torch.stack(Vo), "lam": lam}
    if off:
        got["head_off"] = torch.stack(off)
    return got

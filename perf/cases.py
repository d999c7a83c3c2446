"""The work that users of the library have it do, as cases that can be timed and compared.

A serving engine compresses a prompt's KV cache once its prefill has run: all layers of the step
in one call (ckv_compress_layers, or ckv_compress_layers_lse where the prefill attention hands
over the window rows' log-sum-exp), or layer by layer as the prefill finishes them
(ckv_compress_layer, ckv_compress_layer_lse).  Analysis code reads the scores themselves
(ckv_score_windows), and the offline profiling step sums them over answer spans
(ckv_semantic_retrieval_scores).  Shapes are those of the backbone models the workloads of
ckv_synth name (32 query / 8 KV heads, 28 / 4 heads, head_dim 128), prompts of 300 to 131072
tokens, alone or packed.

A case: the call, `layers`, query and KV heads, `lens` (the prompts' lengths, comma-separated),
`window` rows, `heads` selected per KV group (or, with `scope` "layer", per layer), mean `budget`,
pooling, and whether k and v share one interleaved buffer.  The head mask and the layers' budgets
belong to the model, so they follow from the case and not from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2508_02401_gb300 as ckv

D = 128


def _case(name, call, layers, lens, *, q_heads=32, kv_heads=8, window=32, heads=2, scope="kv_head",
          budget=256, pool=7, pool_type="max", order="pool_then_sum", plant=4, outliers=True,
          pooled=False, interleaved=False):
    c = dict(call=call, layers=layers, q_heads=q_heads, kv_heads=kv_heads,
             lens=",".join(str(n) for n in lens), window=window, heads=heads, scope=scope,
             budget=budget, pool=pool, pool_type=pool_type, order=order, plant=plant,
             outliers=outliers, pooled=pooled, interleaved=interleaved)
    if name:
        c["name"] = name
    return c


def listed():
    ragged = (4981, 23417, 16301, 30725, 8209, 27004, 12873, 25018)
    return [
        # the smallest call: one layer of a short prompt, latency and launches; the pooled scores
        # are asked for as a caller that inspects its selections does
        _case("layer_2048", "compress_layer", 1, (2048,), heads=1, budget=128, outliers=False, pooled=True),
        # one layer as the prefill finishes it, an odd length, the lse at hand
        _case("layer_lse_8191", "compress_layer_lse", 1, (8191,)),
        # one layer of the longest prompt, k and v in one interleaved buffer
        _case("layer_131072", "compress_layer", 1, (131072,), budget=1024, interleaved=True),
        # a whole model, an ordinary prompt
        _case("model_8192", "compress_layers", 32, (8192,)),
        # the paper's hyper-parameters: one index set per layer from four heads, w = 8, avg pool 5
        _case("paper_8192", "compress_layers", 32, (8192,), window=8, heads=4, scope="layer", pool=5,
              pool_type="avg"),
        # a whole model, a long prompt, a large budget: the gather counts
        _case("model_32768", "compress_layers", 32, (32768,), budget=1024),
        # a batch of ragged prompts on the 28 / 4 head shape
        _case("ragged_28_4", "compress_layers", 28, ragged, q_heads=28, kv_heads=4, budget=512),
        # the longest prompt, a needle of 64 tokens, a small budget: the benchmark's workload
        _case("needle_131072", "compress_layers", 32, (131072,), budget=128, plant=64),
        # whole models with the lse at hand: a long prompt, and ragged ones
        _case("model_lse_32768", "compress_layers_lse", 32, (32768,), budget=1024),
        _case("ragged_lse_28_4", "compress_layers_lse", 8, ragged, q_heads=28, kv_heads=4, budget=512),
        # the scores themselves, every head of the group (two head batches a group), odd lengths
        _case("scores_16381", "score_windows", 8, (16381, 5003), heads=4),
        # offline head profiling: every head, eight prompts of odd length
        _case("profile_8x4093", "srs", 1, (4093,) * 8, heads=4, window=32),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    call = rng.choice(("compress_layers", "compress_layers", "compress_layers", "compress_layers_lse",
                       "compress_layers_lse", "compress_layer", "compress_layer_lse", "score_windows", "srs"))
    q_heads, kv_heads = rng.choice(((32, 8), (32, 8), (28, 4)))
    scope = "layer" if call.startswith("compress") and rng.random() < 0.2 else "kv_head"
    window = rng.choice((8, 16, 32, 32, 32, 64, rng.randint(1, 64)))
    heads = 4 if scope == "layer" else rng.choice((1, 2, 2, 3, 4))
    many = call in ("compress_layers", "compress_layers_lse", "score_windows")
    layers = rng.choice((2, 4, 8, 16, 28, 32)) if many else 1
    total = log_int(300, 131072)
    n = rng.choice((1, 1, 1, 2, 3, 5, 8))
    cuts = [rng.uniform(0.3, 1.0) for _ in range(n)]
    lens = [max(window + 1, int(total * x / sum(cuts))) for x in cuts]
    if rng.random() < 0.5:  # half of them round, as padded prompts are
        lens = [-(-x // 128) * 128 for x in lens]
    budget = max(window, log_int(64, 2048))
    pool, pool_type = rng.choice(((7, "max"), (7, "max"), (5, "avg"), (1, "max"), (13, "max"), (9, "avg")))
    c = _case(None, call, layers, lens, q_heads=q_heads, kv_heads=kv_heads, window=window, heads=heads,
              scope=scope, budget=budget, pool=pool, pool_type=pool_type,
              order=rng.choice(("pool_then_sum", "pool_then_sum", "sum_then_pool")),
              plant=rng.choice((0, 4, 64)), outliers=rng.random() < 0.8,
              pooled=call in ("compress_layer", "compress_layer_lse") and rng.random() < 0.5,
              interleaved=rng.random() < 0.3)
    # no more key reads than the largest listed case
    batches = -(-heads * _w_pad(window) // 64)
    most = 32 * 131072 * 8
    while c["layers"] > 1 and c["layers"] * sum(lens) * kv_heads * batches > most:
        c["layers"] //= 2
    return c


# ------------------------------------------------------------------ the model and the batch
def _w_pad(w):
    p = 8
    while p < w:
        p *= 2
    return p


def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def _mask(case):
    """uint8 [layers, q_heads]: `heads` of each group, or of each layer with scope "layer"."""
    r = np.random.RandomState(2508 + case["layers"] + case["q_heads"])
    m = np.zeros((case["layers"], case["q_heads"]), np.uint8)
    G = case["q_heads"] // case["kv_heads"]
    for l in range(case["layers"]):
        if case["scope"] == "layer":
            m[l, r.permutation(case["q_heads"])[:case["heads"]]] = 1
        else:
            for g in range(case["kv_heads"]):
                m[l, g * G + r.permutation(G)[:case["heads"]]] = 1
    return m


def _budgets(case):
    """int32 [layers]: budgets between a quarter of the mean (at least the window) and three times
    it, their sum the layers times the mean where the window allows; one layer has the mean."""
    n, mean = case["layers"], case["budget"]
    b = np.full(n, mean, np.int64)
    lo, hi = max(case["window"], mean // 4), 3 * mean
    r = np.random.RandomState(2401 + n)
    for _ in range(8 * n if n > 1 else 0):
        i, j, d = r.randint(n), r.randint(n), r.randint(mean + 1)
        d = min(d, b[i] - lo, hi - b[j])
        if i != j and d > 0:
            b[i] -= d
            b[j] += d
    return b.astype(np.int32)


def _config(case):
    return ckv.Config(
        num_layers=case["layers"], num_q_heads=case["q_heads"], num_kv_heads=case["kv_heads"],
        window=case["window"], pool_kernel=case["pool"],
        pool_type=ckv.POOL_MAX if case["pool_type"] == "max" else ckv.POOL_AVG,
        head_order=ckv.POOL_THEN_SUM if case["order"] == "pool_then_sum" else ckv.SUM_THEN_POOL,
        head_mask=_mask(case), budgets=_budgets(case),
        scope=ckv.SCOPE_LAYER if case["scope"] == "layer" else ckv.SCOPE_KV_HEAD)


def _inputs(case, gen, layer, mask):
    """(q_win [S, w, Hq, D], k, v [T, Hkv, D]) in bf16: N(0, 1), eight key channels of each head ten
    times as large (the outlier channels of such models), and `plant` keys of each prompt along the
    selected heads' mean window query, six times sqrt(D) long (retrieved tokens; 64: a span)."""
    lens, Hq, Hkv, w = _lens(case), case["q_heads"], case["kv_heads"], case["window"]
    G, T, S = Hq // Hkv, sum(lens), len(lens)
    rand = dict(device="cuda", generator=gen)
    q = torch.randn((S, w, Hq, D), **rand).bfloat16()
    if case["interleaved"]:
        kv = torch.empty((T, 2, Hkv, D), dtype=torch.bfloat16, device="cuda")
        k, v = kv[:, 0], kv[:, 1]
    else:
        k, v = (torch.empty((T, Hkv, D), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    x = torch.randn((T, Hkv, D), **rand)
    if case["outliers"]:
        ch = torch.rand((Hkv, D), **rand).topk(8, dim=1).indices
        x *= torch.ones((Hkv, D), device="cuda").scatter_(1, ch, 10.0)
    n, at = case["plant"], 0
    for s, L in enumerate(lens):
        P = L - w
        if n and P > n:
            if n >= 16:
                pos = torch.randint(0, P - n, (1,), **rand) + torch.arange(n, device="cuda")
            else:
                pos = torch.randperm(P, **rand)[:n]
            for g in range(Hkv):
                hs = [h for h in range(g * G, (g + 1) * G) if mask[h]] or [h for h in range(Hq) if mask[h]]
                u = q[s, :, hs].float().reshape(-1, D).mean(0)
                x[at + pos, g] = 6.0 * math.sqrt(D) * u / u.norm() + torch.randn((n, D), **rand)
        at += L
    k.copy_(x)
    v.copy_(x.normal_(generator=gen))
    return q, k, v


def _logits(case, q, k, s, g, heads, dtype):
    """[heads * w, L] logits of sequence s (heads of group g), keys a row may not see at -inf."""
    lens, w = _lens(case), case["window"]
    t0 = sum(lens[:s])
    L = lens[s]
    x = q[s][:, heads].transpose(0, 1).reshape(-1, D).to(dtype) @ k[t0:t0 + L, g].to(dtype).T
    x *= D ** -0.5
    row = torch.arange(w, device="cuda").repeat(len(heads))
    hidden = torch.arange(w, device="cuda")[None, :] > row[:, None]  # key L - w + i is seen by rows >= i
    x[:, L - w:].masked_fill_(hidden, -math.inf)
    return x


def _lse(case, q, k, dtype=torch.float32):
    """The window rows' lse [Hq, S * w], as a prefill attention returns it."""
    Hq, Hkv, w, S = case["q_heads"], case["kv_heads"], case["window"], len(_lens(case))
    G = Hq // Hkv
    out = torch.empty((Hq, S * w), dtype=dtype, device="cuda")
    for s in range(S):
        for g in range(Hkv):
            hs = list(range(g * G, (g + 1) * G))
            out[hs, s * w:(s + 1) * w] = torch.logsumexp(_logits(case, q, k, s, g, hs, dtype), 1).view(G, w)
    return out


def _generator(seed, layer):
    return torch.Generator("cuda").manual_seed(1000003 * (seed + 1) + layer)


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    cfg, mask = _config(case), _mask(case)
    call, n, lens, Hq, Hkv, w = (case["call"], case["layers"], _lens(case), case["q_heads"],
                                 case["kv_heads"], case["window"])
    S, T = len(lens), sum(lens)
    batch = ckv.Batch(np.concatenate([[0], np.cumsum(lens)]))
    strides = dict(tok_stride=2 * Hkv * D, head_stride=D) if case["interleaved"] else {}
    given_lse = call.endswith("_lse") or call == "srs"
    ios = []
    for l in range(n):
        q, k, v = _inputs(case, _generator(seed, l), l, mask[l])
        ios.append(ckv.LayerIO(layer=l, q_win=q, k=k, v=v if call.startswith("compress") else None,
                               lse=_lse(case, q, k) if given_lse else None, **strides))
    st = dict(case=case, cfg=cfg, batch=batch, ios=ios, strides=strides, out={})
    if call.startswith("compress"):
        keep = [ckv.ckv_keep_lengths(cfg, l, batch)[0] for l in range(n)]
        tk = [int(x[-1]) for x in keep]
        idx = torch.zeros(Hkv * sum(tk), dtype=torch.int32, device="cuda")
        cu = torch.zeros((n, S + 1), dtype=torch.int32, device="cuda")
        ko = torch.zeros((sum(tk), Hkv, D), dtype=torch.bfloat16, device="cuda")
        vo = torch.zeros_like(ko)
        pooled = torch.zeros((n, cfg.num_vectors, T), dtype=torch.float32, device="cuda") if case["pooled"] else None
        at = 0
        for l, io in enumerate(ios):
            io.idx = idx[Hkv * at:Hkv * (at + tk[l])].view(Hkv, tk[l])
            io.cu_keep_dev, io.k_out, io.v_out = cu[l], ko[at:at + tk[l]], vo[at:at + tk[l]]
            io.pooled_out = pooled[l] if pooled is not None else None
            at += tk[l]
        # the kept rows are copies of input rows: their bytes are what is compared
        st["out"] = dict(idx=idx, cu_keep=cu, k=ko.view(torch.int16), v=vo.view(torch.int16))
        if pooled is not None:
            st["out"]["pooled"] = pooled
    elif call == "score_windows":
        rows = [int(m.sum()) for m in mask]
        sc = torch.zeros((sum(rows), -(-T // 4) * 4), dtype=torch.float32, device="cuda")
        flat, at = sc.view(-1), 0
        for l, io in enumerate(ios):  # each layer's [n_sel, T] rows, 16-byte aligned
            io.scores = flat[at:at + rows[l] * T].view(rows[l], T)
            at += -(-rows[l] * T // 4) * 4
        st["out"] = dict(scores=sc)
    else:
        gen = _generator(seed, 777)
        a0 = torch.tensor([int(0.3 * L) for L in lens], dtype=torch.int32, device="cuda")
        end = torch.tensor(lens, dtype=torch.int32, device="cuda")
        st["span"] = torch.stack([a0, torch.minimum(a0 + 32, end)], 1).contiguous()
        st["in_answer"] = (torch.rand(S * w, device="cuda", generator=gen) < 0.5).to(torch.uint8)
        st["srs"] = torch.zeros(Hq, dtype=torch.float32, device="cuda")
        st["out"] = dict(srs=st["srs"])
    if call in ("compress_layers", "compress_layers_lse", "score_windows"):
        st["ws"] = ckv.new_layers_workspace(cfg, ios, batch)
    else:
        st["ws"] = ckv.new_workspace(cfg, 0, batch)
    return st


def run(state):
    case, cfg, batch, ios, ws = (state[x] for x in ("case", "cfg", "batch", "ios", "ws"))
    call, io = case["call"], ios[0]
    if call == "compress_layers":
        ckv.ckv_compress_layers(cfg, ios, batch, ws)
    elif call == "compress_layers_lse":
        ckv.ckv_compress_layers_lse(cfg, ios, batch, ws)
    elif call == "score_windows":
        ckv.ckv_score_windows(cfg, ios, batch, ws)
    elif call == "compress_layer":
        ckv.ckv_compress_layer(cfg, 0, batch, io.q_win, io.k, io.v, io.idx, io.cu_keep_dev, io.k_out,
                               io.v_out, ws, pooled_out=io.pooled_out, **state["strides"])
    elif call == "compress_layer_lse":
        ckv.ckv_compress_layer_lse(cfg, 0, batch, io.q_win, io.k, io.v, io.lse, io.idx, io.cu_keep_dev,
                                   io.k_out, io.v_out, ws, pooled_out=io.pooled_out, **state["strides"])
    else:  # a profiling run starts from zero and adds its prompts up
        state["srs"].zero_()
        ckv.ckv_semantic_retrieval_scores(cfg, 0, batch, io.q_win, io.k, io.lse, state["in_answer"],
                                          state["span"], state["srs"], ws, **state["strides"])
    return state["out"]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    lens, Hkv, w, n = _lens(case), case["kv_heads"], case["window"], case["layers"]
    mask, budgets = _mask(case), _budgets(case)
    G = case["q_heads"] // Hkv
    compress = case["call"].startswith("compress")
    nbytes = flops = 0
    for l in range(n):
        groups = int(sum(mask[l, g * G:(g + 1) * G].any() for g in range(Hkv)))
        n_sel, B = int(mask[l].sum()), int(budgets[l])
        for L in lens:
            if compress:  # k and v rows read and written, their positions
                nbytes += min(L, B) * Hkv * (4 * 2 * D + 4)
            if not compress or L > B:  # keys and window queries read once
                nbytes += L * groups * 2 * D + w * n_sel * 2 * D
                flops += 2 * L * n_sel * w * D
            if case["call"] == "score_windows":
                nbytes += 4 * n_sel * L
            if case["call"].endswith("_lse") or case["call"] == "srs":
                nbytes += 4 * n_sel * w
            if case["pooled"]:
                nbytes += 4 * L * (1 if case["scope"] == "layer" else Hkv)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Scores and pooled scores are sums of exponentials of fp32 logits (up to about 40 in base-2
    units, an ulp of 2e-6): measured 2e-7 to 9e-7 from 64 bits in the 2-norm; four times that.  A
    single score whose rows all carry that error is further off.  Whole values (the kept positions,
    the kept rows' bytes) differ only where two candidates' scores tie to that."""
    return {"rel": 4e-6, "max": 1e-4, "differ": 0.01}


# ------------------------------------------------------------------ 64-bit values
def _scores64(case, q, k, mask, lse=None, skip_le=0):
    """[n_sel, T] window-attention scores in 64 bits; sequences of at most skip_le tokens stay 0."""
    lens, w, Hkv = _lens(case), case["window"], case["kv_heads"]
    G = case["q_heads"] // Hkv
    sel = [h for h in range(case["q_heads"]) if mask[h]]
    out = torch.zeros((len(sel), sum(lens)), dtype=torch.float64, device="cuda")
    t0 = 0
    for s, L in enumerate(lens):
        for g in range(Hkv) if L > skip_le else ():
            hs = [h for h in sel if h // G == g]
            if hs:
                x = _logits(case, q, k, s, g, hs, torch.float64)
                if lse is None:
                    norm = torch.logsumexp(x, 1)
                else:
                    norm = lse[hs, s * w:(s + 1) * w].double().reshape(-1)
                out[[sel.index(h) for h in hs], t0:t0 + L] = (x - norm[:, None]).exp_().view(len(hs), w, L).sum(1)
        t0 += L
    return out


def _pool64(x, case):
    h = case["pool"] // 2
    if case["pool"] == 1:
        return x
    y = torch.nn.functional.pad(x, (h, h), value=-math.inf if case["pool_type"] == "max" else 0.0)
    y = y.unfold(-1, case["pool"], 1)
    return y.amax(-1) if case["pool_type"] == "max" else y.sum(-1) / case["pool"]


def _pooled64(case, scores, mask, skip_le):
    """[n_vec, T]: pooled and combined over a selection's heads; 0 at window positions and in
    sequences that are kept whole."""
    lens, w, Hkv = _lens(case), case["window"], case["kv_heads"]
    G = case["q_heads"] // Hkv
    sel = np.array([h for h in range(case["q_heads"]) if mask[h]])
    vecs = [np.arange(len(sel))] if case["scope"] == "layer" else [np.nonzero(sel // G == g)[0] for g in range(Hkv)]
    out = torch.zeros((len(vecs), sum(lens)), dtype=torch.float64, device="cuda")
    t0 = 0
    for L in lens:
        if L > skip_le:
            for i, rows in enumerate(vecs):
                x = scores[rows.tolist(), t0:t0 + L - w]
                x = _pool64(x, case).sum(0) if case["order"] == "pool_then_sum" else _pool64(x.sum(0), case)
                out[i, t0:t0 + L - w] = x
        t0 += L
    return out


def exact(case, seed):
    call, mask = case["call"], _mask(case)
    T = sum(_lens(case))
    if call == "score_windows":
        rows = [int(m.sum()) for m in mask]
        out = torch.zeros((sum(rows), -(-T // 4) * 4), dtype=torch.float64, device="cuda")
        flat, at = out.view(-1), 0
        for l in range(case["layers"]):
            q, k, _ = _inputs(case, _generator(seed, l), l, mask[l])
            flat[at:at + rows[l] * T] = _scores64(case, q, k, mask[l]).view(-1)
            at += -(-rows[l] * T // 4) * 4
        return dict(scores=out)
    if call.startswith("compress"):
        if not case["pooled"]:
            return None  # positions and copied rows: nothing is computed in floating point
        q, k, _ = _inputs(case, _generator(seed, 0), 0, mask[0])
        lse = _lse(case, q, k) if call.endswith("_lse") else None
        B = int(_budgets(case)[0])
        pooled = _pooled64(case, _scores64(case, q, k, mask[0], lse, B), mask[0], B)
        return dict(idx=None, cu_keep=None, k=None, v=None, pooled=pooled[None])
    state = prepare(case, seed)
    io, w = state["ios"][0], case["window"]
    out = torch.zeros(case["q_heads"], dtype=torch.float64, device="cuda")
    G = case["q_heads"] // case["kv_heads"]
    for s, L in enumerate(_lens(case)):
        a0, a1 = state["span"][s].tolist()
        steps = state["in_answer"][s * w:(s + 1) * w].double()
        for g in range(case["kv_heads"]):
            hs = [h for h in range(g * G, (g + 1) * G) if mask[0][h]]
            x = _logits(case, io.q_win, io.k, s, g, hs, torch.float64).view(len(hs), w, L)
            p = (x - io.lse[hs, s * w:(s + 1) * w].double()[:, :, None]).exp_()
            out[hs] += (p[:, :, a0:a1].sum(2) * steps).sum(1)
    return dict(srs=out)

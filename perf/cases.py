"""The measured work of this library: prefill KV-cache compression calls.

A case is one call of a public entry point (paper_2605_31105_gb300.binding, the
names of include/grkv.h) on caches of a stated shape.  `kind` names the call:

  compress  grkv_compress, what an engine calls after a layer's (or a batch of
            layers') prefill; key=True adds the key step (GRKV_UPDATE_K)
  ragged    grkv_compress_ragged with budgets that fall from layer to layer
            (a pyramid allocation: `heads` units per layer share a budget)
  score     grkv_score alone (window scores, target, row statistics)
  select    grkv_select alone (pooled top-B of given scores)
  merge     grkv_merge alone (the ridge value merge of a given retained set)

The decode-side transfer check is a diagnostic off the serving path and the
portable kernels under GRKV_FORCE_SIMT are for comparison: neither is measured.

Sizes: units U = batch x layers x KV heads, g query heads per KV head, w window
queries per head, n cached tokens, B retained tokens, head size 128.  Keys,
values and queries are drawn as in grkv_inputs (low-rank keys, the same with
outlier channels, or with spans near a topic the queries follow), on the GPU.
"""
import math

import torch

from paper_2605_31105_gb300 import binding as b

D = 128

_DEFAULTS = dict(kind="compress", dtype="bf16", recipe="lowrank", units=8, group=4, window=32,
                 n=8192, budget=512, budget_last=0, heads=8, lambda_v=1e-2, lambda_k=1e-2,
                 pool=7, pool_type="max", causal=True, key=False, deterministic=False)


def _case(**kw):
    return dict(_DEFAULTS, **kw)


def listed():
    return [
        # One KV head of a small fp32 model: the smallest call, launch latency.
        _case(name="compress_head_f32_2k", dtype="f32", units=1, group=1, n=2048, budget=256),
        # One layer with an fp32 cache (8 KV heads, 4 query heads each).
        _case(name="compress_layer_f32_8k", dtype="f32"),
        # A layer of an odd model after a short prompt: nothing is a multiple of a tile.
        _case(name="compress_layer_odd_5k", units=6, group=7, window=16, n=5003, budget=389,
              pool=5, lambda_v=1e-1),
        # One layer of an 8B-sized model, the call an engine makes per layer.
        _case(name="compress_layer_8k"),
        # The same layer for a batch of four prompts.
        _case(name="compress_batch4_16k", units=32, n=16384, recipe="outlier"),
        # A whole 32-layer cache at 32K in one call: the benchmark's workload.
        _case(name="compress_cache_32k", units=256, n=32768, budget=2048, recipe="outlier"),
        # Four layers with a 64-query window at 128K: 256 stacked window rows.
        _case(name="compress_spans_128k", units=32, window=64, n=131072, budget=1024,
              recipe="spans", lambda_v=1e-1),
        # Eight layers with a pyramid of budgets, 8 KV heads each.
        _case(name="ragged_pyramid_16k", kind="ragged", units=64, n=16384, budget=1536,
              budget_last=200, recipe="outlier"),
        # One layer with the key step on: value step, then conjugate gradients.
        _case(name="compress_key_layer_8k", key=True),
        # The scores of a whole 32-layer 128K cache with a 64-query window: the largest call.
        _case(name="score_cache_128k", kind="score", units=256, window=64, n=131072,
              budget=1024, recipe="spans"),
        # Selection over a whole cache's scores, as a caller with its own scores runs it.
        _case(name="select_cache_32k", kind="select", units=256, n=32768, budget=2048),
        # The value merge of a whole cache for a retained set the caller chose.
        _case(name="merge_cache_32k", kind="merge", units=256, n=32768, budget=2048,
              recipe="outlier"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the range's logarithm, capped so that no case does more
    work than the listed one of its kind."""
    kind = rng.choices(["compress", "f32", "key", "ragged", "score", "select", "merge"],
                       [35, 10, 10, 10, 10, 10, 15])[0]
    f32 = kind == "f32"
    window = rng.choice([8, 16, 32, 32, 64])
    most = (128 if kind in ("f32", "key") else 256) // window
    group = rng.choice([g for g in (1, 2, 4, 7, 8) if g <= most])
    blocks = 1 + (group * window - 1) // 128
    n = _log_int(rng, 512, {"f32": 8192, "key": 16384}.get(kind, 131072))
    budget = min(_log_int(rng, window + 32, {"f32": 512, "key": 512}.get(kind, 4096)), n // 2)
    units = _log_int(rng, 1, {"f32": 32, "key": 16}.get(kind, 256))
    # the listed cases' work: tokens scored (per block of 128 window rows), rows merged
    if f32 or kind == "key":
        units = min(units, 8 * 8192 // n, 8 * 512 // budget)
    else:
        units = min(units, 256 * 32768 // (n * blocks), 256 * 2048 // (budget * blocks))
    units = max(1, units)
    c = _case(kind="compress" if kind in ("f32", "key") else kind, dtype="f32" if f32 else "bf16",
              key=kind == "key", units=units, group=group, window=window, n=n, budget=budget,
              recipe=rng.choice(["lowrank", "outlier", "spans"]) if kind != "key" else "lowrank",
              lambda_v=rng.choice([1e-2, 1e-1]), pool=rng.choice([5, 7, 13]),
              pool_type=rng.choice(["max"] * 5 + ["avg"]), causal=rng.random() < 0.85,
              deterministic=kind in ("compress", "score") and rng.random() < 0.2)
    if kind == "ragged":
        c["heads"] = rng.choice([2, 4, 8])
        c["units"] = max(1, units // c["heads"]) * c["heads"]
        c["budget_last"] = max(window + 16, budget // 8)
        c["budget"] = max(c["budget"], c["budget_last"])
    return c


# ------------------------------------------------------------------ inputs --
def _budgets(c):
    """Ragged: one budget per unit, falling linearly from the first layer to the last."""
    if c["kind"] != "ragged":
        return [c["budget"]] * c["units"]
    layers = c["units"] // c["heads"]
    out = []
    for layer in range(layers):
        f = layer / max(1, layers - 1)
        out += [int(round(c["budget"] + f * (c["budget_last"] - c["budget"])))] * c["heads"]
    return out


def _inputs(c, seed):
    """q [U][g][w][d], k and v [U][n][d] in the case's dtype, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    U, n, w, g = c["units"], c["n"], c["window"], c["group"]
    q = torch.empty((U, g, w, D), dtype=dt, device="cuda")
    k = torch.empty((U, n, D), dtype=dt, device="cuda")
    v = torch.empty((U, n, D), dtype=dt, device="cuda")

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    step = max(1, (1 << 22) // n)   # 2 GB of fp32 keys at a time
    for u0 in range(0, U, step):
        u1 = min(U, u0 + step)
        s = u1 - u0
        kk = torch.bmm(randn(s, n, 16), randn(s, 16, D)).mul_(0.25)
        kk.add_(randn(s, n, D), alpha=0.1)
        topic = None
        if c["recipe"] == "outlier":
            ch = torch.rand((s, D), generator=gen, device="cuda").argsort(dim=1)[:, :4]
            kk *= torch.ones((s, D), device="cuda").scatter_(1, ch, 10.0)[:, None, :]
        elif c["recipe"] == "spans":
            topic = torch.nn.functional.normalize(randn(s, D), dim=1)
            span, count = 256, 16
            room = n - w - span * count
            if room > count:
                # starts of 16 spans of 256 tokens that do not overlap
                free = torch.rand((s, room), generator=gen, device="cuda").argsort(dim=1)[:, :count]
                starts = free.sort(dim=1).values + torch.arange(count, device="cuda") * span
                pos = (starts[:, :, None] + torch.arange(span, device="cuda")).reshape(s, -1, 1)
                pos = pos.expand(-1, -1, D)
                blk = kk.gather(1, pos)
                orth = blk - (blk @ topic[:, :, None]) * topic[:, None, :]
                orth = torch.nn.functional.normalize(orth, dim=2)
                kk.scatter_(1, pos, blk.norm(dim=2, keepdim=True)
                            * (0.8 * topic[:, None, :] + 0.6 * orth))
        k[u0:u1] = kk
        v[u0:u1] = randn(s, n, D)
        noise = 0.5 * randn(s, g, w, D)
        if topic is not None:
            q[u0:u1] = 2.0 * math.sqrt(D) * topic[:, None, None, :] + noise
        else:
            rows = torch.randint(0, n, (s, g * w, 1), generator=gen, device="cuda")
            near = k[u0:u1].gather(1, rows.expand(-1, -1, D)).float()
            q[u0:u1] = 2.0 * near.reshape(s, g, w, D) + noise
    return q, k, v


def _scale():
    return float(torch.tensor(1.0 / math.sqrt(D), dtype=torch.float32))


def _visible(c, pos):
    """[m][len(pos)]: whether stacked window row r = h*w + a sees key position pos[j]."""
    m = c["group"] * c["window"]
    if not c["causal"]:
        return torch.ones((m, pos.numel()), dtype=torch.bool, device=pos.device)
    a = torch.arange(m, device=pos.device) % c["window"]
    return pos[None, :] <= (c["n"] - c["window"] + a)[:, None]


def _attention(c, q, k, pos, dt):
    """Softmax attention of one unit's stacked window rows over keys k at positions pos,
    with its row maximum and normaliser."""
    s = (q.reshape(-1, D).to(dt) @ k.to(dt).T).mul_(_scale())
    w = c["window"]
    s[:, -w:].masked_fill_(~_visible(c, pos[-w:]), -math.inf)   # the window comes last
    top = s.amax(dim=1, keepdim=True)
    s.sub_(top).exp_()
    total = s.sum(dim=1, keepdim=True)
    return s.div_(total), top, total


def _pool(c, scores):
    """Pooled fp32 prefix scores of one unit."""
    h = c["pool"] // 2
    if c["pool_type"] == "max":
        return torch.nn.functional.max_pool1d(scores[None, None], c["pool"], 1, h)[0, 0]
    x = torch.nn.functional.pad(scores.double(), (h, h)).unfold(0, c["pool"], 1)
    acc = torch.zeros_like(scores, dtype=torch.float64)
    for t in range(c["pool"]):
        acc = acc + x[:, t]
    return (acc / c["pool"]).float()


def _select(c, scores, budget):
    """Retained positions of one unit: best pooled prefix scores (ties: first), window."""
    P = c["n"] - c["window"]
    best = torch.sort(_pool(c, scores), descending=True, stable=True).indices
    keep = best[: budget - c["window"]].sort().values
    return torch.cat([keep, torch.arange(P, c["n"], device=keep.device)])


def _params(c):
    flags = (b.GRKV_UPDATE_K if c["key"] else 0) | \
        (b.GRKV_DETERMINISTIC if c["deterministic"] else 0)
    return b.params(c["units"], c["group"], c["n"], c["window"], c["budget"], dtype=c["dtype"],
                    pool_kernel=c["pool"], pool_type=c["pool_type"], lambda_v=c["lambda_v"],
                    lambda_k=c["lambda_k"], causal=int(c["causal"]), flags=flags)


def _select_scores(c, seed):
    """Scores of a selection-only call: attention mass, a few orders of magnitude wide."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn((c["units"], c["n"] - c["window"]), generator=gen, device="cuda")
    return torch.exp(x.mul_(2.5))


def _merge_inputs(c, seed, q, k, v):
    """What a caller of grkv_merge holds: scores, target, row statistics, retained set."""
    U, n, w, m = c["units"], c["n"], c["window"], c["group"] * c["window"]
    pos = torch.arange(n, device="cuda")
    scores = torch.empty((U, n - w), device="cuda")
    y = torch.empty((U, m, D), device="cuda")
    stats = torch.empty((U, m, 2), device="cuda")
    idx = torch.empty((U, c["budget"]), dtype=torch.int32, device="cuda")
    for u in range(U):
        a, top, total = _attention(c, q[u], k[u], pos, torch.float32)
        scores[u] = a[:, : n - w].sum(dim=0)
        y[u] = a @ v[u].float()
        stats[u, :, 0:1] = top
        stats[u, :, 1:2] = total
        idx[u] = _select(c, scores[u], c["budget"]).int()
    return scores, y, stats, idx


def prepare(case, seed):
    c, st = case, {}
    kind, U, n, w, m = c["kind"], c["units"], c["n"], c["window"], c["group"] * c["window"]
    st["kind"], st["p"] = kind, _params(c)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    if kind == "ragged":
        st["budgets"] = _budgets(c)
        size = b.grkv_compress_ragged_workspace_size(st["p"], st["budgets"])
    else:
        size = b.grkv_workspace_size(st["p"])
    st["ws"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    if kind == "select":
        st["scores"] = _select_scores(c, seed)
    else:
        st["q"], st["k"], st["v"] = _inputs(c, seed)
    if kind == "merge":
        st["scores"], st["y"], st["stats"], st["idx"] = \
            _merge_inputs(c, seed, st["q"], st["k"], st["v"])
    if kind == "score":
        st["scores"] = torch.empty((U, n - w), device="cuda")
        st["y"] = torch.empty((U, m, D), device="cuda")
        st["stats"] = torch.empty((U, m, 2), device="cuda")
    if kind in ("compress", "select"):
        st["idx"] = torch.empty((U, c["budget"]), dtype=torch.int32, device="cuda")
    if kind in ("compress", "merge"):
        st["k_out"] = torch.empty((U, c["budget"], D), dtype=dt, device="cuda")
        st["v_out"] = torch.empty_like(st["k_out"])
    if kind == "ragged":
        rows = sum(st["budgets"])
        st["idx"] = torch.empty((rows,), dtype=torch.int32, device="cuda")
        st["k_out"] = torch.empty((rows, D), dtype=dt, device="cuda")
        st["v_out"] = torch.empty_like(st["k_out"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "compress":
        b.grkv_compress(st["p"], st["q"], st["k"], st["v"], st["k_out"], st["v_out"], st["idx"],
                        st["ws"])
    elif kind == "ragged":
        b.grkv_compress_ragged(st["p"], st["budgets"], st["q"], st["k"], st["v"], st["k_out"],
                               st["v_out"], st["idx"], st["ws"])
    elif kind == "score":
        b.grkv_score(st["p"], st["q"], st["k"], st["v"], st["scores"], st["y"], st["stats"],
                     st["ws"])
        return {"scores": st["scores"], "y": st["y"], "row_stats": st["stats"]}
    elif kind == "select":
        b.grkv_select(st["p"], st["scores"], st["idx"], st["ws"])
        return {"idx": st["idx"]}
    else:
        b.grkv_merge(st["p"], st["q"], st["k"], st["v"], st["scores"], st["y"], st["idx"],
                     st["k_out"], st["v_out"], st["ws"], row_stats=st["stats"])
        return {"k_out": st["k_out"], "v_out": st["v_out"]}
    return {"idx": st["idx"], "k_out": st["k_out"], "v_out": st["v_out"]}


# ------------------------------------------------------------------- floor --
# Conjugate-gradient iterations that 64-bit arithmetic needs for the listed key-step case
# (low-rank keys, lambda_k = 1e-2, residual 1e-4).
_CG_ITERATIONS = 340


def work(case):
    c = case
    U, n, w, m = c["units"], c["n"], c["window"], c["group"] * c["window"]
    el = 4 if c["dtype"] == "f32" else 2
    rows = sum(_budgets(c))
    kind = c["kind"]
    by = fl = 0
    if kind in ("compress", "ragged", "score"):
        by += U * (m + 2 * n) * D * el           # queries, keys, values
        fl += U * 4 * m * n * D                  # logits and target
    if kind == "score":
        by += U * (n - w + m * D + 2 * m) * 4
    if kind == "select":
        by += U * (n - w) * 4
        fl += U * (n - w) * (c["pool"] - 1)
    if kind in ("compress", "ragged", "select"):
        by += rows * 4                           # retained positions
    if kind == "merge":
        by += U * (m * D * el + (m * D + 2 * m) * 4) + rows * (2 * D * el + 8)
    if kind in ("compress", "ragged", "merge"):
        by += rows * 2 * D * el
        # retained logits, their products with V0 and themselves, the solve, the update
        fl += rows * (6 * m * D + m * m) + U * (m ** 3 // 3 + 2 * m * m * D)
    if c["key"]:
        fl += _CG_ITERATIONS * rows * (4 * m * D + 2 * m * m)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """About four times what one GB300 showed against `exact` (worst 2-norm errors: merged
    values 1.4e-6 in fp32 and 1.8e-3 in bf16, target 1.7e-3 with probabilities held in bf16,
    keys of the key step 1.7e-3).  A bf16 value next to a rounding edge moves by an ulp
    (2^-7 of it), and the key step stops its iterations at a residual of 1e-4."""
    if case["kind"] == "select":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 4e-4}
    return {"rel": 7e-3, "max": 5e-2 if case["key"] else 3e-2}


# ------------------------------------------------------------ 64-bit values --
def _fixed(c, pos, scores, budget):
    """Retained slots that keep their values: sinks, window, the best floor(beta B) others."""
    P = c["n"] - c["window"]
    fixed = (pos < 4) | (pos >= P)
    cand = torch.nonzero(~fixed)[:, 0]
    top = min(int(math.floor(_f32(0.10) * budget)), cand.numel())
    if top:
        order = torch.sort(scores[pos[cand]], descending=True, stable=True).indices
        fixed[cand[order[:top]]] = True
    return fixed


def _f32(x):
    return float(torch.tensor(x, dtype=torch.float32))


def _merge_exact(c, q, k, v, scores, y, pos, budget):
    """The value step (and the key step) of one unit in 64 bits."""
    k0, v0 = k[pos].double(), v[pos].double()
    free = ~_fixed(c, pos, scores, budget)
    x, _, _ = _attention(c, q, k0, pos, torch.float64)
    xg = x * free
    gram = xg @ xg.T + _f32(c["lambda_v"]) * torch.eye(x.shape[0], dtype=x.dtype, device=x.device)
    z = torch.cholesky_solve(y - x @ v0, torch.linalg.cholesky(gram))
    vs = v0 + xg.T @ z
    if not c["key"]:
        return k0, vs
    # the key step linearises at K0 with the merged values as the call writes them
    vw = vs.to(v.dtype).double()
    qd, s = q.reshape(-1, D).double(), _scale()
    e = y - x @ vw

    def jt(a):
        da = a @ vw.T
        ds = x * (da - (x * da).sum(dim=1, keepdim=True))
        return s * (ds.T @ qd) * free[:, None]

    def jj(a):
        ds = s * (qd @ jt(a).T)
        return (x * (ds - (x * ds).sum(dim=1, keepdim=True))) @ vw + _f32(c["lambda_k"]) * a

    alpha, r = torch.zeros_like(e), e.clone()
    p, rs = r.clone(), (r * r).sum()
    stop = 1e-8 * float(rs)
    for _ in range(512):
        if float(rs) <= stop:
            break
        ap = jj(p)
        t = rs / (p * ap).sum()
        alpha, r = alpha + t * p, r - t * ap
        new = (r * r).sum()
        p, rs = r + (new / rs) * p, new
    return k0 + jt(alpha), vs


def exact(case, seed):
    c = case
    kind, U, n, w = c["kind"], c["units"], c["n"], c["window"]
    if kind == "select":
        scores = _select_scores(c, seed)
        return {"idx": torch.stack([_select(c, scores[u], c["budget"]) for u in range(U)])}
    q, k, v = _inputs(c, seed)
    pos = torch.arange(n, device="cuda")
    if kind == "merge":
        scores, y, _, idx = _merge_inputs(c, seed, q, k, v)
        out = [_merge_exact(c, q[u], k[u], v[u], scores[u], y[u].double(), idx[u].long(),
                            c["budget"]) for u in range(U)]
        return {"k_out": torch.stack([o[0] for o in out]),
                "v_out": torch.stack([o[1] for o in out])}
    got = []
    for u, budget in enumerate(_budgets(c)):
        a, top, total = _attention(c, q[u], k[u], pos, torch.float64)
        scores, y = a[:, : n - w].sum(dim=0), a @ v[u].double()
        del a
        if kind == "score":
            got.append((scores, y, torch.cat([top, total], dim=1)))
            continue
        scores = scores.float()   # decisions that turn scores into positions are 32-bit ones
        idx = _select(c, scores, budget)
        got.append((idx, *_merge_exact(c, q[u], k[u], v[u], scores, y, idx, budget)))
    names = ("scores", "y", "row_stats") if kind == "score" else ("idx", "k_out", "v_out")
    join = torch.cat if kind == "ragged" else torch.stack
    return {name: join([t[i] for t in got]) for i, name in enumerate(names)}

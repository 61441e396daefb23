"""The work a user of the library has it do, as measurable cases.

Two halves, as in the paper: Alg. 1 compresses a prefilled KV cache (kinds
``build``), Alg. 2 decodes from the compressed cache (every other kind).  The
shapes are those of ``workloads.WORKLOADS`` (LLaMA-3.1-8B attention: 8 KV heads,
4 query heads each, head_dim 128) at their contexts, budgets and batches.

kind    one pass
layer   one eager reskv_decode_attn call for one layer
step    one decode token: one reskv_decode_attn per layer, all layers in a CUDA
        graph (a layer's queries need the layer before)
grow    the same with reskv_append of the token's keys and values before each
        layer's decode, its ring of appended tokens full (long generation)
stage   every layer in one launch (layer = -1)
host    every layer with queries and outputs in pinned host memory
noalloc one layer from the caller's own device arrays, nothing allocated
build   reskv_build_cache of the prefilled layers, then the first decode

Inputs follow the recipe of ``workloads.py`` (peaked queries 0.7 k + 0.3 n,
outlier channels, drift and needles for the 128K context), from torch's
generator so that every seed is another draw.
"""
import math

import numpy as np
import torch

from paper_2607_29591_gb300 import reskv as R

D = 128
RATIOS = (0.0, 0.05, 0.10, 0.15, 0.20)        # the paper's residual ratios (reskv_config_default)
RECENT = 64
OUTLIER = 8.0


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _decode(kind, layers, batch, heads, group, seq, budget, **more):
    return dict(kind=kind, layers=layers, batch=batch, heads=heads, group=group, seq=seq,
                budget=budget, residual=more.get("residual", "grid"), ragged=more.get("ragged", False),
                append=more.get("append", 0), softmax=more.get("softmax", "shared"))


def _build(layers, batch, heads, group, seq, budget, **more):
    return dict(kind="build", layers=layers, batch=batch, heads=heads, group=group, seq=seq,
                budget=budget, obs=more.get("obs", 128), score=more.get("score", "obs"),
                residual=more.get("residual", "proxy"), budgets=more.get("budgets", "uniform"),
                content=more.get("content", "plain"), export=more.get("export", False))


def listed():
    def named(name, case):
        return dict(case, name=name)

    return [
        # the smallest call: one KV head of one layer, as a unit test or a probe makes it
        named("layer_tiny", _decode("layer", 1, 1, 1, 4, 4096, 256, residual="fixed:32")),
        # one user's decode token: 8 short units a layer, launch and latency bound
        named("step_32k_b1", _decode("step", 32, 1, 8, 4, 32768, 512)),
        # the benchmark's decode token: batch 8, 1 GiB of cache a step
        named("step_32k_b8", _decode("step", 32, 8, 8, 4, 32768, 1024)),
        # serving many users with a small cache: 512 short, unequal units a layer
        named("step_16k_b64", _decode("step", 32, 64, 8, 4, 16384, 128, residual="drawn")),
        # long generation: every token is appended, the oldest joins a residual entry
        named("grow_32k_b8", _decode("grow", 32, 8, 8, 4, 32768, 1024, append=64)),
        # long context, all layers at once (a bandwidth ceiling; speculative or replayed queries)
        named("stage_128k_b4", _decode("stage", 32, 4, 8, 4, 131072, 2048)),
        # a CPU-resident model around the attention: queries and outputs cross the host link
        named("host_32k_b8", _decode("host", 32, 8, 8, 4, 32768, 1024)),
        # the smallest compression: one unit, fixed residual count
        named("build_tiny", _build(1, 1, 1, 4, 4096, 256, residual="fixed:32", export=True)),
        # one user's prompt, a layer compressed as soon as it is prefilled, AdaKV budgets
        named("build_32k_b1", _build(1, 1, 8, 4, 32768, 512, budgets="adakv", export=True)),
        # the benchmark's compression, two of its layers: validation proxy, short window
        named("build_32k_b8", _build(2, 8, 8, 4, 32768, 1024, obs=32)),
        # the long-context compression: drifting keys, needles, the largest budget
        named("build_128k_b4", _build(1, 4, 8, 4, 131072, 2048, content="drift")),
        # many users, query-free scores, residual counts given
        named("build_16k_b64", _build(1, 64, 8, 4, 16384, 128, score="keynorm", residual="drawn")),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    group = rng.choice((4, 4, 4, 2, 1))
    if rng.random() < 0.4:
        score = rng.choice(("obs", "obs", "keynorm"))
        heads = rng.choice((8, 8, 4, 2, 3, 1))
        seq = _log_int(rng, 1024, 131072)
        units = _log_int(rng, heads, max(heads, min(512, (1 << 21) // seq)))
        budget = _log_int(rng, 96, min(2048, seq // 2))
        batch = max(1, units // heads)
        layers = max(1, min(2, (1 << 22) // (seq * batch * heads)))
        if score == "keynorm":
            return _build(layers, batch, heads, group, seq, min(budget, 512), score=score,
                          residual="drawn", export=batch * heads * budget <= 8192)
        return _build(layers, batch, heads, group, seq, budget, obs=rng.choice((32, 64, 128)),
                      budgets=rng.choice(("uniform", "uniform", "adakv")),
                      content=rng.choice(("plain", "plain", "drift")),
                      export=batch * heads * budget <= 8192)
    kind = rng.choice(("layer", "step", "step", "grow", "stage", "host", "noalloc"))
    budget = _log_int(rng, 96, 2048)
    heads = rng.choice((8, 8, 4, 2, 3, 1))
    batch = _log_int(rng, 1, 64)
    layers = 1 if kind in ("layer", "noalloc") else rng.choice((4, 8, 16, 32))
    while layers * batch * heads * budget > (1 << 21):
        batch = max(1, batch // 2)
        layers = max(1, layers // 2) if batch == 1 else layers
    return _decode(kind, layers, batch, heads, group, 16 * budget, budget,
                   residual=rng.choice(("grid", "grid", "drawn")),
                   ragged=kind != "noalloc" and rng.random() < 0.25,
                   append=rng.choice((8, 33, 64)) if kind == "grow" else 0,
                   softmax="separate" if kind != "noalloc" and rng.random() < 0.15 else "shared")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed, tag):
    return torch.Generator(device="cuda").manual_seed(1000003 * (int(seed) % (1 << 40)) + tag)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _outlier_scale(g, n):
    """[n, D]: four channels c, c + 32, c + 64, c + 96 scaled by 8."""
    c = torch.randint(0, D // 4, (n, 1), generator=g, device="cuda")
    sc = torch.ones(n, D, device="cuda")
    return sc.scatter_(1, c + torch.arange(0, D, D // 4, device="cuda"), OUTLIER)


def _residual_counts(case, seed, budgets):
    """r of every unit: the proxy's grid, the small-budget draw, or fixed."""
    U = len(budgets)
    rng = np.random.RandomState((seed * 7919 + 11) % (1 << 32))
    if case["residual"].startswith("fixed:"):
        r = np.full(U, int(case["residual"].split(":")[1]))
    elif case["residual"] == "drawn":            # 0..64 per (layer, head), 1/8 without residual
        H, B = case["heads"], case["batch"]
        per = rng.randint(0, 65, (case["layers"], 1, H)) * (rng.randint(0, 8, (case["layers"], 1, H)) > 0)
        r = np.broadcast_to(per, (case["layers"], B, H)).reshape(-1)
    else:
        r = np.floor(np.asarray(RATIOS)[rng.randint(0, len(RATIOS), U)] * budgets)
    return np.minimum(r, budgets - min(RECENT, int(budgets.min()) // 2)).astype(np.int32)


def _cache_inputs(case, seed):
    """A compressed cache (flat slots, unit u's at off[u]..off[u+1]) and queries."""
    U = case["layers"] * case["batch"] * case["heads"]
    rng = np.random.RandomState((seed * 104729 + 5) % (1 << 32))
    b = np.full(U, case["budget"], np.int64)
    if case["ragged"]:                           # AdaKV budgets spread about 0.8..1.3 of the mean
        b = np.floor(case["budget"] * rng.uniform(0.8, 1.3, U)).astype(np.int64)
    A = case["append"]
    off = np.concatenate([[0], np.cumsum(b + A)])
    n_res = _residual_counts(case, seed, b)
    n_main = (b - n_res).astype(np.int32)
    g = _gen(seed, 1)
    N = int(off[-1])
    unit = torch.repeat_interleave(torch.arange(U, device="cuda"), torch.from_numpy(b + A).cuda())
    j = torch.arange(N, device="cuda") - torch.from_numpy(off[:-1]).cuda()[unit]
    nm, nr = torch.from_numpy(n_main).cuda()[unit], torch.from_numpy(n_res).cuda()[unit]
    res = (j >= nm) & (j < nm + nr)
    slots = []
    for _ in range(2):                           # keys, values: entries are means, so smaller
        sc = _outlier_scale(g, U)
        x = torch.empty(N, D, dtype=torch.bfloat16, device="cuda")
        for lo in range(0, N, 1 << 19):
            hi = min(N, lo + (1 << 19))
            t = _randn(g, hi - lo, D) * sc[unit[lo:hi]]
            x[lo:hi] = torch.where(res[lo:hi, None], 0.3 * t, t).to(torch.bfloat16)
        slots.append(x)
    mean = max(1.0, (case["seq"] - case["budget"]) / max(1.0, float(n_res.mean())))
    u01 = torch.rand(N, generator=g, device="cuda").clamp_min(1e-6)
    counts = torch.where(res, 1 + torch.floor(-mean * torch.log(u01)), 0.0).to(torch.int32)
    logc = torch.where(res, torch.log(counts.clamp_min(1).float()), 0.0)
    # queries: half aim at a kept key, half at a key that was evicted
    G = case["group"]
    pick = torch.from_numpy(off[:-1] + rng.randint(0, 1 << 30, (G, U)) % n_main).cuda().reshape(-1)
    kept = (torch.rand(G * U, 1, generator=g, device="cuda") < 0.5).float()
    k = kept * slots[0][pick].float() + (1 - kept) * _randn(g, G * U, D)
    q = (0.7 * k + 0.3 * _randn(g, G * U, D)).to(torch.bfloat16)
    q = q.reshape(G, U, D).permute(1, 0, 2).reshape(case["layers"], case["batch"], case["heads"] * G, D)
    new = [(_randn(g, U, D) * _outlier_scale(g, U)).to(torch.bfloat16) for _ in range(2)] if A else None
    return dict(b=b, off=off, n_main=n_main, n_res=n_res, K=slots[0], V=slots[1], counts=counts,
                logc=logc, Q=q.contiguous(), new=new)


def _fit_obs(case):
    return (case["obs"] * 3 // 4, case["obs"] // 4)        # fit and validation rows


def _prefill(case, seed):
    """K, V, observation and decode queries of the prefilled layers."""
    L, B, H, s = case["layers"], case["batch"], case["heads"], case["seq"]
    G, n_obs = case["group"], case["obs"] if case["score"] == "obs" else 0
    g = _gen(seed, 2)
    Ks, Vs, Qo, Qd = [], [], [], []
    for _ in range(L):
        K = torch.empty(B, H, s, D, dtype=torch.bfloat16, device="cuda")
        V = torch.empty_like(K)
        qo = torch.empty(B, H * G, n_obs, D, dtype=torch.bfloat16, device="cuda")
        qd = torch.empty(B, H * G, D, dtype=torch.bfloat16, device="cuda")
        ksc, vsc = _outlier_scale(g, H), _outlier_scale(g, H)
        for b in range(B):
            k = _randn(g, H, s, D) * ksc[:, None]
            needles = max(1, s // 100)
            if case["content"] == "drift":       # slowly turning mean, 1 % needles
                ang = torch.arange(s, device="cuda", dtype=torch.float32) * (2 * math.pi / 65536)
                k += (torch.cos(ang)[None, :, None] * _randn(g, H, 1, D)
                      + torch.sin(ang)[None, :, None] * _randn(g, H, 1, D))
                step = (s - RECENT) // needles   # one in every stretch, so no two at one place
                at = torch.randint(0, step, (H, needles), generator=g, device="cuda")
                at += step * torch.arange(needles, device="cuda")
                k.scatter_(1, at[..., None].expand(-1, -1, D), 3 * _randn(g, H, needles, D))
            K[b] = k.to(torch.bfloat16)
            V[b] = (_randn(g, H, s, D) * vsc[:, None]).to(torch.bfloat16)
            pos = torch.randint(0, s, (H, G * (n_obs + 1)), generator=g, device="cuda")
            if case["content"] == "drift":       # half of the queries aim at needles
                pick = torch.randint(0, needles, pos.shape, generator=g, device="cuda")
                half = torch.rand(pos.shape, generator=g, device="cuda") < 0.5
                pos = torch.where(half, at.gather(1, pick), pos)
            kp = K[b].gather(1, pos[..., None].expand(-1, -1, D)).float()
            q = (0.7 * kp + 0.3 * _randn(g, *kp.shape)).to(torch.bfloat16).reshape(H * G, n_obs + 1, D)
            qo[b], qd[b] = q[:, :n_obs], q[:, n_obs]
        Ks.append(K)
        Vs.append(V)
        Qo.append(qo)
        Qd.append(qd)
    return Ks, Vs, (Qo if n_obs else None), torch.stack(Qd)


def _config(case, **more):
    if case.get("softmax") == "separate":
        more["softmax_mode"] = R.RESKV_SOFTMAX_SEPARATE
    return R.reskv_config_default(batch=case["batch"], n_layers=case["layers"], n_kv_heads=case["heads"],
                                  group=case["group"], seq_len=case["seq"], budget=case["budget"], **more)


def _bits(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


_warm = []


def _warm_up():
    """Loads the kernels a captured graph launches (capture cannot load them)."""
    if _warm:
        return
    for append in (0, 1):
        case = _decode("step", 1, 1, 1, 4, 1024, 64, residual="fixed:8", append=append)
        x = _cache_inputs(case, 1)
        c = _import(case, x)
        O = torch.empty(x["Q"].shape, dtype=torch.float32, device="cuda")
        if append:
            R.reskv_append(c, 0, x["new"][0], x["new"][1])
        R.reskv_decode_attn(c, 0, x["Q"], O)
        torch.cuda.synchronize()
    _warm.append(True)


def _import(case, x):
    A = case["append"]
    U = len(x["b"])
    cfg = _config(case, append_capacity=A, unit_budgets=x["b"] if case["ragged"] else None)
    return R.reskv_import_cache(cfg, x["n_main"], x["n_res"], _bits(x["K"]), _bits(x["V"]),
                                x["logc"].cpu().numpy(), counts=x["counts"].cpu().numpy(),
                                n_app=np.full(U, A, np.int32))


def _capture(launches):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        launches()
    return graph


def prepare(case, seed):
    kind = case["kind"]
    if kind == "build":
        Ks, Vs, Qo, Qd = _prefill(case, seed)
        more = {}
        if case["residual"] != "proxy":
            U = case["layers"] * case["batch"] * case["heads"]
            more["residual_override"] = _residual_counts(case, seed, np.full(U, case["budget"]))
        if case["score"] == "keynorm":
            more.update(score_mode=R.RESKV_SCORE_KEYNORM, n_obs=0, n_fit=0, n_val=0)
        else:
            n_fit, n_val = _fit_obs(case)
            more.update(n_obs=case["obs"], n_fit=n_fit, n_val=n_val)
        if case["budgets"] == "adakv":
            more["budget_mode"] = R.RESKV_BUDGET_ADAKV
        return dict(case=case, cfg=_config(case, **more), K=Ks, V=Vs, Qobs=Qo, Q=Qd,
                    O=torch.empty(Qd.shape, dtype=torch.float32, device="cuda"))
    x = _cache_inputs(case, seed)
    s = dict(case=case, Q=x["Q"], O=torch.empty(x["Q"].shape, dtype=torch.float32, device="cuda"))
    if kind == "noalloc":
        U, b = len(x["b"]), case["budget"]
        s.update(K=x["K"].reshape(U, b, D), V=x["V"].reshape(U, b, D), logc=x["logc"].reshape(U, b),
                 n_main=torch.from_numpy(x["n_main"]).cuda(), n_res=torch.from_numpy(x["n_res"]).cuda())
        return s
    cache = s["cache"] = _import(case, x)
    if kind == "host":
        s.update(Q=x["Q"].cpu().pin_memory(), O=torch.empty(x["Q"].shape, dtype=torch.float32).pin_memory())
    elif kind in ("step", "grow"):
        _warm_up()
        Q, O, L = s["Q"], s["O"], case["layers"]
        new = [t.reshape(L, -1, D) for t in x["new"]] if kind == "grow" else None
        s["new"] = new

        def launches():
            for l in range(L):
                if new:
                    R.reskv_append(cache, l, new[0][l], new[1][l])
                R.reskv_decode_attn(cache, l, Q[l], O[l])

        s["graph"] = _capture(launches)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case, Q, O = state["case"], state["Q"], state["O"]
    kind = case["kind"]
    if kind == "build":
        cache = R.reskv_build_cache(state["cfg"], state["K"], state["V"], state["Qobs"])
        R.reskv_decode_attn(cache, -1, Q, O)
        return dict(R.reskv_export_cache(cache), o=O) if case["export"] else dict(o=O)
    if kind in ("step", "grow"):
        state["graph"].replay()
    elif kind == "layer":
        R.reskv_decode_attn(state["cache"], 0, Q[0], O[0])
    elif kind == "stage":
        R.reskv_decode_attn(state["cache"], -1, Q, O)
    elif kind == "host":
        R.reskv_decode_attn_host(state["cache"], Q, O)
    else:
        R.reskv_decode_attn_noalloc(state["K"], state["V"], state["logc"], state["n_main"], state["n_res"],
                                    case["heads"], case["group"], Q, O)
    return dict(o=O)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    U = case["layers"] * case["batch"] * case["heads"]
    G, b, s = case["group"], case["budget"], case["seq"]
    slots = U * (b + case.get("append", 0))
    qo = U * G * D * (2 + 4)
    decode = 4 * slots * G * D                   # q.k and p.v of every slot and query head
    if case["kind"] != "build":
        more = 2 * U * 2 * D * 2 if case["kind"] == "grow" else 0      # the new row in, and into its slot
        return dict(bytes=slots * 4 * D + slots * 4 * 0.1 + qo + more, flops=decode)
    keys_only = case["score"] == "keynorm" and case["residual"] == "fixed:0"
    flops = decode
    fit, val = _fit_obs(case) if case["score"] == "obs" else (0, 0)
    flops += U * s * D * (2 * G * fit if fit else 2)                   # scores
    iters, evicted = 4, max(0, s - b)
    if case["residual"] == "proxy":
        rs = [int(x * b) for x in RATIOS if int(x * b) > 0]
        flops += U * G * val * 4 * D * (s + b * (1 + len(rs)))         # targets and losses
    else:
        rs = [32]                                                      # the drawn counts' mean
    flops += sum(2 * U * evicted * r * D * iters for r in rs)          # nearest centres
    return dict(bytes=U * s * D * 2 * (1 if keys_only else 2) + 2 * slots * 4 * D + qo
                + U * G * (fit + val) * D * 2, flops=flops)


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _attend(q, K, V, logc, main, res, separate):
    """Alg. 2 for one unit: q [G, D], slots [S, D] in float64, masks over slots."""
    a = q @ K.T / math.sqrt(D)
    am, ar = a[:, main], a[:, res] + logc[res]
    m = am.max(1, keepdim=True).values
    if ar.shape[1]:
        m = torch.maximum(m, ar.max(1, keepdim=True).values)
    wm, wr = torch.exp(am - m), torch.exp(ar - m)
    dm, dr = wm.sum(1, keepdim=True), wr.sum(1, keepdim=True)
    p_max = (am.max(1, keepdim=True).values - torch.logsumexp(am, 1, keepdim=True)).exp()
    g = torch.sigmoid(12.0 * (0.25 - p_max))
    nm, nr = wm @ V[main], wr @ V[res]
    if separate:
        return torch.where(dr > 0, (1 - g) * nm / dm + g * nr / dr, nm / dm)
    return (nm + g * nr) / (dm + g * dr)


def _exact_decode(case, seed):
    x = _cache_inputs(case, seed)
    G, A = case["group"], case["append"]
    q = x["Q"].double().reshape(-1, G, D)
    out = torch.empty_like(q)
    for u in range(q.shape[0]):
        lo, hi = int(x["off"][u]), int(x["off"][u + 1])
        K, V, logc = x["K"][lo:hi].double(), x["V"][lo:hi].double(), x["logc"][lo:hi].double()
        j = torch.arange(hi - lo, device="cuda")
        nm, nr = int(x["n_main"][u]), int(x["n_res"][u])
        res = (j >= nm) & (j < nm + nr)
        if A:                                    # the oldest appended token joins its nearest entry
            old = nm + nr
            if nr:
                e = nm + int((K[nm:old] - K[old]).square().sum(1).argmin())
                c = float(x["counts"][lo + e])
                for t in (K, V):
                    t[e] = ((c * t[e] + t[old]) / (c + 1)).to(torch.bfloat16).double()
                logc[e] = math.log(c + 1)
            K[old], V[old] = x["new"][0][u].double(), x["new"][1][u].double()
        out[u] = _attend(q[u], K, V, logc, ~res, res, case["softmax"] == "separate")
    return dict(o=out.reshape(x["Q"].shape))


def _entries(K, V, E, centres, iters=4):
    """Lloyd over the evicted tokens E from the given centres: entries and counts."""
    c, X = centres.clone(), K[E]
    for _ in range(iters):
        a = (c.square().sum(1) - 2 * (X @ c.T)).argmin(1)
        n = torch.bincount(a, minlength=len(c)).double()
        c = torch.where(n[:, None] > 0, torch.zeros_like(c).index_add_(0, a, X) / n.clamp_min(1)[:, None], c)
    v = torch.zeros_like(c).index_add_(0, a, V[E]) / n.clamp_min(1)[:, None]
    return c.to(torch.bfloat16).double(), v.to(torch.bfloat16).double(), n


def _scores(case, K, q):
    """Token scores of one unit; q [G, n_obs, D] or None."""
    if case["score"] == "keynorm":
        return K.square().sum(1)
    fit = q[:, :_fit_obs(case)[0]].reshape(-1, D)
    a = torch.zeros(K.shape[0], dtype=torch.float64, device="cuda")
    for rows in fit.split(64):
        a += torch.softmax(rows @ K.T / math.sqrt(D), 1).sum(0)
    a = torch.nn.functional.pad(a / case["group"], (2, 2))
    return a.unfold(0, 5, 1).sum(1) / 5


def _exact_build(case, seed):
    Ks, Vs, Qo, Qd = _prefill(case, seed)
    L, B, H, G, s, b = (case[k] for k in ("layers", "batch", "heads", "group", "seq", "budget"))
    P = min(RECENT, s)
    ovr = None
    if case["residual"] != "proxy":
        ovr = _residual_counts(case, seed, np.full(L * B * H, b)).reshape(L, B, H)
    out = torch.empty(Qd.shape, dtype=torch.float64, device="cuda")
    for l in range(L):
        for bb in range(B):
            sc = torch.stack([_scores(case, Ks[l][bb, h].double(),
                                      Qo[l][bb].reshape(H, G, -1, D)[h].double() if Qo else None)
                              for h in range(H)])[:, :s - P]
            order = torch.sort(sc, dim=1, descending=True, stable=True).indices
            budgets = [b] * H
            if case["budgets"] == "adakv":       # own safeguard, the other slots by score
                f = int(math.floor(float(np.float32(0.2)) * (b - P)))
                rest = sc.clone()
                rest.scatter_(1, order[:, :f], -1.0)
                top = torch.sort(rest.reshape(-1), descending=True, stable=True).indices[:H * (b - P - f)]
                budgets = [P + f + int(n) for n in torch.bincount(top // (s - P), minlength=H)]
            for h in range(H):
                K, V = Ks[l][bb, h].double(), Vs[l][bb, h].double()
                qd = Qd[l, bb].reshape(H, G, D)[h].double()

                def unit(r):
                    """Slots of the cache with r residual entries, and their attention."""
                    keep = budgets[h] - r - P
                    main = torch.cat([order[h, :keep], torch.arange(s - P, s, device="cuda")])
                    if r == 0:
                        kk, vv, n = K[:0], V[:0], K[:0, 0]
                    else:
                        E = torch.sort(order[h, keep:]).values
                        kk, vv, n = _entries(K, V, E, K[order[h, keep:keep + r]])
                    KK, VV = torch.cat([K[main], kk]), torch.cat([V[main], vv])
                    lc = torch.cat([torch.zeros(len(main), dtype=torch.float64, device="cuda"), torch.log(n)])
                    res = torch.arange(len(lc), device="cuda") >= len(main)
                    return lambda q: _attend(q, KK, VV, lc, ~res, res, False)

                if ovr is not None:
                    best = unit(int(ovr[l, bb, h]))
                else:
                    qv = Qo[l][bb].reshape(H, G, -1, D)[h][:, -_fit_obs(case)[1]:].double().reshape(-1, D)
                    full = torch.softmax(qv @ K.T / math.sqrt(D), 1) @ V
                    loss = lambda f: float((f(qv) - full).square().sum(1).mean())  # noqa: E731
                    rs = sorted({int(math.floor(float(np.float32(x)) * budgets[h])) for x in RATIOS} - {0})
                    plain = unit(0)
                    tried = [(loss(f), r, f) for r in rs if budgets[h] - r >= P for f in (unit(r),)]
                    at = min(tried, key=lambda t: t[:2]) if tried else (math.inf, 0, plain)
                    best = at[2] if at[0] < (1 - float(np.float32(0.01))) * loss(plain) else plain
                out[l, bb, h * G:(h + 1) * G] = best(qd)
    return dict(o=out)


def exact(case, seed):
    with torch.no_grad():
        return _exact_build(case, seed) if case["kind"] == "build" else _exact_decode(case, seed)

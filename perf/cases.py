"""The work that a program using this library has it do, as measurable cases.

Two calls carry the load of a vision-language server that prunes visual tokens:
the pass before the LLM (``provip_similarity_reduce``: critical text rows,
relevance, top-k, merge) and the step at a pruning layer inside it
(``PruneStep`` with given heads or every head, ``VisualHeadsPruneStep`` with
heads found per sample); ``ProgressiveSchedule`` chains them. Sizes follow
``synth.WORKLOADS`` (LLaVA-1.5-7B/13B, LLaVA-NeXT anyres, GQA video), the
ablation without the pre-LLM pass and the longer texts of the tests; ``draw``
spreads over the same ranges, odd and ragged sizes included.

Inputs are drawn on the GPU from the seed. Visual rows hold near-duplicates and
a heavy-tailed share of a few concepts that the text names; at the pruning
layer the keys carry a per-token salience along their group's mean query
direction, and two sink keys. So relevance and attention over the visual tokens
are heavy-tailed, as in earnest, and few samples have two tokens within
rounding of each other at the cut. Every buffer that a call leaves partly
unwritten (rows past a sample's length) is cleared once in ``prepare``.
"""
import math

import torch

from paper_2608_25332_gb300 import provip as P
from paper_2608_25332_gb300.schedule import ProgressiveSchedule

DEV = "cuda"
HEAD = 128  # head dimension of every model served
N_CONCEPTS = 6
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    return [
        # one request at fp32: the smallest call, a few short launches
        dict(name="prune_image_f32_b1", kind="prune", dtype="f32", B=1, n_sys=35, N_v=192, t_min=64, t_max=64,
             H_q=32, H_kv=32, H_sel=4, D=4096, keep=64, P=1, graph=False),
        # an ordinary image batch with ragged questions
        dict(name="prune_image_b16", kind="prune", dtype="bf16", B=16, n_sys=35, N_v=288, t_min=32, t_max=128,
             H_q=32, H_kv=32, H_sel=8, D=4096, keep=64, P=1, graph=False),
        # high-resolution images: the largest plain pruning step
        dict(name="prune_anyres_b8", kind="prune", dtype="bf16", B=8, n_sys=35, N_v=960, t_min=96, t_max=96,
             H_q=32, H_kv=32, H_sel=8, D=4096, keep=320, P=1, graph=False),
        # one video with grouped heads and three rows of position ids; a latency-bound
        # server replays the step from a CUDA graph
        dict(name="prune_video_b1", kind="prune", dtype="bf16", B=1, n_sys=35, N_v=2304, t_min=128, t_max=128,
             H_q=28, H_kv=4, H_sel=4, D=3584, keep=1024, P=3, graph=True),
        # the middle layer's form (every head) under long instructions of odd lengths
        dict(name="prune_all_heads_long_text_b4", kind="prune", dtype="bf16", B=4, n_sys=21, N_v=1003, t_min=150,
             t_max=315, H_q=28, H_kv=4, H_sel=0, D=3584, keep=334, P=3, graph=False),
        # the shallow layer's form: every head's confidence, then the best heads' scores
        dict(name="visual_heads_anyres_b8", kind="visual", dtype="bf16", B=8, n_sys=35, N_v=960, t_min=96, t_max=96,
             H_q=32, H_kv=32, H_sel=6, D=4096, keep=320, P=1, graph=False),
        # before the LLM, one fp32 image
        dict(name="reduce_image_f32_b1", kind="reduce", dtype="f32", B=1, N_v=576, t_min=64, t_max=64, D=4096,
             keep=192, layout="image", graph=False),
        # a large image batch of the wider model
        dict(name="reduce_image_b32", kind="reduce", dtype="bf16", B=32, N_v=576, t_min=64, t_max=64, D=5120,
             keep=192, layout="image", graph=False),
        # high-resolution images: the largest contraction
        dict(name="reduce_anyres_b8", kind="reduce", dtype="bf16", B=8, N_v=2880, t_min=96, t_max=96, D=4096,
             keep=960, layout="image", graph=False),
        # one video of 16 frames, replayed from a CUDA graph
        dict(name="reduce_video_b1", kind="reduce", dtype="bf16", B=1, N_v=9216, t_min=128, t_max=128, D=3584,
             keep=2304, layout="video", graph=True),
        # images under long instructions (past one 128-row block of text)
        dict(name="reduce_long_text_b4", kind="reduce", dtype="bf16", B=4, N_v=1443, t_min=140, t_max=300, D=4096,
             keep=481, layout="image", graph=False),
        # the whole progressive schedule of an image batch in one CUDA graph
        dict(name="schedule_image_b16", kind="schedule", dtype="bf16", B=16, n_sys=35, N_v=576, t_min=32, t_max=128,
             H_q=32, H_kv=32, H_sel=6, D=4096, keep=288, keep2=64, keep3=32, P=1, layout="image", graph=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: batches of 1 to 32, any visual count, text
    of 8 to 320 rows, even and ragged, within the largest listed case's work."""
    most = [work(c) for c in listed()]
    while True:
        c = _draw(rng)
        if all(work(c)[k] <= max(w[k] for w in most) for k in ("bytes", "flops")):
            return c


def _draw(rng):
    kind = rng.choice(["prune", "prune", "prune", "visual", "reduce", "reduce", "reduce", "schedule"])
    f32 = kind in ("prune", "reduce") and rng.random() < 0.2
    H_q, H_kv, D = rng.choice([(32, 32, 4096), (40, 40, 5120), (28, 4, 3584), (32, 8, 4096), (16, 2, 2048)])
    t_max = _log_int(rng, 8, 320)
    t_min = t_max if rng.random() < 0.4 else max(1, int(t_max * rng.uniform(0.25, 1.0)))
    if kind == "reduce":
        N_v = _log_int(rng, 144, 1200 if f32 else 9216)
        B = _log_int(rng, 1, max(1, min(32, (1200 if f32 else 20000) // N_v)))
        if rng.random() < 0.25:
            D += 8 * rng.randint(1, 60)  # widths that are no multiple of a K slice
        return dict(kind=kind, dtype="f32" if f32 else "bf16", B=B, N_v=N_v, t_min=t_min, t_max=t_max, D=D,
                    keep=max(1, int(N_v * rng.uniform(0.15, 0.6))), layout="image", graph=rng.random() < 0.4)
    if kind == "schedule":
        N_v = _log_int(rng, 144, 1440)
        B = _log_int(rng, 1, max(1, min(16, 9000 // N_v)))
        keep = max(8, int(N_v * rng.uniform(0.3, 0.6)))
        keep2 = max(4, int(keep * rng.uniform(0.2, 0.5)))
        return dict(kind=kind, dtype="bf16", B=B, n_sys=rng.randint(1, 60), N_v=N_v, t_min=t_min, t_max=t_max,
                    H_q=H_q, H_kv=H_kv, H_sel=6, D=D, keep=keep, keep2=keep2, keep3=max(1, keep2 // 2), P=1,
                    layout="image", graph=rng.random() < 0.5)
    N_v = _log_int(rng, 48, 400 if f32 else 2400)
    B = _log_int(rng, 1, max(1, min(32, (800 if f32 else 7000) // N_v)))
    if kind == "visual":
        H_sel = 6
    else:
        H_sel = 0 if rng.random() < 0.25 else rng.randint(1, 10)
    return dict(kind=kind, dtype="f32" if f32 else "bf16", B=B, n_sys=rng.randint(1, 60), N_v=N_v, t_min=t_min,
                t_max=t_max, H_q=H_q, H_kv=H_kv, H_sel=H_sel, D=D, keep=max(1, int(N_v * rng.uniform(0.1, 0.7))),
                P=rng.choice([1, 3]), graph=rng.random() < 0.4)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 64 + stream) % (1 << 62))
    return g


def _lengths(c, seed):
    B, lo, hi = c["B"], c["t_min"], c["t_max"]
    tl = torch.randint(lo, hi + 1, (B,), generator=_gen(seed, 0), device=DEV, dtype=torch.int32)
    tl[0] = hi  # the buffers are as long as the longest text
    return tl


def _embeddings(c, seed):
    """Visual rows [B, N_v, D] (unit variance, near-duplicates, a heavy-tailed
    share of one of a few concepts) and text rows [B, t_max, D] at the scale of
    a token embedding table, their norms spread, a quarter naming a concept."""
    B, N, D, T, dt = c["B"], c["N_v"], c["D"], c["t_max"], DTYPES[c["dtype"]]
    g = _gen(seed, 1)
    concepts = torch.nn.functional.normalize(torch.randn(N_CONCEPTS, D, generator=g, device=DEV), dim=1)
    ev = torch.empty(B, N, D, dtype=dt, device=DEV)
    et = torch.empty(B, T, D, dtype=dt, device=DEV)
    for b in range(B):
        x = torch.randn(N, D, generator=g, device=DEV)
        if c["layout"] == "video":  # consecutive frames at a cosine of about 0.9
            per = 576
            for f in range(per, N, per):
                n = min(per, N - f)
                x[f:f + n] = 0.9 * x[f - per:f - per + n] + math.sqrt(0.19) * x[f:f + n]
        else:  # 48 clusters of near-duplicates (cosine about 0.97)
            perm = torch.randperm(N, generator=g, device=DEV)
            m = min(48 * 4, N // 2)
            x[perm[m:2 * m]] = (x[perm[:m]] + 0.25 * x[perm[m:2 * m]]) / math.sqrt(1.0625)
        share = 0.5 * torch.randn(N, 1, generator=g, device=DEV).abs()
        which = torch.randint(0, N_CONCEPTS, (N,), generator=g, device=DEV)
        ev[b] = (x + share * math.sqrt(D) * concepts[which]).to(dt)
        t = 0.02 * torch.randn(T, D, generator=g, device=DEV)
        t *= torch.exp(0.25 * torch.randn(T, 1, generator=g, device=DEV))
        names = torch.rand(T, 1, generator=g, device=DEV) < 0.25
        which = torch.randint(0, N_CONCEPTS, (T,), generator=g, device=DEV)
        et[b] = (t + names * t.norm(dim=1, keepdim=True) * concepts[which]).to(dt)
    return ev, et


def _layer(c, seed, N_v):
    """Q, K, V, hidden states and position ids of a pruning layer over
    [n_sys system rows | N_v visual rows | the text], and the selected heads."""
    B, S, T, Hq, Hkv, D, dt = c["B"], c["n_sys"], c["t_max"], c["H_q"], c["H_kv"], c["D"], DTYPES[c["dtype"]]
    L = S + N_v + T
    g = _gen(seed, 2)
    u = torch.nn.functional.normalize(torch.randn(Hkv, HEAD, generator=g, device=DEV), dim=1)
    Q = torch.randn(B, L, Hq, HEAD, generator=g, device=DEV) + 4.0 * u.repeat_interleave(Hq // Hkv, 0)
    K = torch.randn(B, L, Hkv, HEAD, generator=g, device=DEV)
    # a token's salience, partly shared by the heads: a logit of about unit variance
    sal = torch.randn(B, L, 1, 1, generator=g, device=DEV) + 0.5 * torch.randn(B, L, Hkv, 1, generator=g, device=DEV)
    K += sal * (math.sqrt(HEAD) / 4.0) * u
    sink = torch.randint(0, N_v, (B,), generator=g, device=DEV) + S
    K[:, 0] = 2.0 * math.sqrt(HEAD) * u
    K[torch.arange(B, device=DEV), sink] = 2.0 * math.sqrt(HEAD) * u
    V = torch.randn(B, L, Hkv, HEAD, generator=g, device=DEV)
    hidden = torch.randn(B, L, D, generator=g, device=DEV)
    pos = torch.arange(L, dtype=torch.int32, device=DEV).expand(c["P"], B, L).contiguous()
    heads = torch.randperm(Hq, generator=g, device=DEV)[:c["H_sel"]].sort().values.tolist() if c["H_sel"] else None
    return dict(Q=Q.to(dt), K=K.to(dt), V=V.to(dt), hidden=hidden.to(dt), pos=pos, heads=heads)


def prepare(case, seed):
    c = dict(case)
    s = dict(case=c, text_len=_lengths(c, seed))
    B = c["B"]
    if c["kind"] in ("reduce", "schedule"):
        s["ev"], s["et"] = _embeddings(c, seed)
    if c["kind"] == "reduce":
        N, D, T, dt = c["N_v"], c["D"], c["t_max"], DTYPES[c["dtype"]]
        s["out"] = dict(idx=torch.empty(B, c["keep"], dtype=torch.int32, device=DEV),
                        merged=torch.empty(B, c["keep"], D, dtype=dt, device=DEV),
                        p=torch.empty(B, N, dtype=torch.float32, device=DEV),
                        mask=torch.empty(B, T, dtype=torch.uint8, device=DEV),
                        assign=torch.empty(B, N, dtype=torch.int32, device=DEV))
        s["ws"] = P.workspace(P.lib().provip_similarity_reduce_workspace_size(B, N, D, T, c["keep"]), DEV)
    else:
        N_v = c["keep"] if c["kind"] == "schedule" else c["N_v"]
        s.update(_layer(c, seed, N_v))
        s["text_start"] = torch.full((B,), c["n_sys"] + N_v, dtype=torch.int32, device=DEV)
        s["seq_len"] = s["text_start"] + s["text_len"]
    if c["kind"] == "prune":
        s["step"] = P.PruneStep(s["Q"], s["K"], s["V"], s["hidden"], s["pos"], s["heads"], c["t_max"], c["N_v"],
                                c["keep"])
        _clear(s["step"])
    elif c["kind"] == "visual":
        # the critical rows that the pre-LLM pass found: about half of the text
        s["crit"] = (torch.rand(B, c["t_max"], generator=_gen(seed, 3), device=DEV) < 0.5).to(torch.uint8)
        s["step"] = P.VisualHeadsPruneStep(s["Q"], s["K"], s["V"], s["hidden"], s["pos"], c["t_max"], c["N_v"],
                                           c["keep"], c["H_sel"])
        _clear(s["step"])
    elif c["kind"] == "schedule":
        L1 = c["n_sys"] + c["keep"] + c["t_max"]
        s["step"] = ProgressiveSchedule(B, c["N_v"], c["D"], c["t_max"], L1, c["H_q"], c["H_kv"], c["D"], c["P"],
                                        c["keep"], c["keep2"], c["keep3"], c["H_sel"], dtype=DTYPES[c["dtype"]],
                                        device=DEV)
        _clear(s["step"].shallow)
        _clear(s["step"].middle)
        g = _gen(seed, 4)
        L2 = c["n_sys"] + c["keep2"] + c["t_max"]
        s["Q2"] = (1.5 * torch.randn(B, L2, c["H_q"], HEAD, generator=g, device=DEV)).to(DTYPES[c["dtype"]])
        s["text_start2"] = torch.full((B,), c["n_sys"] + c["keep2"], dtype=torch.int32, device=DEV)
    if c["graph"]:
        # the step as a latency-bound server holds it: captured once, replayed per request
        s["result"] = _call(s)
        s["graph"] = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(s["graph"]):
            s["result"] = _call(s)
    return s


def _clear(step):
    for t in (step.hidden_out, step.K_out, step.V_out):
        t.zero_()


def _call(s):
    c = s["case"]
    if c["kind"] == "reduce":
        return P.provip_similarity_reduce(s["ev"], s["et"], s["text_len"], c["keep"], ws=s["ws"], out=s["out"])
    if c["kind"] == "prune":
        return s["step"](s["Q"], s["K"], s["V"], s["hidden"], s["pos"], s["text_start"], s["text_len"], s["seq_len"],
                         c["n_sys"])
    if c["kind"] == "visual":
        return s["step"](s["Q"], s["K"], s["V"], s["hidden"], s["pos"], s["text_start"], s["text_len"], s["seq_len"],
                         c["n_sys"], crit_mask=s["crit"])
    shallow = {k: s[k] for k in ("Q", "K", "V", "hidden", "pos", "text_start", "seq_len")}
    return s["step"](s["ev"], s["et"], s["text_len"], shallow, dict(Q=s["Q2"], text_start=s["text_start2"]),
                     c["n_sys"])


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["result"]
    return _call(state)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _layer_work(c, N_v, keep, n_heads):
    es = 4 if c["dtype"] == "f32" else 2
    T = (c["t_min"] + c["t_max"]) / 2
    L, kept = c["n_sys"] + N_v + T, c["n_sys"] + keep + T
    kv_used = min(c["H_kv"], n_heads)
    group = c["H_q"] // c["H_kv"]
    if n_heads < c["H_q"]:  # key/value heads that randomly placed heads meet
        kv_used = c["H_kv"] * (1 - (1 - 1 / c["H_kv"]) ** n_heads) if group > 1 else n_heads
    row = HEAD * es
    by = kept * (c["D"] * es + 2 * c["H_kv"] * row + 4 * c["P"])      # rows carried over: read
    by += (L - kept) * kv_used * row                                  # keys scored and dropped
    by += kept * (c["D"] * es + 2 * c["H_kv"] * row + 4 * c["P"])      # and written
    by += T * n_heads * row + 4 * N_v + 4 * keep
    return c["B"] * by, c["B"] * 2.0 * n_heads * T * (L - T / 2) * HEAD


def _reduce_work(c):
    es = 4 if c["dtype"] == "f32" else 2
    T, N, D, k = (c["t_min"] + c["t_max"]) / 2, c["N_v"], c["D"], c["keep"]
    by = (N + T + k) * D * es + 8 * N + 4 * k + T
    return c["B"] * by, c["B"] * 2.0 * D * (T * T + T * N + (N - k) * k)


def work(case):
    c = case
    if c["kind"] == "reduce":
        by, fl = _reduce_work(c)
    elif c["kind"] == "schedule":
        parts = [_reduce_work(c), _layer_work(c, c["keep"], c["keep2"], c["H_q"]),
                 _layer_work(c, c["keep2"], c["keep3"], c["H_q"])]
        by, fl = (sum(x) for x in zip(*parts))
    else:
        every = c["kind"] == "visual" or not c["H_sel"]
        by, fl = _layer_work(c, c["N_v"], c["keep"], c["H_q"] if every else c["H_sel"])
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """About four times the error measured against ``exact``: fp32 sums (scores,
    confidence, p) were within 2.5e-6 and fp32 merged rows within 2e-8; bf16
    merged rows were 1.5e-3 off, which is their rounding. A pruned row between
    two equally near kept rows may move (``differ``), which changes two merged rows."""
    if case["kind"] in ("prune", "visual") or case["dtype"] == "f32":
        return {"rel": 1e-5, "differ": 2e-3}
    return {"rel": 6e-3, "max": 0.5, "differ": 2e-3}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _scores64(Q, K, c, N_v, text_start, text_len, seq_len, heads, conf_mask=None):
    """v [B, N_v] of the given heads per sample (a list, or one list per sample)
    and, with conf_mask, the confidence [B, H_q] of every head."""
    B, dev = Q.shape[0], Q.device
    group = c["H_q"] // c["H_kv"]
    v = torch.zeros(B, N_v, dtype=torch.float64, device=dev)
    conf = torch.zeros(B, c["H_q"], dtype=torch.float64, device=dev)
    for b in range(B):
        t0, n, L = int(text_start[b]), int(text_len[b]), int(seq_len[b])
        hs = heads[b] if heads and isinstance(heads[0], (list, tuple)) else heads
        hs = range(c["H_q"]) if hs is None else hs
        causal = torch.arange(L, device=dev)[None, :] <= (t0 + torch.arange(n, device=dev))[:, None]
        for h in hs:
            s = Q[b, t0:t0 + n, h].double() @ K[b, :L, h // group].double().T / math.sqrt(HEAD)
            a = torch.softmax(s.masked_fill(~causal, -math.inf), dim=1)[:, c["n_sys"]:c["n_sys"] + N_v]
            v[b] += a.sum(0) / (len(hs) * n)
            if conf_mask is not None:
                conf[b, h] = (a.var(1, unbiased=False) * (conf_mask[b, :n] != 0)).sum()
    return v, conf


def _visual64(s, c, N_v, crit):
    _, conf = _scores64(s["Q"], s["K"], c, N_v, s["text_start"], s["text_len"], s["seq_len"], None, crit)
    heads = [sorted(conf[b].topk(c["H_sel"]).indices.tolist()) for b in range(c["B"])]
    v, _ = _scores64(s["Q"], s["K"], c, N_v, s["text_start"], s["text_len"], s["seq_len"], heads)
    return v, conf


def _reduce64(s, c):
    """(p [B, N_v], merged [B, keep, D] or None where a choice that it follows
    lies within rounding of another)."""
    B, N, D, k = c["B"], c["N_v"], c["D"], c["keep"]
    p = torch.empty(B, N, dtype=torch.float64, device=DEV)
    merged = torch.zeros(B, k, D, dtype=torch.float64, device=DEV)
    clear = True
    for b in range(B):
        t, v = s["et"][b, :int(s["text_len"][b])].double(), s["ev"][b].double()
        r = torch.softmax(t @ t.T, dim=1).mean(0)
        T = r > r.mean()
        if not bool(T.any()):
            T = torch.ones_like(T)
        clear &= bool(((r - r.mean()).abs() > 1e-5 * r.mean()).all())
        vn = torch.nn.functional.normalize(v, dim=1)
        M = torch.nn.functional.normalize(t[T], dim=1) @ vn.T
        p[b] = (M - M.mean(1, keepdim=True)).max(0).values
        top = p[b].sort(descending=True)
        clear &= k == N or bool(top.values[k - 1] - top.values[k] > 2e-6)
        idx = top.indices[:k].sort().values
        rest = torch.ones(N, dtype=torch.bool, device=DEV)
        rest[idx] = False
        to = (vn[rest] @ vn[idx].T).argmax(1)
        merged[b] = v[idx]
        merged[b].index_add_(0, to, v[rest])
        merged[b] /= (1 + torch.bincount(to, minlength=k))[:, None]
    return p, merged if clear else None


def exact(case, seed):
    c = dict(case, graph=False)
    s = prepare(c, seed)
    if c["kind"] == "reduce":
        p, merged = _reduce64(s, c)
        return dict(idx=None, merged=merged, p=p, mask=None, assign=None)
    rows = dict(hidden=None, K=None, V=None, pos=None, idx=None, seq_len=None)
    if c["kind"] == "prune":
        v, _ = _scores64(s["Q"], s["K"], c, c["N_v"], s["text_start"], s["text_len"], s["seq_len"], s["heads"])
        return dict(rows, scores=v)
    if c["kind"] == "visual":
        v, conf = _visual64(s, c, c["N_v"], s["crit"])
        return dict(rows, scores=v, vis_heads=None, conf=conf)
    p, merged = _reduce64(s, c)
    # the layers' values follow the choices before them: each is compared in the cases of its own
    return dict(pre=dict(idx=None, merged=merged, p=p, mask=None, assign=None),
                shallow=dict(rows, scores=None, vis_heads=None, conf=None), middle=dict(rows, scores=None))

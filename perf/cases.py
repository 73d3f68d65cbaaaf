"""The work that users of this library have it do, as measurable cases.

A case is one pass through the public entry points of the Python binding
(vp_decode_step, vp_decode_gather, vp_compact_kv) on caches that live on the
GPU.  The listed cases are the repository's own workloads (the tiny fp32
reference, the Qwen2.5-VL-7B-shaped decode, batched paged serving, long
reasoning, the visual-length sweep, FastV prefill compaction) and the options
that change the path: per-kv-head sets, top-p budgets with diagnostics, fp32
caches, the anchor-layer pipeline.  Inputs follow the recipe of
paper_2605_31457_gb300/workloads.py.

Fields of a case:
  kind      "step"     one vp_decode_step call per layer (anchor = -1), or the
                       anchor pipeline: layers before `anchor` attend densely,
                       `anchor` selects, later layers reuse its kept set;
            "gather"   one vp_decode_gather call over a given kept set;
            "compact"  FastV compaction of one layer's K and V caches.
  layers, batch, heads, kv_heads, head_dim, dtype ("bf16" / "fp32")
  vis, text longest visual span and text (the current token included);
            ragged = true draws every sequence's own lengths below them
  pre       prompt tokens before the visual span
  room      tokens the caches (and the context) still have room for: a context
            is made once for the longest answer, a step runs at any length
  page      page size of a paged cache, 0 for a contiguous one
  layout    "bhtd" (dense per head) or "bthd" (heads interleaved per token)
  mode, tau, r_lo, r_hi, ratio, fixed_k, gran   the budget (vp_budget)
  diag      N_act / activity bits on
  sink, beta_lo, beta_hi, scale_hi, sigma       query and key recipe
  graph     the program captured the step in a CUDA graph when it started (as
            a decode loop does) and a pass replays it
"""

import math
import random

import torch

from paper_2605_31457_gb300 import vp
from paper_2605_31457_gb300 import workloads as W

ADAPTIVE, RATIO, FIXED_K, DENSE, TOP_P = 0, 1, 2, 3, 4

BASE = dict(kind="step", layers=1, anchor=-1, batch=1, heads=28, kv_heads=4, head_dim=128, dtype="bf16", vis=1296,
            text=2561, pre=0, ragged=False, room=63, page=0, layout="bhtd", mode=ADAPTIVE, tau=0.1, r_lo=10_000,
            r_hi=50_000, ratio=0, fixed_k=0, gran=0, diag=False, sink=1.0, beta_lo=0.3, beta_hi=0.85, scale_hi=1.0,
            sigma=0.0, graph=False)


def listed():
    def case(name, **kw):
        return dict(BASE, name=name, **kw)

    return [
        # The fp32 reference configuration: the smallest call anyone makes.
        case("tiny-fp32", heads=8, kv_heads=2, head_dim=64, dtype="fp32", vis=576, text=128, room=15, sink=0.0,
             beta_lo=1.0, beta_hi=1.0),
        # A numerics check of a full-precision model: fp32 caches, a few
        # sequences of the 7B shape.
        case("fp32-batch", batch=4, dtype="fp32", vis=1296, text=1500, pre=15, ragged=True, room=100),
        # One decode step of the 7B-shaped decoder for a single user, every
        # layer its own anchor: 28 dependent calls, latency and launches.
        case("qwen7b-step", layers=28, room=255, graph=True),
        # The same step as the paper runs it (layer 17 is the anchor).
        case("qwen7b-anchor-step", layers=28, anchor=16, room=255, graph=True),
        # Batched serving over a paged cache, ragged text, one layer call.
        case("serving-paged", batch=32, vis=2304, text=4096, ragged=True, page=16, sink=1.6, beta_lo=0.6, beta_hi=1.0,
             scale_hi=1.4),
        # Long reasoning: long text, heavy-tailed key norms.
        case("long-reasoning", batch=8, vis=4096, text=16384, room=511, sigma=0.5),
        # One kept set per kv-head at the 10% setting, early in an answer: the
        # context has room for 8192 tokens, the sequences are still short.
        case("per-head-early", batch=8, vis=1023, text=700, pre=21, ragged=True, room=6469, page=16, tau=0.4,
             r_lo=50_000, r_hi=100_000, gran=1),
        # Top-p budget with the step-wise diagnostics on.
        case("top-p-diagnostics", batch=16, heads=32, kv_heads=8, vis=6400, text=1024, mode=TOP_P, ratio=100_000,
             diag=True),
        # The visual-length sweep: short spans at 5%, video-like spans at 20%
        # and 50% (the largest call).
        case("sweep-576-r5", batch=64, heads=32, kv_heads=8, vis=576, text=1024, room=15, mode=RATIO, ratio=50_000),
        case("sweep-6400-r20", batch=64, heads=32, kv_heads=8, vis=6400, text=1024, room=15, mode=RATIO,
             ratio=200_000),
        case("sweep-16384-r50", batch=64, heads=32, kv_heads=8, vis=16384, text=1024, room=15, mode=RATIO,
             ratio=500_000),
        # FastV at the prefill stage: half of the visual rows survive.
        case("fastv-compact", kind="compact", batch=8, vis=4096, text=513, pre=14, mode=RATIO, ratio=500_000),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choices(["step", "gather", "compact"], [7, 2, 1])[0]
    fp32 = kind != "gather" and rng.random() < 0.2
    heads, kv_heads, dim = rng.choice([(28, 4, 128), (28, 4, 128), (32, 8, 128), (16, 8, 128), (8, 2, 64), (12, 2, 128)])
    esz = 4 if fp32 else 2
    vis, text, batch = logu(64, 16384), logu(64, 16384), logu(1, 64)
    row = kv_heads * dim * esz * 2
    most = 4e8 if fp32 else 2.5e9  # fp32 is for checks, not for large batches
    while batch > 1 and batch * (vis + text) * row > most:
        batch -= 1
    while batch * (vis + text) * row > most:
        vis, text = vis // 2, text // 2
    c = dict(BASE, kind=kind, batch=batch, heads=heads, kv_heads=kv_heads, head_dim=dim, dtype="fp32" if fp32 else "bf16",
             vis=vis, text=text, pre=min(rng.choice([0, 14, 21, 35]), text // 4), ragged=rng.random() < 0.5,
             room=int(rng.choice([1, 15, 63, 255, 0.5 * (vis + text)])), page=rng.choice([0, 0, 16, 64]),
             layout=rng.choice(["bhtd", "bhtd", "bthd"]), gran=int(rng.random() < 0.15),
             sigma=rng.choice([0.0, 0.0, 0.5]))
    mode = rng.choices([ADAPTIVE, RATIO, FIXED_K, TOP_P], [4, 3, 1, 1])[0]
    if kind == "compact" or (mode == TOP_P and c["gran"]):
        mode = RATIO
    c["mode"] = mode
    if mode == ADAPTIVE and rng.random() < 0.5:
        c.update(tau=0.4, r_lo=50_000, r_hi=100_000)
    if mode == RATIO:
        c["ratio"] = rng.choice([10_000, 50_000, 200_000, 500_000])
    if mode == FIXED_K:
        c["fixed_k"] = logu(16, 512)
    if mode == TOP_P:
        c["ratio"] = 100_000
    if kind == "compact":
        c["gran"] = 0
    c["diag"] = kind == "step" and rng.random() < 0.1
    return c


# ------------------------------------------------------------------ lengths

def lengths(c):
    """Visual and text length of every sequence (a function of the case alone)."""
    r = random.Random("%d %d %d" % (c["batch"], c["vis"], c["text"]))
    vis, text = [c["vis"]] * c["batch"], [c["text"]] * c["batch"]
    if c["ragged"]:
        # Images of one service share a resolution range; texts differ more.
        vis = [r.randint(max(1, 3 * c["vis"] // 4), c["vis"]) for _ in vis]
        text = [r.randint(max(c["pre"] + 1, c["text"] // 8), c["text"]) for _ in text]
        vis[0], text[-1] = c["vis"], c["text"]
    return vis, text


def least_kept(c, nv):
    """Rows the budget keeps at least."""
    if c["mode"] == RATIO:
        return min(nv, max(1, -(-c["ratio"] * nv // 1_000_000)))
    if c["mode"] == FIXED_K:
        return min(nv, c["fixed_k"])
    if c["mode"] == DENSE:
        return nv
    return -(-c["r_lo"] * nv // 1_000_000) if c["mode"] == ADAPTIVE else 1


def work(c):
    esz = 4 if c["dtype"] == "fp32" else 2
    row = c["kv_heads"] * c["head_dim"] * esz  # one token's K (or V) over the kv-heads
    vis, text = lengths(c)
    b = f = 0
    for nv, tl in zip(vis, text):
        k = least_kept(c, nv)
        io = 2 * c["heads"] * c["head_dim"] * esz
        pruned, after, dense = nv + k + 2 * tl, 2 * (k + tl), 2 * (nv + tl)  # rows of K and of V
        if c["kind"] == "compact":
            b += 2 * 2 * (k + tl) * row  # K and V, read and written
            continue
        if c["kind"] == "gather":
            rows = after
        elif c["anchor"] < 0:
            rows = c["layers"] * pruned
        else:
            rows = c["anchor"] * dense + pruned + (c["layers"] - 1 - c["anchor"]) * after
        b += rows * row + c["layers"] * io
        f += 2 * c["heads"] * c["head_dim"] * rows
    return {"bytes": b, "flops": f}


def tolerance(c):
    if c["kind"] == "compact":
        return "exact"
    # Measured against `exact`: bf16 outputs 1.7e-3 off (their own rounding and
    # that of the probabilities in the P.V products); with fp32 caches the
    # outputs 7e-7 and the masses up to 4e-5 (float32 logits, multiplied by
    # 1 / tau before the exponential).  Four times that.  Kept lists and
    # activity bits may differ where two scores meet in the last bits of
    # float32.
    return {"rel": 7e-3, "max": 0.1, "differ": 0.01} if c["dtype"] == "bf16" else {"rel": 1.6e-4, "max": 2e-3, "differ": 0.01}


# ------------------------------------------------------------------- states

class State:
    def __init__(self):
        self.ctx = None

    def __del__(self):
        if self.ctx is not None:
            vp.vp_free(self.ctx)


def _recipe(c, seed):
    vis, text = lengths(c)
    r = random.Random(seed)
    scale = tuple(r.uniform(1.0, c["scale_hi"]) for _ in vis) if c["scale_hi"] > 1.0 else ()
    return W.Recipe(name="case", layers=c["layers"], batch=c["batch"], heads=c["heads"], kv_heads=c["kv_heads"],
                    head_dim=c["head_dim"], dtype=c["dtype"], vis_len=tuple(vis), vis_start=(c["pre"],) * len(vis),
                    text_len=tuple(text), steps=1, planted_frac=0.05 if c["dtype"] == "fp32" else 0.03, seed=seed,
                    beta_range=(c["beta_lo"], c["beta_hi"]), planted_scale=scale, beta_sink=c["sink"],
                    key_sigma=c["sigma"], paged=c["page"] > 0, page_size=c["page"] or 16)


def _inputs(c, seed):
    """Inputs on the GPU: per layer (q, K, V) with K and V in
    cache order [B, Hkv, T, D], plus the lengths."""
    dev = torch.device("cuda")
    r = _recipe(c, seed)
    cap = r.capacity(1) + c["room"]
    layers = []
    for layer in range(c["layers"]):
        k, v, focus, sink = W.make_layer_torch(r, layer, cap, dev)
        q = W.make_queries_torch(r, layer, 1, focus, sink, dev)[0].contiguous()
        layers.append((q, k, v))
    i32 = dict(dtype=torch.int32, device=dev)
    return layers, torch.tensor(r.vis_starts, **i32), torch.tensor(r.vis_lens, **i32), torch.tensor(r.text_lens, **i32), cap


def _given_kept(c, seed, cap):
    """A kept set of an earlier layer: random visual rows, ascending."""
    vis, _ = lengths(c)
    gen = torch.Generator().manual_seed(seed + 5)
    nsel = c["kv_heads"] if c["gran"] else 1
    kept = torch.full((c["batch"], nsel, cap), -1, dtype=torch.int32)
    count = torch.zeros((c["batch"], nsel), dtype=torch.int32)
    for b, nv in enumerate(vis):
        hi = min(nv, max(1, nv * c["r_hi"] // 1_000_000)) if c["mode"] == ADAPTIVE else least_kept(c, nv)
        k = min(hi, cap)
        for g in range(nsel):
            kept[b, g, :k] = torch.randperm(nv, generator=gen)[:k].sort().values.to(torch.int32)
            count[b, g] = k
    return kept.cuda(), count.cuda()


def prepare(c, seed):
    s = State()
    s.c = c
    layers, s.vs, s.vl, s.tl, cap = _inputs(c, seed)
    s.B, H, Hkv, D = c["batch"], c["heads"], c["kv_heads"], c["head_dim"]
    dev = torch.device("cuda")
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    s.q, s.kc, s.vc, s.keep = [], [], [], []
    if c["page"]:
        bt, n_pages, _ = W.page_table(s.B, cap, c["page"], seed)
        bt_dev = torch.from_numpy(bt).to(dev)
    for q, k, v in layers:
        if c["page"]:
            k, v = (W.scatter_pages(x, bt, n_pages, c["page"]) for x in (k, v))
        if c["layout"] == "bthd":
            k, v = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (k, v))
        s.q.append(q)
        s.keep.append((k, v))
        s.kc.append(vp.kv_paged(k, bt_dev) if c["page"] else vp.kv_contiguous(k))
        s.vc.append(vp.kv_paged(v, bt_dev) if c["page"] else vp.kv_contiguous(v))
    del layers
    if c["page"]:
        s.keep.append(bt_dev)
    s.span = vp.span(s.vs, s.vl)
    s.ctx = vp.vp_init(vp.make_config(s.B, H, Hkv, D, c["vis"], cap, vp.VP_FP32 if c["dtype"] == "fp32" else vp.VP_BF16,
                                      1 if c["page"] else 0, c["page"] or 16))
    s.budget = vp.make_budget(c["mode"], tau=c["tau"], r_lo_ppm=c["r_lo"], r_hi_ppm=c["r_hi"], ratio_ppm=c["ratio"],
                              fixed_k=c["fixed_k"], granularity=c["gran"])
    s.cap = max(1, vp.vp_max_kept(s.budget, c["vis"]))
    nsel, L = (Hkv if c["gran"] else 1), c["layers"]
    if c["kind"] == "compact":
        # The survivors that the selection at the pruning layer left.
        s.kept, s.count = _given_kept(c, seed, s.cap)
        rows = s.cap + c["text"]
        s.dst = [torch.zeros((s.B, Hkv, rows, D), dtype=dt, device=dev) for _ in range(2)]
        s.dkv = [vp.kv_contiguous(x) for x in s.dst]
        return s
    s.out = torch.zeros((L, s.B, H, D), dtype=dt, device=dev)
    if c["kind"] == "gather":
        s.kept, s.count = _given_kept(c, seed, s.cap)
        return s
    n_sel = L if c["anchor"] < 0 else 1  # layers that select
    s.kept = torch.full((n_sel, s.B, nsel, s.cap), -1, dtype=torch.int32, device=dev)
    s.count = torch.zeros((n_sel, s.B, nsel), dtype=torch.int32, device=dev)
    s.mass = torch.zeros((n_sel, s.B, H), dtype=torch.float32, device=dev)
    s.stats = torch.zeros((n_sel, s.B, 4), dtype=torch.float32, device=dev)
    if c["anchor"] > 0:
        s.all_rows = torch.arange(c["vis"], dtype=torch.int32, device=dev).repeat(s.B, 1).contiguous()
    s.n_act = s.bits = None
    if c["diag"]:
        s.n_act = torch.zeros((s.B, nsel), dtype=torch.int32, device=dev)
        s.bits = torch.zeros((s.B, nsel, (c["vis"] + 31) // 32), dtype=torch.int32, device=dev)
        vp.vp_set_diagnostics(s.ctx, 1.0 / (c["vis"] + c["text"]), s.n_act, s.bits)
    # Views a program keeps for its layers.
    s.o, s.k_, s.n_ = list(s.out), list(s.kept), list(s.count)
    s.m_, s.st_ = list(s.mass), list(s.stats)
    s.g = None
    if c["graph"]:
        _enqueue(s)  # first use outside the capture
        torch.cuda.synchronize()
        s.g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.g):
            _enqueue(s)
    return s


def _enqueue(s):
    """The calls of one decode step, layer by layer."""
    a = s.c["anchor"]
    for i in range(s.c["layers"]):
        if a < 0 or i == a:
            j = i if a < 0 else 0
            vp.vp_decode_step(s.ctx, s.B, s.q[i], s.kc[i], s.vc[i], s.span, s.tl, s.budget, s.o[i], s.k_[j], s.cap,
                              s.n_[j], s.m_[j], s.st_[j])
        elif i < a:
            vp.vp_decode_gather(s.ctx, s.B, s.q[i], s.kc[i], s.vc[i], s.span, s.tl, s.all_rows, s.c["vis"], s.vl, s.o[i])
        else:
            vp.vp_decode_gather(s.ctx, s.B, s.q[i], s.kc[i], s.vc[i], s.span, s.tl, s.k_[0], s.cap, s.n_[0], s.o[i],
                                granularity=s.c["gran"])


def run(s):
    kind = s.c["kind"]
    if kind == "compact":
        for src, dst in zip((s.kc[0], s.vc[0]), s.dkv):
            vp.vp_compact_kv(s.ctx, s.B, src, dst, s.span, s.tl, s.kept, s.cap, s.count)
        return {"k": s.dst[0], "v": s.dst[1]}
    if kind == "gather":
        vp.vp_decode_gather(s.ctx, s.B, s.q[0], s.kc[0], s.vc[0], s.span, s.tl, s.kept, s.cap, s.count, s.out[0],
                            granularity=s.c["gran"])
        return {"out": s.out}
    if s.g is not None:
        s.g.replay()
    else:
        _enqueue(s)
    r = {"out": s.out, "kept": s.kept, "count": s.count, "mass": s.mass, "stats": s.stats}
    if s.c["diag"]:
        r.update(n_act=s.n_act, bits=s.bits)
    return r


# --------------------------------------------------------- the same in 64 bits

def _k_of(c, mmax, nv, order, s_sorted):
    if c["mode"] == ADAPTIVE:
        lo = -(-c["r_lo"] * nv // 1_000_000)
        hi = max(lo, c["r_hi"] * nv // 1_000_000)
        return min(nv, min(max(math.ceil(mmax * nv), lo), hi))
    if c["mode"] == TOP_P:
        cum = torch.cumsum(s_sorted, 0)
        return min(nv, int((cum < c["ratio"] * 1e-6 * cum[-1]).sum()) + 1)
    return least_kept(c, nv)


def exact(c, seed):
    if c["kind"] == "compact":
        return None  # a copy: compared bit by bit
    layers, _, _, _, _ = _inputs(c, seed)
    vis, text = lengths(c)
    G, D, Hkv = c["heads"] // c["kv_heads"], c["head_dim"], c["kv_heads"]
    vs = c["pre"]
    nsel = Hkv if c["gran"] else 1
    outs, masses, stats, chosen = [], [], [], [None] * c["batch"]
    given = None
    if c["kind"] == "gather":
        budget = vp.make_budget(c["mode"], tau=c["tau"], r_lo_ppm=c["r_lo"], r_hi_ppm=c["r_hi"], ratio_ppm=c["ratio"],
                                fixed_k=c["fixed_k"], granularity=c["gran"])
        given = _given_kept(c, seed, max(1, vp.vp_max_kept(budget, c["vis"])))
    for i, (q, k, v) in enumerate(layers):
        out = torch.zeros((c["batch"], c["heads"], D), dtype=torch.float64, device=q.device)
        mass = torch.zeros((c["batch"], c["heads"]), dtype=torch.float64, device=q.device)
        st = torch.zeros((c["batch"], 4), dtype=torch.float64, device=q.device)
        selects = c["kind"] == "step" and (c["anchor"] < 0 or i == c["anchor"])
        for b, (nv, tl) in enumerate(zip(vis, text)):
            T = nv + tl
            kk, vv = k[b, :, :T].double(), v[b, :, :T].double()
            z = torch.matmul(q[b].double().view(Hkv, G, D), kk.transpose(1, 2)) / math.sqrt(D)  # [Hkv, G, T]
            if selects:
                m = torch.softmax(z / c["tau"], -1)[..., vs:vs + nv].sum(-1).reshape(-1)
                p1 = torch.softmax(z, -1)[..., vs:vs + nv]  # [Hkv, G, nv]
                sc = p1.mean(1) if c["gran"] else p1.mean((0, 1))[None]
                srt, order = sc.sort(dim=-1, descending=True, stable=True)
                kt = _k_of(c, float(m.max()), nv, order[0], srt[0])
                chosen[b] = order[:, :kt]
                mass[b] = m
                st[b] = torch.stack([m.mean(), m.max(), p1.sum(-1).mean(), torch.tensor(float(kt), device=q.device, dtype=torch.float64)])
            if c["kind"] == "gather":
                n = int(given[1][b, 0])
                chosen[b] = given[0][b, :, :n].long()
            keep = torch.ones((nsel, T), dtype=torch.bool, device=q.device)
            if not (c["kind"] == "step" and i < c["anchor"]):
                keep[:, vs:vs + nv] = False
                keep.scatter_(1, vs + chosen[b], True)
            a = torch.softmax(z.masked_fill(~keep[:, None, :], -math.inf), -1)
            out[b] = torch.matmul(a, vv).view(c["heads"], D)
        outs.append(out)
        if selects:
            masses.append(mass)
            stats.append(st)
    r = {"out": torch.stack(outs)}
    if c["kind"] == "step":
        r.update(kept=None, count=None, mass=torch.stack(masses), stats=torch.stack(stats))
        if c["diag"]:
            r.update(n_act=None, bits=None)
    return r

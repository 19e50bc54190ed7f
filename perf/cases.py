"""What the performance of the compression stage is measured on.

A case is one call, or the few calls a model makes per layer, through the
public binding (``paper_2606_01790_gb300.starkv``).  Its kinds:

* ``step``    the whole compression step of every layer (``starkv.step``), the
              call an agent makes once per screenshot;
* ``layer``   score_layer, select and compact of one layer: a model that
              compresses each layer inside its own forward pass;
* ``attn``    window_attention: the prefill side, which computes the window
              rows' attention output and the normalisers a step can take;
* ``host``    the step on a cache that lives in page-locked host memory.

The shapes are the repository's workloads: UI-TARS GQA (28 query heads, 4 KV
heads, window 32, 52 x 52 patches) with 5 screenshots, a trajectory's later
steps (a compressed cache plus one screenshot), 20 screenshots, a ragged batch
of trajectories, the MHA granularity, and other attention shapes; inputs are
its synthetic ones (standard normal K, V, Q with a Gaussian bump of key
directions on the screenshot grid), drawn on the GPU.  Every trajectory is
resumed in the middle (``import_slot``: the MI prior past its warm-up, a
temporal EMA to compare with), which is where all terms of the score are
active.

Selected indices, metadata and the gathered K' / V' are compared as whole
numbers (K' and V' are bit copies of input rows, seen as 16-bit words); the
fused scores and the per-layer statistics are compared as floats.
"""
import math

import numpy as np
import torch

from paper_2606_01790_gb300 import starkv as sk

D = 128                 # head dimension
STEPS_SEEN = 20         # n of a resumed trajectory: past the 5 + 10 steps of the lambda schedule


def _case(name, kind, **over):
    c = dict(name=name, kind=kind, layers=28, heads=28, kv_heads=4, window=32, grid_rows=52, grid_cols=52, shots=5,
             text=512, kept=0, pct=20, seqs=1, per_head=False, lse_given=False, decay_mode=0, aeb_mode=0,
             kv_source=0)
    c.update(over)
    return c


def listed():
    return [
        # the smallest call: one layer of two 16 x 16 screenshots; latency and launches only
        _case("step_tiny", "step", layers=1, window=8, grid_rows=16, grid_cols=16, shots=2, text=64),
        # one layer inside a model's forward pass, through the three per-layer calls
        _case("layer_5shot", "layer", layers=1),
        # the step an agent makes most: a compressed cache plus one new screenshot and 64 text tokens
        _case("step_traj_28l", "step", shots=1, text=64, kept=2736),
        # the headline step: a fresh 5-screenshot prompt over the whole stack
        _case("step_5shot_28l", "step"),
        # the largest single prompt: 20 screenshots and 2048 text tokens
        _case("step_long_28l", "step", shots=20, text=2048),
        # serving: 16 trajectories of 1 to 12 screenshots and 128 to 1024 text tokens in one call
        _case("step_ragged_16", "step", shots=12, text=1024, seqs=16),
        # per-KV-head selection on a later trajectory step, odd length
        _case("step_per_head_28l", "step", shots=2, text=333, kept=3040, per_head=True),
        # the MI prior at MHA granularity: every query head has its own replicated K and V
        _case("step_mha_28l", "step", kv_heads=28, kv_source=4),
        # the step whose normalisers the prefill attention already gave, on a 32 / 8-head model
        _case("step_lse_gqa8_32l", "step", layers=32, heads=32, kv_heads=8, window=16, shots=3, text=403,
              lse_given=True),
        # prefill: the window rows' attention over the 5-screenshot cache, every layer
        _case("attn_5shot_28l", "attn"),
        # prefill of a small ragged batch on a 32 / 8-head model
        _case("attn_gqa8_3seq", "attn", layers=8, heads=32, kv_heads=8, window=16, shots=2, text=301, seqs=3),
        # a cache kept in page-locked host memory, a later trajectory step
        _case("host_traj_28l", "host", shots=1, text=64, kept=2736),
    ]


_SHAPES = [(28, 4, 32), (28, 4, 32), (28, 4, 24), (32, 8, 16), (16, 2, 32), (8, 8, 16), (40, 8, 8), (12, 1, 16)]
_MAX_TOKEN_LAYERS = 1_500_000    # layers x tokens of a drawn case (the 20-screenshot step has 1.57 M)


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["layer"] * 2 + ["attn"] * 2 + ["host"])
    heads, kv_heads, window = rng.choice(_SHAPES)
    c = _case("", kind, heads=heads, kv_heads=kv_heads, window=window)
    del c["name"]
    c["grid_rows"], c["grid_cols"] = rng.choice([(52, 52), (52, 52), (37, 66), (28, 45), (16, 16)])
    c["layers"] = 1 if kind == "layer" else int(round(math.exp(rng.uniform(0, math.log(32)))))
    c["text"] = rng.randint(64, 1024)
    c["pct"] = rng.choice([10, 20, 30, 40])
    if rng.random() < 0.4:     # a later step of a trajectory
        c["kept"], c["shots"] = int(math.exp(rng.uniform(math.log(300), math.log(9000)))), 1
    else:
        c["shots"] = int(round(math.exp(rng.uniform(0, math.log(20)))))
    if kind == "step":
        c["per_head"] = rng.random() < 0.2
        c["lse_given"] = rng.random() < 0.25
        c["decay_mode"] = rng.choice([0, 0, 0, 1, 2])
        c["aeb_mode"] = rng.choice([0, 0, 0, 1])
        if heads == 28 and not c["per_head"] and rng.random() < 0.1:
            c["kv_heads"], c["kv_source"] = 28, 4
    if kind in ("step", "attn") and rng.random() < 0.3:
        c["seqs"] = rng.randint(2, 8)
    while c["layers"] > 1 and _token_layers(c) > _MAX_TOKEN_LAYERS * (0.25 if kind == "host" else 1.0):
        c["layers"] -= 1
    while c["seqs"] > 1 and _token_layers(c) > _MAX_TOKEN_LAYERS:
        c["seqs"] -= 1
    return c


def _token_layers(c):
    tokens = c["shots"] * c["grid_rows"] * c["grid_cols"] + c["text"] + c["kept"]
    return c["layers"] * c["seqs"] * tokens * c["kv_heads"] / 4


# ---------------------------------------------------------------- shapes of one case

def _shapes(c):
    """[(screenshots, text tokens, budget percent)] of the sequences: the case's own, and smaller ones
    drawn from a fixed stream for the further sequences of a batch (sizes depend on the case alone)."""
    rng = np.random.default_rng([c["shots"], c["text"], c["seqs"]])
    out = [(c["shots"], c["text"], c["pct"])]
    for _ in range(1, c["seqs"]):
        out.append((int(rng.integers(1, c["shots"] + 1)), int(rng.integers(min(128, c["text"]), c["text"] + 1)),
                    int(rng.choice([10, 20, 30]))))
    return out


def _dims(c, i):
    """(L, B, newest frame) of sequence i."""
    shots, text, pct = _shapes(c)[i]
    per_shot = c["grid_rows"] * c["grid_cols"]
    old = 5 if c["kept"] else 0     # a kept cache holds tokens of five earlier frames
    L = c["kept"] + shots * per_shot + max(text, c["window"])
    B = min(pct * (old + shots) * per_shot // 100, L - c["window"])
    return L, B, old + shots - 1


def _layout(c, i, rng):
    """Metadata words of sequence i: [L] for a fresh prompt (text runs between the screenshots, the last
    run at least the window), [layers][L] for a compressed cache plus new tokens."""
    shots, text, _ = _shapes(c)[i]
    text = max(text, c["window"])
    R, C = c["grid_rows"], c["grid_cols"]
    row, col = (a.reshape(-1) for a in np.meshgrid(np.arange(R), np.arange(C), indexing="ij"))

    def frames(first, n, runs):
        parts = []
        for f in range(n):
            parts += [np.zeros(runs[f], np.uint32), sk.pack_meta(np.ones(R * C), np.full(R * C, first + f), row, col)]
        return np.concatenate(parts + [np.zeros(runs[n], np.uint32)])

    old = 5 if c["kept"] else 0
    last = max(c["window"], text // (shots + 1)) if not old else text
    runs = [(text - last) // shots] * shots + [last]
    runs[0] += text - sum(runs)
    new = frames(old, shots, runs)
    if not old:
        return new
    before = frames(0, old, [512 // (old + 1)] * (old + 1))
    if c["kept"] > before.size:
        before = np.concatenate([np.zeros(c["kept"] - before.size, np.uint32), before])
    kept = [np.sort(rng.permutation(before.size)[:c["kept"]]) for _ in range(c["layers"])]
    return np.stack([np.concatenate([before[k], new]) for k in kept])


def _inputs(c, seed):
    """The tensors of every sequence, drawn on the GPU from the seed."""
    nl, H, G, w, R, C = (c[k] for k in ("layers", "heads", "kv_heads", "window", "grid_rows", "grid_cols"))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    src = c["kv_source"] or G

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    def uniform(*shape):
        return torch.rand(*shape, generator=gen, device="cuda")

    seqs = []
    for i in range(c["seqs"]):
        L, B, frame = _dims(c, i)
        words = sk.meta_tensor(_layout(c, i, rng)).cuda()
        vis, fr, rw, cl = _fields(words)
        u = torch.nn.functional.normalize(normal(nl, src, 1, D), dim=3)
        cen = uniform(2, nl, src, 1) * torch.tensor([R, C], device="cuda").view(2, 1, 1, 1)
        amp = (0.5 + 3.5 * uniform(frame + 1)) if c["shots"] >= 12 else torch.full((frame + 1,), 2.0, device="cuda")
        tok = [t.view(-1, 1, L) for t in (vis, fr, rw, cl)]
        dist2 = (tok[2] - cen[0]) ** 2 + (tok[3] - cen[1]) ** 2
        bump = torch.where(tok[0] != 0, amp[tok[1].long()] * torch.exp(-dist2 / 18.0), 0.0)   # [nl][src][L]
        k = torch.empty(nl, src, L, D, dtype=torch.bfloat16, device="cuda")
        v = torch.empty_like(k)
        for l in range(nl):
            k[l] = normal(src, L, D) + bump[l].unsqueeze(2) * u[l]
            v[l] = normal(src, L, D)
        q = normal(nl, src, H // src * w, D) + math.sqrt(D) * u
        if src != G:
            k, v = (t.repeat_interleave(G // src, dim=1) for t in (k, v))
        seqs.append(dict(L=L, B=B, frame=frame, words=words, k=k, v=v,
                         q=q.to(torch.bfloat16).reshape(nl, H, w, D).contiguous(),
                         mi=rng.uniform(0.02, 0.3, (nl, G)),
                         m=(np.float32(w / L) * rng.lognormal(0.0, 0.4, (nl, G, R * C))).astype(np.float32)))
        if c["lse_given"]:
            seqs[-1]["lse"] = _lse(c, seqs[-1]).float()
    return seqs


def _fields(words):
    """(visual, frame, row, column) of metadata words."""
    return (words >> 31) & 1, (words >> 20) & 0x7FF, (words >> 10) & 0x3FF, words & 0x3FF


# ---------------------------------------------------------------- the calls

def _config(c):
    return sk.Config(n_layers=c["layers"], n_heads=c["heads"], n_kv_heads=c["kv_heads"], window=c["window"],
                     grid_rows=c["grid_rows"], grid_cols=c["grid_cols"], max_seqs=c["seqs"],
                     decay_mode=c["decay_mode"], aeb_mode=c["aeb_mode"],
                     select_mode=sk.SELECT_PER_HEAD if c["per_head"] else sk.SELECT_GLOBAL)


def _resume(st, c, slot, x):
    """Puts a running trajectory's state into a slot, as a program that resumes one does."""
    buf = sk.export_slot(st, slot)
    torch.cuda.synchronize()
    n = np.full(c["layers"], STEPS_SEEN, np.int32).tobytes()
    body = n + b"\0" * (-len(n) % 8) + x["mi"].astype(np.float64).tobytes() + x["m"].tobytes()
    buf[32:] = torch.from_numpy(np.frombuffer(body, np.uint8).copy())
    sk.import_slot(st, slot, buf)
    return buf


def prepare(case, seed):
    c = case
    nl, H, G, w = c["layers"], c["heads"], c["kv_heads"], c["window"]
    P = G if c["per_head"] else 1
    host = c["kind"] == "host"
    attn = c["kind"] == "attn"
    xs = _inputs(c, seed)
    st = sk.init_state(_config(c))
    keep = [] if attn else [_resume(st, c, i, x) for i, x in enumerate(xs)]

    def room(sizes, dtype):
        """One buffer for every sequence's output of a kind, and the sequences' views of it."""
        buf = (torch.empty(sum(sizes), dtype=dtype, pin_memory=True) if host
               else torch.empty(sum(sizes), dtype=dtype, device="cuda"))
        return buf, list(buf.split(sizes))

    out, seqs = {}, [sk.Seq(L=x["L"], cur_frame=x["frame"], budget=x["B"], slot=i) for i, x in enumerate(xs)]
    if attn:
        kinds = dict(attn_o=(torch.float32, [nl * H * w * D] * len(xs)), attn_lse=(torch.float32, [nl * H * w] * len(xs)))
    else:
        rows = [G * (x["B"] + w) * D * nl for x in xs]
        kinds = dict(idx=(torch.int32, [nl * P * x["B"] for x in xs]), k_out=(torch.bfloat16, rows),
                     v_out=(torch.bfloat16, rows), meta_out=(torch.int32, [nl * P * (x["B"] + w) for x in xs]),
                     score=(torch.float32, [nl * P * (x["L"] - w) for x in xs]),
                     stats=(torch.float32, [nl * sk.stats_stride(G)] * len(xs)))
        if c["kind"] == "layer":
            kinds["S"] = (torch.float32, [nl * G * (x["L"] - w) for x in xs])
    for name, (dtype, sizes) in kinds.items():
        out[name], views = room(sizes, dtype)
        for s, view in zip(seqs, views):
            setattr(s, name, view)
        if dtype == torch.bfloat16:
            out[name] = out[name].view(torch.int16)     # bit copies of input rows
    for s, x in zip(seqs, xs):
        for name in ("k", "v", "q"):
            setattr(s, name, x[name].cpu().pin_memory() if host else x[name])
        if not attn:
            s.meta = x["words"].cpu().pin_memory() if host else x["words"]
            s.meta_layer_stride = s.L if s.meta.dim() == 2 else 0
            s.lse = x.get("lse")
    ws = sk.workspace(st, seqs, host=host)
    return dict(case=c, st=st, seqs=seqs, ws=ws, out=out, keep=keep)


def run(state):
    st, seqs, ws = state["st"], state["seqs"], state["ws"]
    kind = state["case"]["kind"]
    if kind == "step":
        sk.step(st, seqs, ws)
    elif kind == "layer":
        for layer in range(state["case"]["layers"]):
            sk.score_layer(st, layer, seqs, ws)
            sk.select(st, layer, seqs, ws)
            sk.compact(st, layer, seqs, ws)
    elif kind == "attn":
        sk.window_attention(st, seqs, ws)
    else:
        sk.step_host(st, seqs, ws)
    return state["out"]


def work(case):
    """Each input that the result depends on read once, each output written once; one Q K^T (and one P V)."""
    c = case
    nl, H, G, w = c["layers"], c["heads"], c["kv_heads"], c["window"]
    P = G if c["per_head"] else 1
    nbytes = flops = 0
    for i in range(c["seqs"]):
        L, B, _ = _dims(c, i)
        q, k = H * w * D * 2, G * L * D * 2
        if c["kind"] == "attn":
            nbytes += nl * (2 * k + q + H * w * (D + 1) * 4)
            flops += nl * 4 * H * w * (L - w) * D
            continue
        rows = G * (B + w) * D * 2
        nbytes += nl * (k + q + rows + 2 * rows                                   # K, Q, the kept V; K', V'
                        + 4 * L + 4 * P * (2 * B + w + L - w)                     # metadata; idx, metadata', scores
                        + 8 * G * c["grid_rows"] * c["grid_cols"]                 # the temporal EMA, read and written
                        + (H * w * 4 if c["lse_given"] else 0)
                        + (4 * G * (L - w) if c["kind"] == "layer" else 0))       # S
        flops += nl * 2 * H * w * (L - w) * D
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # attn: P is rounded to fp16 before the product with V, so an element is off by about 2^-12 of the terms'
    # root sum of squares; the 32-bit sums behind the normalisers and the scores are good to about 1e-6.
    # step, layer: a token whose score lies within rounding of the B-th may be swapped for its neighbour, and
    # every row between the two then moves by one.
    if case["kind"] == "attn":
        return {"rel": 8e-4, "max": 1e-2}      # measured: attn_o 2.1e-4, attn_lse 5e-8 from 64 bits
    return {"rel": 1e-5, "max": 1e-3, "differ": 0.01}     # measured: score 0.3e-6 to 3e-6, stats 1e-8 from 64 bits


# ---------------------------------------------------------------- the same results in 64 bits, in plain torch

def _logits(c, x, layer, g):
    """[H / G * w][L - w] logits of one layer and group in float64."""
    n = c["heads"] // c["kv_heads"]
    q = x["q"][layer, g * n:(g + 1) * n].reshape(n * c["window"], D).double()
    return q @ x["k"][layer, g, :x["L"] - c["window"]].double().t() / math.sqrt(D)


def _lse(c, x):
    n = c["heads"] // c["kv_heads"]
    out = torch.empty(c["layers"], c["kv_heads"], n * c["window"], dtype=torch.float64, device="cuda")
    for l in range(c["layers"]):
        for g in range(c["kv_heads"]):
            out[l, g] = torch.logsumexp(_logits(c, x, l, g), dim=1)
    return out.reshape(c["layers"], c["heads"], c["window"])


def _group_scores(c, x, layer):
    """S [G][L - w] (Eqs. 2-4): softmax over the past keys, summed over the group's window rows, pooled over
    five tokens with zero padding, averaged over the group's heads."""
    rows = []
    for g in range(c["kv_heads"]):
        p = torch.softmax(_logits(c, x, layer, g), dim=1).sum(dim=0)
        pooled = torch.nn.functional.avg_pool1d(p.view(1, 1, -1), 5, stride=1, padding=2, count_include_pad=True)
        rows.append(pooled.view(-1) * c["kv_heads"] / c["heads"])
    return torch.stack(rows)


def _mutual_information(s, cells, bins=8, n_cells=64):
    n = s.numel()
    if n == 0:
        return 0.0
    rank = torch.empty(n, dtype=torch.int64, device=s.device)
    rank[torch.argsort(s, stable=True)] = torch.arange(n, device=s.device)
    joint = torch.bincount(rank * bins // n * n_cells + cells, minlength=bins * n_cells).double().view(bins, n_cells) / n
    prod = joint.sum(1, keepdim=True) * joint.sum(0, keepdim=True)
    return float(torch.where(joint > 0, joint * torch.log(joint / prod), 0.0).nansum())


def _calibrated(c, x, layer, S):
    """(fused score [P][L - w], statistics) of one layer from its S: Eqs. 5-9, Sec. 3.6."""
    G, R, C = c["kv_heads"], c["grid_rows"], c["grid_cols"]
    lp = S.shape[1]
    words = x["words"] if x["words"].dim() == 1 else x["words"][layer]
    vis, fr, rw, cl = (t[:lp].long() for t in _fields(words))
    vis = vis != 0
    cells = (rw * 8 // R) * 8 + cl * 8 // C
    newest = vis & (fr == x["frame"])
    mi = torch.tensor([_mutual_information(S[g][vis], cells[vis]) for g in range(G)], dtype=torch.float64, device="cuda")
    bar = 0.9 * torch.from_numpy(x["mi"][layer]).cuda() + 0.1 * mi
    norm = (bar - bar.min()) / (bar.max() - bar.min() + 1e-6)
    wg = torch.softmax(norm, 0)
    m = torch.from_numpy(x["m"][layer]).cuda().double()
    cur = torch.zeros(G, R * C, dtype=torch.float64, device="cuda")
    cur[:, rw[newest] * C + cl[newest]] = S[:, newest]
    phi = (cur * m).sum(1) / torch.clamp(cur.norm(dim=1) * m.norm(dim=1), min=1e-300)
    sbar, top = S.mean(0), S.argmax(0)
    lam = 0.5

    def fused(s, g):
        age = (x["frame"] - fr) * phi[g]
        shape = [lambda: torch.exp(-0.2 * age), lambda: torch.clamp(1 - 0.2 * age, min=0),
                 lambda: (1 + age) ** -0.2][c["decay_mode"]]()
        d = torch.where(vis, 0.1 + 0.9 * shape, 1.0)
        z = s.sum()
        if c["aeb_mode"]:
            h = s.max() / (z + 1e-12)
            temp = 0.95 + 0.1 * (1 - h)
        else:
            p = s / (z + 1e-12)
            h = -(p * torch.log(p + 1e-12)).sum() / math.log(lp)
            temp = 0.95 + 0.1 * h
        return torch.clamp(s * ((1 - lam) + lam * G * wg[g]) * d, min=0) ** (1 / temp), h, temp

    parts = [fused(S[g], g) for g in range(G)] if c["per_head"] else [fused(sbar, top)] * G
    score = torch.stack([p[0] for p in parts[:G if c["per_head"] else 1]])
    h, temp = (torch.stack([p[k] for p in parts]) for k in (1, 2))
    head = torch.stack([h.mean(), temp.mean(), h.new_tensor(lam), h.new_tensor(STEPS_SEEN), sbar.sum(), vis.sum().double(),
                        h.new_tensor(x["B"]), h.new_tensor(0)])
    return score, torch.cat([head, mi, bar, wg, phi, h, temp])


def exact(case, seed):
    c = case
    xs = _inputs(c, seed)
    nl = c["layers"]
    if c["kind"] == "attn":
        o, lse = [], []
        for x in xs:
            lp = x["L"] - c["window"]
            for l in range(nl):
                for g in range(c["kv_heads"]):
                    z = _logits(c, x, l, g)
                    lse.append(torch.logsumexp(z, dim=1))
                    o.append((torch.softmax(z, dim=1) @ x["v"][l, g, :lp].double()).reshape(-1))
        return {"attn_o": torch.cat(o), "attn_lse": torch.cat(lse)}
    score, stats, maps = [], [], []
    for x in xs:
        for l in range(nl):
            S = _group_scores(c, x, l)
            a, b = _calibrated(c, x, l, S)
            maps.append(S.reshape(-1))
            score.append(a.reshape(-1))
            stats.append(b)
    # the selected rows follow the scores but for ties within rounding, so they have no value of their own here
    out = dict(score=torch.cat(score), stats=torch.cat(stats), idx=None, k_out=None, v_out=None, meta_out=None)
    if c["kind"] == "layer":
        out["S"] = torch.cat(maps)
    if c["kind"] == "host":
        out = {k: t.cpu() if t is not None else None for k, t in out.items()}
    return out

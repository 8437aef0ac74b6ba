"""Performance cases of the KV-cache translation library, through its public entry points.

Each case is one call a serving program makes: a translation of a batch of context caches
(MLP translators, dense or Top-K routed; MoT-h activations; backbone translators) or one target
layer's replay attention. Shapes are those of the repository's own workloads (the model pairs of
``synth``); lengths, ragged batches, windows of layers and types vary as in use.

Inputs are drawn on the GPU from the seed: caches with per-channel LogNormal(0, 0.5) scales,
weights N(0, 1 / fan_in), guidance maps with a sink, recency, heavy columns and LogNormal noise.
``exact`` restates each path in plain torch in 64 bits.
"""
import math

import torch

import paper_2607_28979_gb300.mot as M

DEV = "cuda"

# Model pairs: source layers, heads, head dim; target layers, heads, head dim; translator width H.
PAIRS = {
    "gpt2s_opt125m": dict(ls=12, hs=12, ds=64, lt=12, ht=12, dt=64, hidden=1536),
    "qwen05_qwen15": dict(ls=24, hs=2, ds=64, lt=28, ht=2, dt=128, hidden=1024),
    "gpt2m_qwen7": dict(ls=24, hs=16, ds=64, lt=28, ht=4, dt=128, hidden=2048),
    "qwen7_qwen7": dict(ls=28, hs=4, ds=128, lt=28, ht=4, dt=128, hidden=2048),
}
# MoT-h: source activation width in place of the heads; act = the target's activation width.
PAIRS_H = {
    "gpt2s_opt125m": dict(ls=12, da=768, lt=12, ht=12, dt=64, hidden=1536, act=768),
    "qwen05_qwen15": dict(ls=24, da=896, lt=28, ht=2, dt=128, hidden=1024, act=1536),
}
# Backbone windows: first target layer, slots; rows of width 128, 4 heads, FFN 512.
PAIRS_BT = {"gpt2s_opt125m": (4, 4), "qwen05_qwen15": (10, 8)}
BT_WIDTH, BT_HEADS, BT_FFN = 128, 4, 512
# Replay: query heads, key/value heads, head dim of the target.
PAIRS_R = {"qwen15": (12, 2, 128), "opt125m": (12, 12, 64), "qwen7": (28, 4, 128)}


def _mlp(pair, lens, **kw):
    c = dict(kind="mlp", pair=pair, lens=",".join(map(str, lens)), dtype="bf16", experts=4,
             top_k=0, first=0, layers=PAIRS[pair]["lt"])
    c.update(kw)
    return c


def listed():
    return [
        # The parity-precision call: fp32 caches of the first four layers, one 64-token context
        # (the paper's training context length).
        _mlp("gpt2s_opt125m", (64,), name="mlp_fp32_64", dtype="fp32", experts=2, src_layers=4,
             layers=4, hidden=768),
        # The smallest bf16 call: one short prompt handed from a small model to a larger one.
        _mlp("qwen05_qwen15", (64,), name="mlp_qwen05_64"),
        # An ordinary batch of full-length contexts (the repository's benchmark pair).
        _mlp("gpt2s_opt125m", (1024,) * 8, name="mlp_gpt2s_8x1024"),
        # A ragged batch with odd lengths.
        _mlp("qwen05_qwen15", (4096, 2913, 1001, 77), name="mlp_qwen05_ragged"),
        # The largest: four long contexts, every layer of the 7B pair (the headline benchmark).
        _mlp("qwen7_qwen7", (32768, 16384, 8192, 4096), name="mlp_qwen7_long"),
        # Top-2 routing of eight translators over the paper's default channel window
        # (ratio 0.3: 9 of the 28 target layers).
        _mlp("gpt2m_qwen7", (8192, 8192), name="routed_gpt2m_top2", experts=8, top_k=2, first=10,
             layers=9),
        # MoT-h: activations translated, K and V restored by the target's projections.
        dict(name="moth_qwen05", kind="moth", pair="qwen05_qwen15", lens="4096,4096,4096,4096",
             experts=4),
        # Backbone translators with the paper's default Top-1 of 2: many heads per token.
        dict(name="bt_gpt2s_top1", kind="bt", pair="gpt2s_opt125m",
             lens=",".join(["1024"] * 8), experts=2, top_k=1),
        # The same with two heads per token, a longer window and a ragged batch.
        dict(name="bt_qwen05_ragged", kind="bt", pair="qwen05_qwen15", lens="4096,2500,1023,300",
             experts=2, top_k=1),
        # One source-guided replay layer at the paper's S = 128 (26 of 28 layers of a replay).
        dict(name="replay_guided_qwen15", kind="replay", pair="qwen15",
             lens="4096,4096,4096,4096", top_s=128, guided=True),
        # The same for a target without grouped heads and with head width 64.
        dict(name="replay_guided_opt125m", kind="replay", pair="opt125m",
             lens=",".join(["1024"] * 8), top_s=128, guided=True),
        # One of the bottom layers that replay with full causal attention.
        dict(name="replay_full_qwen15", kind="replay", pair="qwen15",
             lens="4096,4096,4096,4096", top_s=128, guided=False),
    ]


def _draw_lens(rng, lo, hi, most):
    """1 to 8 lengths, log-uniform in [lo, hi], often odd; at most `most` positions with padding."""
    n = rng.choice((1, 1, 2, 3, 4, 8))
    top = max(lo, min(hi, most // n))
    lens = [int(round(math.exp(rng.uniform(math.log(lo), math.log(top))))) for _ in range(n)]
    if rng.random() < 0.3:
        lens = [max(lens)] * n
    return ",".join(map(str, lens))


def draw(rng):
    kind = rng.choice(("mlp", "mlp", "routed", "fp32", "moth", "bt", "replay", "replay", "full"))
    if kind == "fp32":
        lens = _draw_lens(rng, 16, 512, 1024)
        return _mlp("gpt2s_opt125m", [int(x) for x in lens.split(",")], dtype="fp32",
                    experts=rng.choice((2, 4)), src_layers=4, layers=4,
                    hidden=rng.choice((768, 1536)))
    if kind in ("mlp", "routed"):
        pair = rng.choice(sorted(PAIRS))
        lens = [int(x) for x in _draw_lens(rng, 16, 8192, 16384).split(",")]
        c = _mlp(pair, lens)
        if rng.random() < 0.5 or pair == "gpt2m_qwen7":   # a channel window
            c["layers"] = max(1, round(0.3 * PAIRS[pair]["lt"]))
            c["first"] = rng.randrange(0, PAIRS[pair]["lt"] - c["layers"] + 1)
        if kind == "routed":
            c["experts"] = rng.choice((2, 4, 8))
            c["top_k"] = 1 if c["experts"] == 2 else rng.choice((1, 2))
        return c
    if kind == "moth":
        return dict(kind="moth", pair=rng.choice(sorted(PAIRS_H)),
                    lens=_draw_lens(rng, 16, 4096, 16384), experts=rng.choice((2, 4)))
    if kind == "bt":
        return dict(kind="bt", pair=rng.choice(sorted(PAIRS_BT)),
                    lens=_draw_lens(rng, 16, 4096, 16384), experts=2, top_k=rng.choice((0, 1, 1)))
    return dict(kind="replay", pair=rng.choice(sorted(PAIRS_R)),
                lens=_draw_lens(rng, 64, 4096, 16384), top_s=rng.choice((32, 64, 128, 128, 256)),
                guided=kind != "full")


# ---------------------------------------------------------------- shapes

class _Shape:
    """The dimensions of a translation case and its channel map."""

    def __init__(self, c):
        self.lens = [int(x) for x in c["lens"].split(",")]
        self.B, self.S, self.T = len(self.lens), max(self.lens), sum(self.lens)
        self.kind, self.E, self.K = c["kind"], c["experts"], c.get("top_k", 0)
        p = dict((PAIRS_H if self.kind == "moth" else PAIRS)[c["pair"]])
        self.Ls, self.Lt = c.get("src_layers", p["ls"]), p["lt"]
        if "src_layers" in c:
            self.Lt = c["layers"]
        self.Hs, self.ds = (1, p["da"]) if self.kind == "moth" else (p["hs"], p["ds"])
        self.Ht, self.dt = p["ht"], p["dt"]
        self.H = c.get("hidden", p["hidden"])
        self.Ds, self.Dt = self.Hs * self.ds, self.Ht * self.dt
        self.act = p.get("act", 0)
        self.dtype = c.get("dtype", "bf16")
        ratio = [0 if self.Lt == 1 else (2 * l * (self.Ls - 1) + self.Lt - 1) // (2 * (self.Lt - 1))
                 for l in range(self.Lt)]
        if self.kind == "bt":
            self.first, self.N = PAIRS_BT[c["pair"]]
            self.map, self.tl = ratio, list(range(self.first, self.first + self.N))
        else:
            first, n = c.get("first", 0), c.get("layers", self.Lt)
            self.tl = list(range(first, first + n))
            self.map = [ratio[l] if l in self.tl else -1 for l in range(self.Lt)]
        self.tdtype = torch.float32 if self.dtype == "fp32" else torch.bfloat16

    def tensors(self):
        """(name, shape, mean, standard deviation) of one block of the weight blob, in order."""
        E, Ds, Dt, H = self.E, self.Ds, self.Dt, self.H
        if self.kind == "bt":
            P, s, d, f, N = self.Hs, self.ds, BT_WIDTH, BT_FFN, self.N
            out = [("wg", (E, N * Ds), 0, N * Ds), ("bg", (E,), 0, N * Ds)]
            for m in range(E):
                out += [(f"ling{m}", (s,), 1, 100), (f"linb{m}", (s,), 0, 100),
                        (f"win{m}", (d, s), 0, s), (f"bin{m}", (d,), 0, s)]
                for r in range(N):
                    k = f"{m}_{r}"
                    out += [("lqg" + k, (d,), 1, 100), ("lqb" + k, (d,), 0, 100),
                            ("lcg" + k, (d,), 1, 100), ("lcb" + k, (d,), 0, 100)]
                    for w in "qkvo":
                        out += [(f"w{w}{k}", (d, d), 0, d), (f"b{w}{k}", (d,), 0, d)]
                    out += [("lfg" + k, (d,), 1, 100), ("lfb" + k, (d,), 0, 100),
                            ("wf1" + k, (f, d), 0, d), ("bf1" + k, (f,), 0, d),
                            ("wf2" + k, (d, f), 0, f), ("bf2" + k, (d,), 0, f)]
                out += [(f"log{m}", (P * d,), 1, 100), (f"lob{m}", (P * d,), 0, 100),
                        (f"wout{m}", (Dt, P * d), 0, P * d), (f"bout{m}", (Dt,), 0, P * d)]
            return out
        Dm = self.act or Dt
        out = [("wg", (E, Ds), 0, Ds), ("bg", (E,), 0, Ds)]
        for m in range(E):
            out += [(f"w1{m}", (H, Ds), 0, Ds), (f"b1{m}", (H,), 0, Ds),
                    (f"w2{m}", (Dm, H), 0, H), (f"b2{m}", (Dm,), 0, H)]
        if self.act:
            out += [("wk", (Dt, Dm), 0, Dm), ("wv", (Dt, Dm), 0, Dm)]
        return out

    def blocks(self):
        return 2 if self.kind == "bt" else len(self.tl) * (1 if self.act else 2)

    def src_shape(self):
        if self.act:
            return (self.Ls, self.B, self.S, self.Ds)
        return (self.Ls, self.B, self.Hs, self.S, self.ds)

    def dst_shape(self):
        return (self.Lt, self.B, self.Ht, self.S, self.dt)


def _draw_cache(sh, gen):
    out = torch.empty(sh.src_shape(), dtype=sh.tdtype, device=DEV)
    chan = (1, 1, sh.Ds) if sh.act else (1, sh.Hs, 1, sh.ds)
    for l in range(sh.Ls):
        s = torch.exp(0.5 * torch.randn(chan, generator=gen, device=DEV))
        out[l] = torch.randn(out[l].shape, generator=gen, device=DEV) * s
    return out


def _draw_blob(sh, gen):
    """The packed weights, [blocks][elements of a block], on the GPU."""
    items = sh.tensors()
    n = [math.prod(shape) for _, shape, _, _ in items]
    rep = torch.tensor(n)
    std = torch.repeat_interleave(torch.tensor([f ** -0.5 for *_, f in items]), rep).to(DEV)
    mean = torch.repeat_interleave(torch.tensor([float(m) for _, _, m, _ in items]), rep).to(DEV)
    out = torch.empty((sh.blocks(), sum(n)), dtype=sh.tdtype, device=DEV)
    for g in range(sh.blocks()):
        out[g] = torch.randn(sum(n), generator=gen, device=DEV) * std + mean
    return out


def _translation_inputs(c, seed):
    sh = _Shape(c)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    src = [_draw_cache(sh, gen) for _ in range(1 if sh.act else 2)]
    return sh, src, _draw_blob(sh, gen)


def _replay_inputs(c, seed):
    Hq, Hkv, d = PAIRS_R[c["pair"]]
    lens = [int(x) for x in c["lens"].split(",")]
    B, N = len(lens), max(lens)
    gen = torch.Generator(device=DEV).manual_seed(seed)

    def normal(h):
        return torch.randn((B, h, N, d), generator=gen, device=DEV).to(torch.bfloat16)

    q, k, v = normal(Hq), normal(Hkv), normal(Hkv)
    guide = None
    if c["guided"]:   # a source model's head-averaged attention: rows u, columns j <= u
        guide = torch.empty((B, N, N), dtype=torch.bfloat16, device=DEV)
        j = torch.arange(N, device=DEV)
        for b in range(B):
            heavy = torch.rand(N, generator=gen, device=DEV) < 0.02
            col = torch.where(heavy, 8.0, 1.0)
            col[0] = 60.0
            for u0 in range(0, N, 1024):
                u = torch.arange(u0, min(N, u0 + 1024), device=DEV)[:, None]
                noise = torch.exp(torch.randn((u.shape[0], N), generator=gen, device=DEV))
                s = noise * (col + 20.0 * torch.exp(-(u - j).clamp(min=0) / 16.0))
                s = torch.where(j <= u, s, 0.0)
                guide[b, u0:u0 + u.shape[0]] = s / s.sum(1, keepdim=True)
    return (Hq, Hkv, d), lens, q, k, v, guide


# ---------------------------------------------------------------- prepare and run

def _host(blob):
    return (blob.view(torch.int16) if blob.dtype == torch.bfloat16 else blob).cpu().numpy()


def prepare(case, seed):
    if case["kind"] == "replay":
        (Hq, Hkv, d), lens, q, k, v, guide = _replay_inputs(case, seed)
        n_full = 2
        h = M.mot_create_replay(M.mot_replay_config(Hq, Hkv, d, len(lens), max(lens),
                                                    case["top_s"], n_full))
        return dict(kind="replay", h=h, layer=n_full if case["guided"] else 0, q=q, k=k, v=v,
                    guide=guide, batch=len(lens), out=torch.zeros_like(q),
                    lens=torch.tensor(lens, dtype=torch.int32, device=DEV))
    sh, src, blob = _translation_inputs(case, seed)
    if sh.kind == "moth":
        h = M.mot_create_h(M.mot_h_config(sh.Ls, sh.Ds, sh.Lt, sh.act, sh.Ht, sh.dt, sh.E, sh.K,
                                          sh.H, sh.B, sh.S, M.MOT_BF16))
    else:
        cfg = M.make_config(sh.Ls, sh.Hs, sh.ds, sh.Lt, sh.Ht, sh.dt, sh.E,
                            0 if sh.kind == "bt" else sh.H, sh.B, sh.S, sh.dtype, sh.K, sh.map)
        if sh.kind == "bt":
            h = M.mot_create_bt(cfg, M.mot_bt_config(sh.first, sh.N, BT_WIDTH, BT_HEADS, BT_FFN))
        else:
            h = M.mot_create(cfg)
    M.mot_load_weights(h, _host(blob))
    dst = [torch.zeros(sh.dst_shape(), dtype=sh.tdtype, device=DEV) for _ in range(2)]
    return dict(kind=sh.kind, h=h, src=src, dst=dst, batch=sh.B,
                lens=torch.tensor(sh.lens, dtype=torch.int32, device=DEV))


def run(state):
    s = state
    if s["kind"] == "replay":
        M.mot_replay_attention(s["h"], s["layer"], s["q"], s["k"], s["v"], s["guide"], s["lens"],
                               s["batch"], s["out"])
        return s["out"]
    if s["kind"] == "moth":
        M.mot_translate_h(s["h"], s["src"][0], s["lens"], s["batch"], *s["dst"])
    elif s["kind"] == "bt":
        M.mot_translate_bt(s["h"], *s["src"], s["lens"], s["batch"], *s["dst"])
    else:
        M.mot_translate(s["h"], *s["src"], s["lens"], s["batch"], *s["dst"])
    return s["dst"]


# ---------------------------------------------------------------- work and tolerance

def work(case):
    if case["kind"] == "replay":
        Hq, Hkv, d = PAIRS_R[case["pair"]]
        lens = [int(x) for x in case["lens"].split(",")]
        byts = sum(lens) * d * 2 * 2 * (Hq + Hkv)
        if case["guided"]:
            byts += sum(n * (n + 1) for n in lens)
            S = case["top_s"]
            keys = sum(min(n, S) * (min(n, S) + 1) // 2 + max(0, n - S) * S for n in lens)
        else:
            keys = sum(n * (n + 1) // 2 for n in lens)
        return {"bytes": byts, "flops": 4 * keys * Hq * d}
    sh = _Shape(case)
    es = 4 if sh.dtype == "fp32" else 2
    per_block = sum(math.prod(s) for _, s, _, _ in sh.tensors())
    used = len({sh.map[l] for l in sh.tl})
    caches = sh.T * (used * sh.Ds * (1 if sh.act else 2) + len(sh.tl) * sh.Dt * 2)
    k = sh.K or sh.E
    if sh.kind == "bt":
        d, f, P = BT_WIDTH, BT_FFN, sh.Hs
        row = 2 * d * sh.ds + 8 * d * d + 4 * P * d + 4 * d * f
        per = sh.N * (2 * sh.Ds * sh.E + k * (P * row + 2 * P * d * sh.Dt))
        flops = 2 * sh.T * per
    else:
        Dm = sh.act or sh.Dt
        per = 2 * sh.Ds * sh.E + k * (2 * sh.Ds * sh.H + 2 * sh.H * Dm)
        per += 4 * Dm * sh.Dt if sh.act else 0
        flops = sh.T * per * sh.blocks()
    return {"bytes": es * (caches + sh.blocks() * per_block), "flops": flops}


def tolerance(case):
    """About four times the error measured against ``exact`` (relative; largest)."""
    if case["kind"] == "replay":   # 2.1e-3; 0.04: bf16 operands and probabilities, fp32 sums
        return {"rel": 0.01, "max": 0.2}
    if case.get("dtype") == "fp32":   # 1.1e-6; 8e-6
        return {"rel": 5e-6, "max": 4e-5}
    # Routed: a token whose scores tie to fp32 rounding may take either translator.
    top = {"max": 0.99} if case.get("top_k") else {}
    if case["kind"] == "bt":   # 4.7e-3; 0.07: bf16 rows between the stages of every slot
        return {"rel": 0.02, "max": 0.3, **top}
    # 1.8e-3; 0.008: fp16 hidden, bf16 output. MoT-h 2.4e-3; 0.015: bf16 activations between.
    return {"rel": 0.01, "max": 0.06, **top}


# ---------------------------------------------------------------- the same in 64 bits

def _unpack(sh, block):
    out, at = {}, 0
    for name, shape, _, _ in sh.tensors():
        n = math.prod(shape)
        out[name] = block[at:at + n].double().view(shape)
        at += n
    return out


def _gate(sh, z, w):
    """Softmax scores, zero outside the Top-K and renormalised over it (ties: lower index)."""
    g = torch.softmax(z @ w["wg"].T + w["bg"], dim=1)
    if 0 < sh.K < sh.E:
        keep = torch.sort(g, dim=1, descending=True, stable=True).indices[:, :sh.K]
        g = torch.zeros_like(g).scatter(1, keep, g.gather(1, keep))
        g = g / g.sum(1, keepdim=True)
    return g


def _tokens(sh, src, layer):
    """The real tokens of one source layer, one after another, heads flattened: [T][Ds]."""
    rows = []
    for b, n in enumerate(sh.lens):
        x = src[layer, b]
        rows.append(x[:n] if sh.act else x[:, :n].permute(1, 0, 2).reshape(n, sh.Ds))
    return torch.cat(rows).double()


def _store(sh, dst, layer, y):
    at = 0
    for b, n in enumerate(sh.lens):
        dst[layer, b, :, :n] = y[at:at + n].view(n, sh.Ht, sh.dt).permute(1, 0, 2)
        at += n


def _mixture(sh, z, w):
    g = _gate(sh, z, w)
    y = torch.zeros((z.shape[0], sh.act or sh.Dt), dtype=torch.float64, device=DEV)
    for m in range(sh.E):
        at = torch.nonzero(g[:, m]).squeeze(1)
        h = torch.nn.functional.gelu(z[at] @ w[f"w1{m}"].T + w[f"b1{m}"])
        y[at] += g[at, m:m + 1] * (h @ w[f"w2{m}"].T + w[f"b2{m}"])
    return y


def _ln(x, g, b):
    return torch.nn.functional.layer_norm(x, x.shape[-1:], g, b, 1e-5)


def _backbone(sh, zs, w, m):
    """One backbone over the window: zs [N] of [T][P][ds] -> [N] of [T][Dt]."""
    gelu, (d, na), out, h = torch.nn.functional.gelu, (BT_WIDTH, BT_HEADS), [], None
    for r, x in enumerate(zs):
        k = f"{m}_{r}"

        def heads(t):
            return t.view(t.shape[0], t.shape[1], na, d // na).transpose(1, 2)

        z = gelu(_ln(x, w[f"ling{m}"], w[f"linb{m}"]) @ w[f"win{m}"].T + w[f"bin{m}"])
        h = z if h is None else h
        hq = _ln(h, w["lqg" + k], w["lqb" + k])
        zc = _ln(z, w["lcg" + k], w["lcb" + k])
        q = heads(hq @ w["wq" + k].T + w["bq" + k])
        kk = heads(zc @ w["wk" + k].T + w["bk" + k])
        v = heads(zc @ w["wv" + k].T + w["bv" + k])
        a = torch.softmax(q @ kk.transpose(2, 3) / math.sqrt(d // na), dim=3) @ v
        ht = h + a.transpose(1, 2).reshape(h.shape) @ w["wo" + k].T + w["bo" + k]
        f = gelu(_ln(ht, w["lfg" + k], w["lfb" + k]) @ w["wf1" + k].T + w["bf1" + k])
        h = ht + f @ w["wf2" + k].T + w["bf2" + k]
        o = _ln(h.reshape(h.shape[0], -1), w[f"log{m}"], w[f"lob{m}"])
        out.append(gelu(o @ w[f"wout{m}"].T + w[f"bout{m}"]))
    return out


def _exact_bt(sh, src, blob):
    dst = [torch.zeros(sh.dst_shape(), dtype=torch.float64, device=DEV) for _ in range(2)]
    for x in (0, 1):
        w = _unpack(sh, blob[x])
        toks = [_tokens(sh, src[x], sh.map[l]) for l in sh.tl]
        g = _gate(sh, torch.cat(toks, dim=1), w)
        parts = [[] for _ in sh.tl]
        for t0 in range(0, sh.T, 4096):
            zs = [t[t0:t0 + 4096].view(-1, sh.Hs, sh.ds) for t in toks]
            ys = [_backbone(sh, zs, w, m) for m in range(sh.E)]
            for r in range(sh.N):
                parts[r].append(sum(g[t0:t0 + 4096, m:m + 1] * ys[m][r] for m in range(sh.E)))
        for l, y in zip(sh.tl, parts):
            _store(sh, dst[x], l, torch.cat(y))
    return dst


def _exact_replay(case, seed):
    (Hq, Hkv, d), lens, q, k, v, guide = _replay_inputs(case, seed)
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    G, S, scale = Hq // Hkv, case["top_s"], 1.0 / math.sqrt(d)
    for b, n in enumerate(lens):
        j = torch.arange(n, device=DEV)
        for u0 in range(0, n, 256):
            u = torch.arange(u0, min(n, u0 + 256), device=DEV)[:, None]
            allowed = j <= u
            if case["guided"]:
                # positive scores order as their bits; ties go to the lower position
                bits = guide[b, u0:u0 + u.shape[0], :n].contiguous().view(torch.int16).long()
                key = torch.where(allowed, (bits << 17) + (n - j), -1)
                top = torch.topk(key, min(S, n), dim=1).indices
                allowed = torch.zeros_like(allowed).scatter(1, top, True) & allowed
            for hk in range(Hkv):
                qq = q[b, hk * G:(hk + 1) * G, u0:u0 + u.shape[0]].double()
                s = (qq @ k[b, hk, :n].double().T) * scale
                p = torch.softmax(s.masked_fill(~allowed, -math.inf), dim=2)
                out[b, hk * G:(hk + 1) * G, u0:u0 + u.shape[0]] = p @ v[b, hk, :n].double()
    return out


def exact(case, seed):
    if work(case)["flops"] > 15e12:   # over about 20 seconds at the 64-bit rate
        return None
    if case["kind"] == "replay":
        return _exact_replay(case, seed)
    sh, src, blob = _translation_inputs(case, seed)
    if sh.kind == "bt":
        return _exact_bt(sh, src, blob)
    dst = [torch.zeros(sh.dst_shape(), dtype=torch.float64, device=DEV) for _ in range(2)]
    for i, l in enumerate(sh.tl):
        if sh.act:
            w = _unpack(sh, blob[i])
            a = _mixture(sh, _tokens(sh, src[0], sh.map[l]), w)
            _store(sh, dst[0], l, a @ w["wk"].T)
            _store(sh, dst[1], l, a @ w["wv"].T)
            continue
        for x in (0, 1):
            w = _unpack(sh, blob[2 * i + x])
            _store(sh, dst[x], l, _mixture(sh, _tokens(sh, src[x], sh.map[l]), w))
    return dst

"""The work that users of this library have it do, as cases to be timed.

Each case is one pass through the public entry points of
``paper_2608_29809_gb300.regioncache`` on the sizes of the seeded workloads
(``synth``): PixArt-alpha-shaped blocks of hidden 1152 at 256 to 16384 image
tokens, whole 28-block denoising steps, the localisation mask and the set-up
of an editing turn.  ``exact`` restates a case in float64 with plain torch.

Kinds
  mask   rc_localize_mask on a cross-attention score map
  block  rc_block_forward_region through `layers` consecutive blocks, then the
         last block's refreshed cache slot read back: H (the merged block
         output, bf16), K and V.  (The f32 rows of `hidden` hold the same
         outputs before that rounding; every stage between them rounds to
         bf16, so their last bits depend on the order of each sum.)
  turn   what an editing turn starts with: rc_set_text with the new prompt,
         then rc_localize_scores from the cached states
  step   rc_localize_mask and one denoising step of a session (a CUDA graph
         replay, or rc_step); the last block's cache slot is read back
  serve  one rc_step_batched over several sessions with ragged edit regions;
         the sessions' merged last hidden states are read back
"""
import ctypes
import math

import numpy as np
import torch

from paper_2608_29809_gb300 import regioncache as R
from paper_2608_29809_gb300 import synth

T_INDEX = 1  # the timestep slot that the cases step, of `timesteps` = 3
TIMESTEPS = 3


def _block(name, gh, gw, dirty, layers, count="device", head_dim=72, text=120):
    return {"name": name, "kind": "block", "gh": gh, "gw": gw, "dirty": dirty, "layers": layers,
            "count": count, "head_dim": head_dim, "text": text}


def listed():
    return [
        # one edit's mask at 512 px, five changed words: a call every turn,
        # all latency
        {"name": "mask_512px", "kind": "mask", "gh": 32, "gw": 32, "slices": 1, "text": 120,
         "deltas": 5, "dilation": 1},
        # a mask at 2048 px averaged over 16 heads' maps, eight changed words
        {"name": "mask_2048px_16_heads", "kind": "mask", "gh": 128, "gw": 128, "slices": 16,
         "text": 120, "deltas": 8, "dilation": 1},
        # one block of the smallest grid with a 15 % rectangle-sized edit
        _block("block_256tok", 16, 16, 39, 1, count="host"),
        # two blocks at 512 px, 13 % dirty
        _block("block_512px", 32, 32, 132, 2),
        # two blocks at 1024 px, a small (5 %) edit: weights and launches count
        _block("block_1024px_5pct", 64, 64, 201, 2),
        # two blocks at 1024 px, the headline 20 % edit
        _block("block_1024px_20pct", 64, 64, 831, 2),
        # two blocks at 1024 px with every token recomputed (the leading steps
        # of a turn)
        _block("block_1024px_dense", 64, 64, 4096, 2, count="host"),
        # one block at 2048 px, 20 % dirty: long key range
        _block("block_2048px_20pct", 128, 128, 3248, 1, count="host"),
        # a turn's start at 1024 px: the prompt's text keys for 28 blocks, then
        # the localisation scores of four changed words from the cache
        {"name": "turn_1024px", "kind": "turn", "gh": 64, "gw": 64, "layers": 28, "text": 120,
         "deltas": 4, "head_dim": 72},
        # the headline: mask and 28-block sparse step at 1024 px, 20 % dirty,
        # replayed as a CUDA graph
        {"name": "step_1024px_20pct", "kind": "step", "gh": 64, "gw": 64, "dirty": 831,
         "layers": 28, "graph": True, "head_dim": 72, "text": 120},
        # batched serving: 8 sessions at 512 px, 2 to 35 % dirty each
        {"name": "serve_8x512px", "kind": "serve", "gh": 32, "gw": 32, "items": 8, "dirty": 20,
         "dirty_most": 358, "layers": 28, "head_dim": 72, "text": 120},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["mask", "block", "block", "block", "block", "turn", "step", "serve"])
        gh, gw = _log_int(rng, 12, 128), _log_int(rng, 12, 128)
        N = gh * gw
        text = rng.choice([77, 120, 120, 120, 128])
        head_dim = rng.choice([72, 72, 72, 64])
        if kind == "mask":
            c = {"kind": kind, "gh": gh, "gw": gw, "slices": _log_int(rng, 1, 28), "text": text,
                 "deltas": _log_int(rng, 1, 24), "dilation": rng.randint(0, 3)}
        elif kind == "block":
            dirty = N if rng.random() < 0.15 else max(1, int(N * math.exp(
                rng.uniform(math.log(0.02), math.log(0.6)))))
            c = _block("", gh, gw, dirty, rng.randint(1, 2), rng.choice(["device", "host"]),
                       head_dim, text)
            del c["name"]
        elif kind == "turn":
            gh, gw = min(gh, 72), min(gw, 72)
            c = {"kind": kind, "gh": gh, "gw": gw, "layers": rng.randint(14, 28), "text": text,
                 "deltas": rng.randint(1, 8), "head_dim": head_dim}
        elif kind == "step":
            gh, gw = min(gh, 72), min(gw, 72)
            dirty = max(1, int(gh * gw * math.exp(rng.uniform(math.log(0.02), math.log(0.4)))))
            c = {"kind": kind, "gh": gh, "gw": gw, "dirty": dirty, "layers": 28,
                 "graph": rng.random() < 0.5, "head_dim": head_dim, "text": text}
        else:
            gh, gw = min(gh, 40), min(gw, 40)
            lo = max(1, int(gh * gw * rng.uniform(0.02, 0.15)))
            c = {"kind": kind, "gh": gh, "gw": gw, "items": rng.randint(2, 8), "dirty": lo,
                 "dirty_most": int(gh * gw * rng.uniform(0.16, 0.35)), "layers": 28,
                 "head_dim": head_dim, "text": text}
        # whole steps up to the rows that 8 sessions' edits have together
        rows = sum(_item_dirty(c)) if kind == "serve" else c["dirty"] if kind == "step" else 0
        if work(c)["flops"] <= most and rows <= 1512:
            return c


# ------------------------------------------------------------------- sizes
def _dims(case):
    hd = case.get("head_dim", 72)
    h = 16 * hd
    return synth.Dims(hidden=h, heads=16, mlp=4 * h, layers=case.get("layers", 1),
                      grid_h=case["gh"], grid_w=case["gw"], text_len=case["text"],
                      timesteps=TIMESTEPS)


def _item_dirty(case):
    n, lo, hi = case["items"], case["dirty"], case["dirty_most"]
    return [lo + (hi - lo) * ((5 * i) % n) // max(1, n - 1) for i in range(n)]


def _block_work(d, D, weights=True):
    """Bytes and FLOPs of one region-sparse block with D dirty tokens."""
    h, f, N, M = d.hidden, d.mlp, d.tokens, d.text_len
    clean = N - D
    b = 2 * clean * h * 2 + 3 * D * h * 2 + M * 2 * h * 2
    if weights:
        b += 2 * (6 * h * h + 2 * h * f)
    return b, D * (2 * (6 * h * h + 2 * h * f) + 4 * N * h + 4 * M * h)


def work(case):
    N = case["gh"] * case["gw"]
    if case["kind"] == "mask":
        n = N * case["deltas"] * case["slices"]
        return {"bytes": 4 * n + 5 * N, "flops": n}
    d = _dims(case)
    h, L, M = d.hidden, d.layers, d.text_len
    latent = 4 * d.in_ch * N * d.patch ** 2
    if case["kind"] == "turn":
        return {"bytes": L * (3 * h * h * 2 + N * h * 2) + M * h * 2 + N * M * 4 + latent,
                "flops": L * (4 * M * h * h + 2 * N * h * h + 2 * N * M * h)}
    if case["kind"] == "serve":
        b, fl = 0, 0
        for i, D in enumerate(_item_dirty(case)):
            bb, ff = _block_work(d, D, weights=i == 0)
            b, fl = b + L * bb + N * h * 2 + 2 * latent, fl + L * ff + 32 * N * h
        return {"bytes": b, "flops": fl}
    b, fl = _block_work(d, case["dirty"])
    if case["kind"] == "block":
        return {"bytes": L * b + 2 * 4 * case["dirty"] * h, "flops": L * fl}
    return {"bytes": L * b + N * h * 2 + 2 * latent + 3 * 4 * N, "flops": L * fl + 32 * N * h}


# ------------------------------------------------------------------ inputs
def _distance(d, seed, blobs):
    """Per blob, each token's squared distance from a random centre in the
    metric of a random ellipse, [blobs][N]."""
    rng = np.random.default_rng([seed, 17])
    ys, xs = np.meshgrid(np.arange(d.grid_h), np.arange(d.grid_w), indexing="ij")
    out = []
    for _ in range(blobs):
        cy, cx = rng.uniform(0, d.grid_h), rng.uniform(0, d.grid_w)
        ratio, th = rng.uniform(0.5, 2.0), rng.uniform(0, math.pi)
        dy, dx = ys - cy, xs - cx
        u, v = dx * math.cos(th) + dy * math.sin(th), dy * math.cos(th) - dx * math.sin(th)
        out.append((u * u / ratio + v * v * ratio).reshape(-1))
    return np.stack(out)


def _region(d, seed, dirty):
    """`dirty` tokens of one to three blobs, ascending (int64 numpy)."""
    r = _distance(d, seed, 1 + seed % 3).min(axis=0)
    return np.sort(np.argsort(r, kind="stable")[:dirty])


def _dev_i32(a):
    return torch.as_tensor(np.asarray(a, np.int32)).cuda()


def _bump_scores(d, seed, slices, deltas):
    """Softmax score maps [slices][N][M] whose delta columns have a bump."""
    rng = np.random.default_rng([seed, 23])
    ids = rng.choice(d.text_len, size=deltas, replace=False).astype(np.int32)
    dist = _distance(d, seed, deltas)
    sig = rng.uniform(1.2, 2.6, size=(deltas, 1)) * d.grid_h / 32
    bump = torch.as_tensor(6.0 * np.exp(-dist / (2 * sig * sig)), dtype=torch.float32).cuda()
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(slices, d.tokens, d.text_len, generator=g, device="cuda")
    x[:, :, torch.as_tensor(ids, dtype=torch.int64).cuda()] += bump.T
    return torch.softmax(x, dim=2), ids


def _region_scores(d, seed, idx):
    """A score map [1][N][M] whose one delta column is high exactly on idx."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.rand(1, d.tokens, d.text_len, generator=g, device="cuda")
    j = seed % d.text_len
    A[0, :, j] *= 0.4
    A[0, idx, j] = 0.6 + 0.4 * torch.rand(len(idx), generator=g, device="cuda")
    return A, np.array([j], np.int32)


def _turn_ids(d, seed, deltas):
    rng = np.random.default_rng([seed, 29])
    return rng.choice(d.text_len, deltas, replace=False).astype(np.int32)


def _mask_state(d, scores, ids, dilation):
    N = d.tokens
    return {"scores": scores, "ids": ids, "dilation": dilation, "d": d,
            "ws": torch.empty(R.rc_localize_workspace_size(N, len(ids)), dtype=torch.uint8,
                              device="cuda"),
            "mask": torch.zeros(N, dtype=torch.uint8, device="cuda"),
            "idx": torch.zeros(N, dtype=torch.int32, device="cuda"),
            "cnt": torch.zeros(1, dtype=torch.int32, device="cuda")}


def _localize(s):
    d, A = s["d"], s["scores"]
    R.rc_localize_mask(A, A.shape[0], d.tokens, A.shape[2], d.grid_h, d.grid_w, s["ids"], 0.5,
                       s["dilation"], s["mask"], s["idx"], s["cnt"], s["ws"])


def _model(d, seed, sessions=1, max_batch=1):
    m = R.Model(d, synth.make_weights(d, seed, device="cuda"), sessions=sessions,
                max_batch=max_batch)
    R.rc_set_schedule(m.ctx, *synth.ddim_tables(d.timesteps))
    for s in range(sessions):
        R.rc_set_text(m.ctx, m.cache, s, synth.make_text(d, seed + 1000 * s, "cuda"))
        for l in range(d.layers):
            R.rc_cache_fill(m.cache, s, l, T_INDEX,
                            *synth.make_cache_slice(d, seed, s, l, T_INDEX, "cuda"))
    torch.cuda.synchronize()
    return m


def _slot(d, parts=3):
    return [torch.zeros(d.tokens, d.hidden, dtype=torch.bfloat16, device="cuda")
            for _ in range(parts)]


def _mods(d, w, seed):
    return [synth.make_mod6(d, w.layers[l]["table"], seed + l) for l in range(d.layers)]


def prepare(case, seed):
    d = _dims(case)
    if case["kind"] == "mask":
        A, ids = _bump_scores(d, seed, case["slices"], case["deltas"])
        return {"kind": "mask", **_mask_state(d, A, ids, case["dilation"])}
    if case["kind"] == "block":
        m = _model(d, seed)
        idx = _region(d, seed, case["dirty"])
        x = synth.make_hidden(d, seed, "cuda")
        s = {"kind": "block", "d": d, "m": m, "x": x, "hidden": x.clone(),
             "mods": _mods(d, m.w, seed), "idx": _dev_i32(idx), "D": len(idx), "cnt": None}
        if case["count"] == "device":  # as after rc_localize_mask: the count stays there
            s["D"], s["cnt"] = -1, _dev_i32([len(idx)])
        s["slot"] = _slot(d)
        return s
    if case["kind"] == "turn":
        m = _model(d, seed)
        return {"kind": "turn", "m": m, "text": synth.make_text(d, seed + 7, "cuda"),
                "latent": synth.make_latent(d, seed, "cuda"),
                "ids": _turn_ids(d, seed, case["deltas"]),
                "scores": torch.zeros(d.tokens, d.text_len, device="cuda")}
    sched = np.full(d.timesteps, R.RC_MODE_SPARSE, np.uint8)
    if case["kind"] == "step":
        m = _model(d, seed)
        noise = synth.make_latent(d, seed, "cuda")
        s = {"kind": "step", "m": m, "noise": noise, "latent": noise.clone(), "sched": sched,
             "local": _mask_state(d, *_region_scores(d, seed, _region(d, seed, case["dirty"])), 0),
             "slot": _slot(d), "graph": None}
        if case["graph"]:
            s["graph"] = _Graph(m, s["latent"], sched, s["local"])
        return s
    n = case["items"]
    m = _model(d, seed, sessions=n, max_batch=n)
    noise = torch.stack([synth.make_latent(d, seed + i, "cuda") for i in range(n)])
    latents, items = noise.clone(), []
    for i, D in enumerate(_item_dirty(case)):
        items.append({"session": i, "latent": latents[i], "t": T_INDEX,
                      "mode": R.RC_MODE_SPARSE, "dirty_idx": _dev_i32(_region(d, seed + i, D)),
                      "D": -1, "dirty_count": _dev_i32([D])})
    return {"kind": "serve", "m": m, "noise": noise, "latents": latents, "items": items,
            "H": _slot(d, n)}


class _Graph:
    """A step's graph, given back before its model is."""

    def __init__(self, m, latent, sched, local):
        self.m = m
        self.g = ctypes.c_void_p(R.rc_step_graph_create(m.ctx, m.cache, 0, latent, T_INDEX, sched,
                                                        local["idx"], -1, local["cnt"]))

    def __del__(self):
        R.rc_graph_destroy(self.g)


# -------------------------------------------------------------------- run
def run(s):
    kind = s["kind"]
    if kind == "mask":
        _localize(s)
        return {"mask": s["mask"], "idx": s["idx"], "count": s["cnt"]}
    m = s["m"]
    if kind == "block":
        s["hidden"].copy_(s["x"])  # the caller's input rows, updated in place below
        for l, mod6 in enumerate(s["mods"]):
            R.rc_block_forward_region(m.ctx, m.cache, 0, l, T_INDEX, s["hidden"], s["idx"],
                                      s["D"], s["cnt"], mod6)
        R.rc_cache_read(m.cache, 0, s["d"].layers - 1, T_INDEX, *s["slot"])
        return s["slot"]
    if kind == "turn":
        R.rc_set_text(m.ctx, m.cache, 0, s["text"])
        R.rc_localize_scores(m.ctx, m.cache, 0, T_INDEX, s["latent"], s["ids"], s["scores"])
        return s["scores"]
    if kind == "step":
        s["latent"].copy_(s["noise"])
        lo = s["local"]
        _localize(lo)
        if s["graph"] is not None:
            R.rc_graph_launch(s["graph"].g)
        else:
            R.rc_step(m.ctx, m.cache, 0, s["latent"], T_INDEX, s["sched"], lo["idx"], -1,
                      lo["cnt"])
        R.rc_cache_read(m.cache, 0, m.dims.layers - 1, T_INDEX, *s["slot"])
        return {"latent": s["latent"], "mask": lo["mask"], "slot": s["slot"]}
    s["latents"].copy_(s["noise"])
    R.rc_step_batched(m.ctx, m.cache, s["items"])
    for it, H in zip(s["items"], s["H"]):
        R.rc_cache_read(m.cache, it["session"], m.dims.layers - 1, T_INDEX, H, None, None)
    return {"latents": s["latents"], "H": s["H"]}


# ------------------------------------------------------------------ exact
def _ln(x):
    return torch.nn.functional.layer_norm(x, x.shape[-1:], eps=1e-6)


def _lin(x, W, b):
    return torch.nn.functional.linear(x, W.double(), b.double())


def _attend(q, k, v, heads):
    hd = q.shape[1] // heads
    out = torch.empty_like(q)
    for h in range(heads):
        c = slice(h * hd, (h + 1) * hd)
        out[:, c] = torch.softmax(q[:, c] @ k[:, c].T / math.sqrt(hd), dim=1) @ v[:, c]
    return out


def _exact_block(x, idx, K, V, w, m6, text, heads):
    """Block outputs of the dirty rows x; K, V (float64 [N][h]) are updated."""
    h = x.shape[1]
    q, k, v = _lin(_ln(x) * (1 + m6[1]) + m6[0], w["W_qkv"], w["b_qkv"]).split(h, dim=1)
    K[idx], V[idx] = k, v
    x = x + m6[2] * _lin(_attend(q, K, V, heads), w["W_o"], w["b_o"])
    tk, tv = _lin(text, w["W_xkv"], w["b_xkv"]).split(h, dim=1)
    o = _attend(_lin(x, w["W_xq"], w["b_xq"]), tk, tv, heads)
    x = x + _lin(o, w["W_xo"], w["b_xo"])
    a = _lin(_ln(x) * (1 + m6[4]) + m6[3], w["W_1"], w["b_1"])
    a = torch.nn.functional.gelu(a, approximate="tanh")
    return x + m6[5] * _lin(a, w["W_2"], w["b_2"])


def _embed(d, w, latent):
    p = torch.nn.functional.unfold(latent.double()[None], d.patch, stride=d.patch)[0].T
    return _lin(p, w.glob["W_e"], w.glob["b_e"]) + w.pos.double()


def _exact_step(d, w, seed, session, text, latent, idx):
    tv, ab = synth.ddim_tables(d.timesteps)
    g, half = w.glob, d.freq_dim // 2
    om = torch.exp(-math.log(10000.0) * torch.arange(half, device="cuda",
                                                     dtype=torch.float64) / half)
    a = float(tv[T_INDEX]) * om
    f = torch.cat([torch.cos(a), torch.sin(a)])[None]
    silu = torch.nn.functional.silu
    temb = _lin(silu(_lin(f, g["W_t1"], g["b_t1"])), g["W_t2"], g["b_t2"])
    tb = _lin(silu(temb), g["W_tb"], g["b_tb"]).reshape(6, -1)
    x = _embed(d, w, latent)[idx]
    for l, wl in enumerate(w.layers):
        H, K, V = (t.double() for t in synth.make_cache_slice(d, seed, session, l, T_INDEX,
                                                              "cuda"))
        x = _exact_block(x, idx, K, V, wl, wl["table"].double() + tb, text, d.heads)
    H[idx] = x
    tf = g["table_f"].double()
    out = _lin(_ln(H) * (1 + tf[1] + temb) + tf[0] + temb, g["W_f"], g["b_f"])
    p = d.patch
    eps = out.reshape(d.grid_h, d.grid_w, p, p, d.out_ch).permute(4, 0, 2, 1, 3)
    eps = eps.reshape(d.out_ch, d.grid_h * p, d.grid_w * p)[:d.in_ch]
    at, an = float(ab[T_INDEX]), float(ab[T_INDEX + 1])
    x0 = (latent.double() - math.sqrt(1 - at) * eps) / math.sqrt(at)
    return math.sqrt(an) * x0 + math.sqrt(1 - an) * eps, [H, K, V]


def exact(case, seed):
    if case["kind"] == "mask":
        return None  # whole numbers, decided in float32 by definition
    d = _dims(case)
    w = synth.make_weights(d, seed, device="cuda")
    if case["kind"] == "block":
        idx = torch.as_tensor(_region(d, seed, case["dirty"])).cuda()
        hidden = synth.make_hidden(d, seed, "cuda").double()
        text = synth.make_text(d, seed, "cuda").double()
        for l, m6 in enumerate(_mods(d, w, seed)):
            H, K, V = (t.double() for t in synth.make_cache_slice(d, seed, 0, l, T_INDEX, "cuda"))
            x = _exact_block(hidden[idx], idx, K, V, w.layers[l], m6.double(), text, d.heads)
            hidden[idx], H[idx] = x, x
        return [H, K, V]
    if case["kind"] == "turn":
        text = synth.make_text(d, seed + 7, "cuda").double()
        latent = synth.make_latent(d, seed, "cuda")
        ids = torch.as_tensor(_turn_ids(d, seed, case["deltas"]), dtype=torch.int64).cuda()
        scores = torch.zeros(d.tokens, d.text_len, dtype=torch.float64, device="cuda")
        hd = d.head_dim
        for l, wl in enumerate(w.layers):
            x = _embed(d, w, latent) if l == 0 else H
            q = _lin(x, wl["W_xq"], wl["b_xq"])
            k = _lin(text, wl["W_xkv"], wl["b_xkv"])[:, :d.hidden]
            for h in range(d.heads):
                c = slice(h * hd, (h + 1) * hd)
                p = torch.softmax(q[:, c] @ k[:, c].T / math.sqrt(hd), dim=1)
                scores[:, ids] += p[:, ids] / (d.layers * d.heads)
            H = synth.make_cache_slice(d, seed, 0, l, T_INDEX, "cuda")[0].double()
        return scores
    if case["kind"] == "step":
        idx = torch.as_tensor(_region(d, seed, case["dirty"])).cuda()
        text = synth.make_text(d, seed, "cuda").double()
        latent, slot = _exact_step(d, w, seed, 0, text, synth.make_latent(d, seed, "cuda"), idx)
        return {"latent": latent, "mask": None, "slot": slot}
    out, last = [], []
    for i, D in enumerate(_item_dirty(case)):
        text = synth.make_text(d, seed + 1000 * i, "cuda").double()
        idx = torch.as_tensor(_region(d, seed + i, D)).cuda()
        latent, slot = _exact_step(d, w, seed, i, text, synth.make_latent(d, seed + i, "cuda"),
                                   idx)
        out.append(latent)
        last.append(slot[0])
    return {"latents": torch.stack(out), "H": last}

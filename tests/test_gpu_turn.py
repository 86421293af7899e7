"""A turn's start (rc_set_text, rc_localize_scores) at the edges of its tiles:
partial token tiles, one to 128 text tokens, both head sizes, more layers than
one launch takes, against the same definition in float64 torch."""
import math

import numpy as np
import pytest
import torch

from paper_2608_29809_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache
    return regioncache


def _scores64(d, w, text, latent, caches, ids):
    lin = torch.nn.functional.linear
    p = torch.nn.functional.unfold(latent.double()[None], d.patch, stride=d.patch)[0].T
    x = lin(p, w.glob["W_e"].double(), w.glob["b_e"].double()) + w.pos.double()
    out = torch.zeros(d.tokens, d.text_len, dtype=torch.float64, device="cuda")
    dh = d.head_dim
    for l, wl in enumerate(w.layers):
        q = lin(x, wl["W_xq"].double(), wl["b_xq"].double())
        k = lin(text.double(), wl["W_xkv"].double(), wl["b_xkv"].double())[:, :d.hidden]
        for h in range(d.heads):
            c = slice(h * dh, (h + 1) * dh)
            out[:, ids] += torch.softmax(q[:, c] @ k[:, c].T / math.sqrt(dh), dim=1)[:, ids]
        x = caches[l].double()
    return out / (d.layers * d.heads)


@pytest.mark.parametrize("grid,heads,dh,M,layers,n", [
    ((1, 1), 2, 64, 1, 1, 1), ((3, 43), 2, 64, 5, 33, 3), ((16, 16), 16, 72, 128, 2, 8),
    ((7, 37), 16, 72, 77, 3, 2), ((64, 64), 16, 64, 120, 2, 4)])
def test_scores_from_the_cache_at_tile_edges(R, grid, heads, dh, M, layers, n):
    d = synth.Dims(hidden=heads * dh, heads=heads, mlp=256, layers=layers, grid_h=grid[0],
                   grid_w=grid[1], text_len=M, timesteps=2)
    seed = 501 + M
    m = R.Model(d, synth.make_weights(d, seed, device="cuda"), sessions=2)
    try:
        R.rc_set_schedule(m.ctx, *synth.ddim_tables(d.timesteps))
        text = synth.make_text(d, seed, "cuda")
        latent = synth.make_latent(d, seed, "cuda")
        R.rc_set_text(m.ctx, m.cache, 1, text)
        caches = []
        for l in range(layers):
            H, K, V = synth.make_cache_slice(d, seed, 1, l, 1, "cuda")
            R.rc_cache_fill(m.cache, 1, l, 1, H, K, V)
            caches.append(H)
        ids = np.random.default_rng(seed).choice(M, n, replace=False).astype(np.int32)
        got = torch.full((d.tokens, M), 7.0, device="cuda")
        R.rc_localize_scores(m.ctx, m.cache, 1, 1, latent, ids, got)
        R.rc_sync(m.ctx)
        cols = torch.as_tensor(ids, dtype=torch.int64).cuda()
        want = _scores64(d, m.w, text, latent, caches, cols)
        assert (got.double()[want == 0] == 0).all()
        # K and G are rounded to bf16 (2^-9 each): a logit of RMS about 1 is
        # off by about 2^-8 of it, a probability by as much of itself
        err = (got.double() - want).abs()
        assert float((err / want.clamp_min(1e-30))[want > 0].max()) <= 2.0 ** -5
        assert float(err.norm() / want.norm()) <= 2.0 ** -8
    finally:
        m.close()

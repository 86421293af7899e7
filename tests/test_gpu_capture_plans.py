"""Localisation scores of texts longer than the one-pass attention takes (129 to
448 tokens), captured by the general attention kernel with units of one query
tile and of two, against the same definition in float64 torch."""
import numpy as np
import pytest
import torch

from paper_2608_29809_gb300 import synth
from tests.test_gpu_turn import _scores64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache
    return regioncache


@pytest.mark.parametrize("grid,heads,dh,M,n", [
    ((13, 23), 16, 72, 129, 1), ((32, 32), 16, 72, 200, 8), ((16, 16), 16, 64, 300, 5),
    ((1, 3), 2, 64, 161, 2), ((64, 72), 16, 72, 448, 8)])
def test_captured_scores_of_long_texts(R, grid, heads, dh, M, n):
    d = synth.Dims(hidden=heads * dh, heads=heads, mlp=256, layers=2, grid_h=grid[0],
                   grid_w=grid[1], text_len=M, timesteps=2)
    seed = 601 + M
    m = R.Model(d, synth.make_weights(d, seed, device="cuda"))
    try:
        R.rc_set_schedule(m.ctx, *synth.ddim_tables(d.timesteps))
        text = synth.make_text(d, seed, "cuda")
        latent = synth.make_latent(d, seed, "cuda")
        R.rc_set_text(m.ctx, m.cache, 0, text)
        caches = []
        for l in range(d.layers):
            H, K, V = synth.make_cache_slice(d, seed, 0, l, 1, "cuda")
            R.rc_cache_fill(m.cache, 0, l, 1, H, K, V)
            caches.append(H)
        ids = np.random.default_rng(seed).choice(M, n, replace=False).astype(np.int32)
        got = torch.full((d.tokens, M), 7.0, device="cuda")
        R.rc_localize_scores(m.ctx, m.cache, 0, 1, latent, ids, got)
        R.rc_sync(m.ctx)
        want = _scores64(d, m.w, text, latent, caches, torch.as_tensor(ids, dtype=torch.int64).cuda())
        assert (got.double()[want == 0] == 0).all()
        # q and K are rounded to bf16 (2^-9 each): a logit of RMS about 1 is off
        # by about 2^-8 of it, a probability by as much of itself
        err = (got.double() - want).abs()
        assert float((err / want.clamp_min(1e-30))[want > 0].max()) <= 2.0 ** -5
        assert float(err.norm() / want.norm()) <= 2.0 ** -8
    finally:
        m.close()

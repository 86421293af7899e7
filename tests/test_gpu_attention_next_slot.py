"""Self-attention through the cache where the last key block reaches past a
layer's last token: the rows behind a layer's values are the next layer's H
rows, and whatever they hold (NaN here) stays out of the result when the token
count is a multiple of 16."""
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


# 80-key blocks: 16, 32, 48 and 64 keys in the last one, and whole blocks only
@pytest.mark.parametrize("gh,gw", [(16, 16), (12, 16), (13, 16), (14, 16), (15, 16)])
@pytest.mark.parametrize("head_dim", [72, 64])
def test_rows_of_the_next_layer_stay_out(R, gh, gw, head_dim):
    d = synth.Dims(hidden=16 * head_dim, heads=16, mlp=512, layers=2, grid_h=gh, grid_w=gw,
                   timesteps=1)
    w = synth.make_weights(d, 5, device="cuda")
    m = R.Model(d, w)
    try:
        R.rc_set_deterministic(m.ctx, True)
        R.rc_set_text(m.ctx, m.cache, 0, synth.make_text(d, 5, "cuda"))
        x = synth.make_hidden(d, 5, "cuda")
        mod6 = synth.make_mod6(d, w.layers[0]["table"], 5)
        slices = [synth.make_cache_slice(d, 5, 0, l, 0, "cuda") for l in range(2)]
        for dirty in (40, 150, d.tokens):  # one query tile, two, every token
            idx = torch.from_numpy(np.sort(np.random.default_rng(dirty).choice(
                d.tokens, dirty, replace=False)).astype(np.int32)).cuda()
            outs = []
            for behind in (slices[1][0], torch.full_like(slices[1][0], float("nan"))):
                R.rc_cache_fill(m.cache, 0, 0, 0, *slices[0])
                R.rc_cache_fill(m.cache, 0, 1, 0, behind, *slices[1][1:])
                hidden = x.clone()
                R.rc_block_forward_region(m.ctx, m.cache, 0, 0, 0, hidden, idx, dirty, None, mod6)
                R.rc_sync(m.ctx)
                outs.append(hidden)
            assert bool(torch.isfinite(outs[0]).all())
            assert torch.equal(outs[0], outs[1])
    finally:
        m.close()

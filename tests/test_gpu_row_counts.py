"""One block at row counts around the 128-row tiles of its GEMMs, where the
split of a matrix's k range changes (up to eight parts for one row tile) and
where the folded cross-attention's CTAs take one or two (tile, head) units,
against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from paper_2608_29809_gb300 import synth
from tests.gpu_cases import LATENT_REL_L2, Problem, block_close, rel_l2
from tests.test_gpu_batched import Sessions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def problem():
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache as R
    p = Problem(R, dataclasses.replace(synth.ONE_BLOCK_256, grid_h=48, grid_w=48), 4321)
    yield p
    p.close()


@pytest.mark.parametrize("rows", [1, 128, 129, 256, 385, 640, 897, 1217, 2047])
def test_block_at_row_tile_edges(problem, rows):
    p, d = problem, problem.d
    idx = np.sort(np.random.default_rng(rows).choice(d.tokens, rows, replace=False))
    x = synth.make_hidden(d, p.seed)
    mod6 = synth.make_mod6(d, p.model.w.layers[0]["table"].cpu(), p.seed)
    H, K, V = synth.make_cache_slice(d, p.seed, 0, 0, 0)
    p.R.rc_cache_fill(p.model.cache, 0, 0, 0, H.cuda(), K.cuda(), V.cuda())
    hidden = x.clone().cuda()
    idx_d = torch.from_numpy(idx.astype(np.int32)).cuda()
    p.R.rc_block_forward_region(p.model.ctx, p.model.cache, 0, 0, 0, hidden, idx_d, rows, None,
                                mod6.cuda())
    p.R.rc_sync(p.model.ctx)
    cache, out = O.region_block(O.to64(x)[idx], idx, p.cache64[(0, 0)], p.layers64[0],
                                O.to64(mod6), p.tkv64[0], d.heads)
    block_close(hidden.cpu().numpy()[idx], out, "block output rows")
    after = p.read_slot(0, 0)
    for k in "HKV":
        block_close(after[k][idx], cache[k][idx], f"cache {k}")


def test_batch_rows_of_neighbouring_items():
    """Items whose rows meet within one CTA's share of the LayerNorm rows."""
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache as R
    d = dataclasses.replace(synth.PIXART_512, layers=1, timesteps=2)
    S = Sessions(R, d, 4322, 3, max_batch=3)
    try:
        items, idxs, lats = [], [], []
        for s, rows in enumerate((1, 457, 333)):
            S.fill(s, s % 2)
            idx = np.sort(np.random.default_rng(s).choice(d.tokens, rows, replace=False))
            lat = synth.make_latent(d, 4322 + s)
            items.append(dict(session=s, latent=lat.clone().cuda(), t=s % 2, mode=O.MODE_SPARSE,
                              dirty_idx=torch.from_numpy(idx.astype(np.int32)).cuda(), D=rows,
                              dirty_count=None))
            idxs.append(idx)
            lats.append(lat)
        R.rc_step_batched(S.model.ctx, S.model.cache, items)
        R.rc_sync(S.model.ctx)
        for s, it in enumerate(items):
            want, _, cache = S.oracle(s, O.to64(lats[s]), s % 2, O.MODE_SPARSE, idxs[s])
            assert rel_l2(it["latent"].cpu().double().numpy(), want) <= LATENT_REL_L2, s
            sl = S.read(s, 0, s % 2)
            for k in "HKV":
                block_close(sl[k][idxs[s]], cache[0][k][idxs[s]], f"session {s} {k}")
    finally:
        S.close()

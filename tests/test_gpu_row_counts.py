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
from tests.gpu_cases import Problem, block_close

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

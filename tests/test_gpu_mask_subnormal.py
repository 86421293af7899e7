"""The localisation mask on score columns whose range is so small that its
reciprocal is not a float32 (below 2^-128), or only just is: the threshold is
the correctly rounded quotient all the same, bit for bit as in the oracle, in
the one-launch and the two-launch form."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2608_29809_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache
    return regioncache


@pytest.mark.parametrize("gh,gw,S,n", [(16, 16, 1, 1), (16, 16, 1, 3), (37, 53, 2, 2),
                                       (96, 96, 1, 1), (61, 64, 1, 3)])
@pytest.mark.parametrize("thr", [0.5, 0.3, 1.5, 0.0, -0.5])
@pytest.mark.parametrize("lo,rng", [(0.0, 1e-42), (0.0, 1e-39), (0.0, 2e-39), (1e-42, 1e-39),
                                    (-2e-39, 2.9e-39), (0.0, 2.0 ** -128), (0.0, 3e-39),
                                    (0.0, 1.1e-38), (0.0, 2e-45)])
def test_threshold_of_subnormal_ranges(R, gh, gw, S, n, thr, lo, rng):
    N, M = gh * gw, 6
    r = np.random.default_rng(synth.tensor_seed(31, gh, gw, S, n))
    # eighths of the range in the delta columns, thresholds among them
    A = (lo + rng * r.integers(0, 9, (S, N, M)) / 8).astype(np.float32)
    ids = r.choice(M, n, replace=False).astype(np.int32)
    want, idx = O.localize_mask(A, ids, gh, gw, thr, 0)
    ws = torch.empty(R.rc_localize_workspace_size(N, n), dtype=torch.uint8, device="cuda")
    mask = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
    out = torch.full((N,), -5, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    R.rc_localize_mask(torch.from_numpy(A).cuda(), S, N, M, gh, gw, ids, thr, 0, mask, out, cnt,
                       ws)
    torch.cuda.synchronize()
    assert int(cnt.item()) == len(idx)
    assert np.array_equal(mask.cpu().numpy(), want)
    assert np.array_equal(out.cpu().numpy()[:len(idx)], idx)

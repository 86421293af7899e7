"""The localisation mask at the sizes where its one- and two-launch forms and
the token split over the cluster can go wrong, bit for bit against the oracle:
one token, part of a word, uneven shares, the largest grid, one row, wide
dilations, many slices and delta tokens, values on the threshold."""
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


@pytest.mark.parametrize("gh,gw,S,M,n,thr,dil,grid_values", [
    (1, 1, 1, 3, 2, 0.5, 1, True), (1, 31, 1, 4, 3, 0.5, 2, True), (3, 11, 2, 5, 5, 0.25, 0, True),
    (16, 16, 1, 120, 32, 0.5, 1, True), (37, 53, 1, 77, 4, 0.9, 3, False),
    (37, 53, 9, 20, 20, 0.5, 8, True), (64, 64, 1, 120, 2, 0.5, 1, False),
    (64, 64, 1, 120, 64, 0.999, 1, False), (1, 16384, 1, 8, 1, 0.75, 8, True),
    (16384, 1, 3, 8, 4, 0.75, 8, True), (128, 128, 8, 12, 8, 0.9, 1, False),
    (127, 129, 17, 12, 5, 1.0, 0, True), (25, 41, 1, 9, 3, -0.5, 1, False),
    (25, 41, 1, 9, 9, 1.5, 1, False), (60, 61, 1, 9, 3, 0.0, 1, False)])
def test_mask_matches_the_oracle(R, gh, gw, S, M, n, thr, dil, grid_values):
    N = gh * gw
    rng = np.random.default_rng(synth.tensor_seed(9, gh, gw, S, n))
    A = rng.random((S, N, M), np.float32)
    if grid_values:  # eighths: many values lie on the threshold exactly
        A = np.round(A * 8).astype(np.float32) / np.float32(8)
    ids = rng.choice(M, n, replace=False).astype(np.int32)
    if n > 2:
        A[:, :, ids[0]] = 0.25                      # a constant column
        A[-1, N // 2, ids[1]] = np.inf              # a dropped column
        A[:, :, ids[2]] *= np.float32(1e-38)        # subnormal range
    if n > 3:
        A[:, :, ids[3]] = np.where(A[:, :, ids[3]] > 0.5, 3e38, -3e38) / np.float32(S)
    with np.errstate(over="ignore", invalid="ignore"):
        want, idx = O.localize_mask(A, ids, gh, gw, thr, dil)
    ws = torch.empty(R.rc_localize_workspace_size(N, n), dtype=torch.uint8, device="cuda")
    mask = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
    out = torch.full((N,), -5, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    R.rc_localize_mask(torch.from_numpy(A).cuda(), S, N, M, gh, gw, ids, thr, dil, mask, out, cnt,
                       ws)
    torch.cuda.synchronize()
    assert int(cnt.item()) == len(idx)
    assert np.array_equal(mask.cpu().numpy(), want)
    assert np.array_equal(out.cpu().numpy()[:len(idx)], idx)
    assert (out[len(idx):] == -5).all()

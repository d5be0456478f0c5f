"""GPU parity of the XBF GEMM where its tiling changes: row blocks in twos with
one left over, twos in the full waves and ones in the last, fewer tiles than SMs,
rows short of a block, and k blocks fewer than ring stages."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from tests.helpers import REDUCED_TOL, rel_err_planes
from tests.test_xbf_gpu import hermitian_vis, planes, run_xbf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,K,C,n", [
    (5, 4, 101, 64),       # 13 row blocks (the last short) x 16: all in twos, one left over
    (4, 2, 70, 128),       # 5 row blocks x 64: 50 blocks in twos, 14 one by one
    (30, 1, 64, 128),      # 2 row blocks x 64, 15 k blocks: fewer tiles than SMs
    (1, 1, 33, 256),       # one pair, one k block, 2 row blocks x 256
])
def test_tilings(hai, S, K, C, n):
    rng = np.random.default_rng(S * n + C)
    cell, lam = 19.0, 3.0
    pos = rng.uniform(-n * cell / 3, n * cell / 3, (S, 2))
    dirs = rng.uniform(-0.1, 0.1, (K, 2))
    vis = hermitian_vis(rng, K, C, S)
    want = planes(O.station_xbf(n, pos, lam, cell, dirs, vis.astype(np.int64)))
    ctx = hai.hai_create(0)
    try:
        got, _ = run_xbf(hai, ctx, pos, lam, cell, n, dirs, vis, hai.HAI_XBF_ALL_PAIRS)
        assert rel_err_planes(got, want).max() < REDUCED_TOL
        img = torch.from_numpy(got).cuda()
        twice, _ = run_xbf(hai, ctx, pos, lam, cell, n, dirs, vis, hai.HAI_XBF_ALL_PAIRS, img, 1)
        assert np.array_equal(twice, 2 * got)
    finally:
        hai.hai_destroy(ctx)

"""XBF GEMM with an odd number of row blocks and a Phi block that outgrows L2
between a pixel block's twos and its last one: row blocks go one by one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_odd_row_blocks_of_a_long_sum_equal_the_even_ones(hai):
    # 128 channels of 4 planes: 4 row blocks in twos; the first 96: 3, one by one
    S, n, cell = 256, 256, 19.0
    rng = np.random.default_rng(4)
    pos = rng.uniform(-0.38 * n, 0.38 * n, (S, 2)) * cell
    vis = torch.randint(-1000, 1000, (128, S * (S + 1) // 2, 2, 2, 2), device="cuda", dtype=torch.int32)
    img = {C: torch.full((C, 4, n, n), float("nan"), device="cuda") for C in (128, 96)}
    ctx = hai.hai_create(0)
    lay = hai.hai_xbf_layout_create(ctx, pos, 3.0, cell, n, None, hai.HAI_XBF_OFFGRID_PAIRS, 128, hai.HAI_PREC_FP16)
    try:
        assert hai.hai_xbf_layout_info(lay)[0] > 7000
        for C, out in img.items():
            hai.hai_xbf_station_image(ctx, lay, vis[:C].contiguous(), C, out)
            hai.hai_sync(ctx)
        assert torch.isfinite(img[128]).all() and torch.equal(img[96], img[128][:96])
    finally:
        hai.hai_xbf_layout_destroy(lay)
        hai.hai_destroy(ctx)

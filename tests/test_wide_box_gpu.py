"""Tensor-core EPIC at 512^2 with kernel boxes of 129 to 256 columns (5 to 8 k
blocks in stage 1, whose DFT operand then comes in blocks of half as many l_x),
against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_17804_gb300 import inputs as I
from tests.helpers import BF16_SPLIT_TOL, BF16_TOL, FP32_TOL, REDUCED_TOL, SPLIT_PIXEL_TOL, frob_err_planes, pixel_err_planes

pytestmark = pytest.mark.gpu

TOL = {"FP16": (REDUCED_TOL, REDUCED_TOL), "BF16": (BF16_TOL, BF16_TOL), "FP16_SPLIT": (FP32_TOL, SPLIT_PIXEL_TOL),
       "BF16_SPLIT": (BF16_SPLIT_TOL, BF16_SPLIT_TOL)}


@pytest.mark.parametrize("pname", list(TOL))
@pytest.mark.parametrize("bw,bh,ne,k,C,T", [
    (128, 40, 300, 1, 1, 3),       # the last box of the other form: 4 k blocks
    (129, 128, 500, 1, 2, 3),      # 5 k blocks, the fifth with one column
    (200, 17, 400, 3, 1, 5),       # 7, several entries a cell
    (256, 128, 900, 1, 3, 40),     # 8: the widest box; items split between CTAs
])
def test_wide_boxes_match_oracle(hai, pname, bw, bh, ne, k, C, T):
    n = 512
    rng = np.random.default_rng(bw)
    lo = np.stack([rng.integers(0, bw - k + 1, ne), rng.integers(0, bh - k + 1, ne)], 1)
    lo[0], lo[-1] = (0, 0), (bw - k, bh - k)
    anchors = (lo + [n // 2 - bw // 2, n // 2 - bh // 2]).astype(np.int32)
    taps = rng.standard_normal((ne, k, k, 2)).astype(np.float32)
    volt = I.random_voltages((C, T, 2, ne, 2), seed=bw + T)
    want = O.epic_image(n, anchors, taps, volt.numpy())
    ctx = hai.hai_create(0)
    lay = hai.hai_layout_create(ctx, anchors, taps, n, 2)
    try:
        img = torch.full((C, 4, n, n), float("nan"), device="cuda")
        for rep in (1, 2):
            hai.hai_epic_image(ctx, lay, volt.cuda(), C, T, getattr(hai, "HAI_PREC_" + pname), img, rep - 1)
            hai.hai_sync(ctx)
            got = img.cpu().numpy()
            assert frob_err_planes(got, rep * want).max() < TOL[pname][0]
            assert pixel_err_planes(got, rep * want).max() < TOL[pname][1]
    finally:
        hai.hai_layout_destroy(lay)
        hai.hai_destroy(ctx)

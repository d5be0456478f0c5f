"""GPU parity of the FP32 EPIC path at 512^2, two polarisations, where its forms
and batches change (box of at most 128 cells or wider, at most 128 rows or
taller, one unit tap or several entries a cell, channels in whole batches and
left over), against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_17804_gb300 import inputs as I
from tests.helpers import FP32_TOL, rel_err_planes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bw,bh,k,ne,C,T", [
    (128, 128, 1, 300, 8, 3),      # an uneven last batch of channels
    (129, 128, 1, 90, 2, 1),       # one column beyond the pruned row transform
    (128, 129, 3, 90, 3, 2),       # one row beyond the warp column transform
    (61, 127, 3, 400, 1, 5),       # several entries a cell, rows short of a group of 8
    (512, 512, 2, 50, 1, 2),       # the whole grid
    (1, 1, 1, 1, 1, 1),
])
def test_forms_and_batches(hai, bw, bh, k, ne, C, T):
    n, P = 512, 2
    rng = np.random.default_rng(1000 * bw + bh)
    x0, y0 = n - bw, (n - bh) // 2
    ax = rng.integers(x0, x0 + bw - k + 1, ne)
    ay = rng.integers(y0, y0 + bh - k + 1, ne)
    if ne > 1:
        ax[0], ay[0], ax[-1], ay[-1] = x0, y0, x0 + bw - k, y0 + bh - k
    anchors = np.stack([ax, ay], 1).astype(np.int32)
    taps = rng.standard_normal((ne, k, k, 2)).astype(np.float32)
    volt = I.random_voltages((C, T, P, ne, 2), seed=bw + bh)
    want = O.epic_image(n, anchors, taps, volt.numpy())
    ctx = hai.hai_create(0)
    lay = hai.hai_layout_create(ctx, anchors, taps, n, P)
    try:
        v = volt.cuda()
        img = torch.full(want.shape, float("nan"), device="cuda")
        for rep in (1, 2):
            hai.hai_epic_image(ctx, lay, v, C, T, hai.HAI_PREC_FP32, img, rep - 1)
            hai.hai_sync(ctx)
            assert rel_err_planes(img.cpu().numpy(), rep * want).max() < FP32_TOL
    finally:
        hai.hai_layout_destroy(lay)
        hai.hai_destroy(ctx)

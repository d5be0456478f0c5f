"""Tensor-core EPIC at the limit of shared memory: the largest gather table of
complex taps that fits beside the voltages at 64^2."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_17804_gb300 import inputs as I
from tests.helpers import REDUCED_TOL, rel_err_planes

pytestmark = pytest.mark.gpu


def test_complex_table_at_the_limit(hai):
    # 1,496 elements dealt to 97 cells (41 of 16, 56 of 15): with its 32 bytes of
    # warp ranges the table of 1,984 entries took the last byte of 227 KB
    n, ne, cells, C, T = 64, 1496, 97, 2, 5
    rng = np.random.default_rng(5)
    spot = np.stack(np.divmod(rng.permutation(30 * 30)[:cells], 30), 1)
    anchors = (n // 4 + spot[np.arange(ne) % cells]).astype(np.int32)
    taps = rng.standard_normal((ne, 1, 1, 2)).astype(np.float32)
    volt = I.random_voltages((C, T, 2, ne, 2), seed=9)
    want = O.epic_image(n, anchors, taps, volt.numpy())
    ctx = hai.hai_create(0)
    lay = hai.hai_layout_create(ctx, anchors, taps, n, 2)
    try:
        img = torch.full((C, 4, n, n), float("nan"), device="cuda")
        hai.hai_epic_image(ctx, lay, volt.cuda(), C, T, hai.HAI_PREC_FP16, img)
        hai.hai_sync(ctx)
        assert rel_err_planes(img.cpu().numpy(), want).max() < REDUCED_TOL
    finally:
        hai.hai_layout_destroy(lay)
        hai.hai_destroy(ctx)

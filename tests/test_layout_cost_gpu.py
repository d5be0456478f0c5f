"""What creating a layout costs: the gather table's order takes time linear in its
entries, also where one cell holds them all."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ne,span", [(64, 16000, 1), (128, 20000, 2)])
def test_many_elements_on_a_few_cells(hai, n, ne, span):
    """1.3 and 7.8 ms (7 of them the 128^2 scratch); quadratic: 275 and 161 ms."""
    rng = np.random.default_rng(ne)
    anchors = (n // 2 + rng.integers(0, span, (ne, 2))).astype(np.int32)
    taps = np.ones((ne, 1, 1, 2), np.float32)
    taps[..., 1] = 0
    ctx = hai.hai_create(0)
    try:
        best = float("inf")
        for _ in range(4):
            t = time.perf_counter()
            lay = hai.hai_layout_create(ctx, anchors, taps, n, 2)
            best = min(best, time.perf_counter() - t)
            hai.hai_layout_destroy(lay)
        assert best < 0.04
    finally:
        hai.hai_destroy(ctx)

"""A call that is refused after its checks leaves the profile readable."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 64])
def test_refused_call_leaves_no_open_record(hai, n):
    ctx = hai.hai_create(0)
    ne = 200_000                                     # two samples of it exceed shared memory
    taps = np.ones((ne, 1, 1, 2), np.float32)
    big = hai.hai_layout_create(ctx, np.full((ne, 2), n // 2, np.int32), taps, n, 1)
    small = hai.hai_layout_create(ctx, np.full((3, 2), n // 2, np.int32), taps[:3], n, 1)
    try:
        img = torch.zeros((1, 1, n, n), device="cuda")
        hai.hai_profile_enable(ctx)
        with pytest.raises(hai.HaiError) as e:
            hai.hai_epic_image(ctx, big, torch.zeros((1, 2, 1, ne, 2), dtype=torch.int8, device="cuda"), 1, 2,
                               hai.HAI_PREC_FP32, img)
        assert "UNSUPPORTED" in str(e.value)
        assert hai.hai_profile_read(ctx)[1] == 0
        hai.hai_epic_image(ctx, small, torch.ones((1, 2, 1, 3, 2), dtype=torch.int8, device="cuda"), 1, 2,
                           hai.HAI_PREC_FP32, img)
        hai.hai_sync(ctx)
        assert hai.hai_profile_read(ctx)[1] == 1
    finally:
        hai.hai_layout_destroy(big)
        hai.hai_layout_destroy(small)
        hai.hai_destroy(ctx)

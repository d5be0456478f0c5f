"""Kernels whose warpgroups move registers refuse to run on a build with fewer
registers a thread than their shares add up to (injected on the host: such a
launch would wait without end)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

UNSUPPORTED = 4


def test_too_few_registers_are_refused(hai, monkeypatch):
    ctx = hai.hai_create(0)
    S, C, T, K, N = 2, 1, 16, 8, 16
    volt = torch.ones((S, C, T, 2, N, 2), dtype=torch.int8, device="cuda")
    w = torch.ones((S, K, 2, N, 2), dtype=torch.int8, device="cuda")
    beams = torch.zeros((S, C, T, K, 2, 2), dtype=torch.int32, device="cuda")
    lays = {}
    for n in (32, 64, 128):
        taps = np.zeros((4, 1, 1, 2), np.float32)
        taps[..., 0] = 1
        lays[n] = hai.hai_layout_create(ctx, np.full((4, 2), n // 2, np.int32), taps, n, 2)
    v = torch.ones((1, 4, 2, 4, 2), dtype=torch.int8, device="cuda")
    try:
        monkeypatch.setenv("HAI_FAULT", "registers")
        with pytest.raises(hai.HaiError) as e:
            hai.hai_beamform(ctx, volt, w, S, C, T, K, N, 2, -1, beams)
        assert e.value.status == UNSUPPORTED and "registers" in str(e.value)
        for n, lay in lays.items():
            img = torch.zeros((1, 4, n, n), device="cuda")
            with pytest.raises(hai.HaiError) as e:
                hai.hai_epic_image(ctx, lay, v, 1, 4, hai.HAI_PREC_FP16, img)
            assert e.value.status == UNSUPPORTED and "registers" in str(e.value)
        monkeypatch.delenv("HAI_FAULT")
        hai.hai_beamform(ctx, volt, w, S, C, T, K, N, 2, -1, beams)
        hai.hai_sync(ctx)
        # conj(1 + i) (1 + i) = 2 for each of N elements
        assert torch.equal(beams[..., 0], torch.full_like(beams[..., 0], 2 * N)) and not beams[..., 1].any()
    finally:
        for lay in lays.values():
            hai.hai_layout_destroy(lay)
        hai.hai_destroy(ctx)

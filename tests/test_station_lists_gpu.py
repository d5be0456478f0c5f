"""Gather lists of the inter-station XFFT: units of several chunks against the
FP64 oracle and bit for bit on repeat, what creating a large layout costs, and the time of a short
array."""
import time

import numpy as np
import pytest
import torch

from oracle import oracle as O
from tests.helpers import FP32_TOL, rel_err_planes

pytestmark = pytest.mark.gpu


def hermitian_vis(rng, K, C, S):
    vis = rng.integers(-2**16, 2**16, (K, C, S * (S + 1) // 2, 2, 2, 2)).astype(np.int32)
    auto = [a * (a + 1) // 2 + a for a in range(S)]
    vis[:, :, auto, 0, 0, 1] = 0
    vis[:, :, auto, 1, 1, 1] = 0
    vis[:, :, auto, 1, 0, 0] = vis[:, :, auto, 0, 1, 0]
    vis[:, :, auto, 1, 0, 1] = -vis[:, :, auto, 0, 1, 1]
    return vis


@pytest.mark.parametrize("n,S,K,C,spread", [
    (64, 80, 2, 3, 2.0),       # 3,240 pairs around the corner of four tiles: several chunks a unit, 6 images
    (16, 50, 1, 5, 3.0),       # one tile, which is its own mirror
    (128, 60, 1, 1, 20.0),     # one image
    (256, 70, 3, 3, 0.0),      # every station on one spot: one cell holds every pair and every mirror
])
def test_units_of_several_chunks(hai, n, S, K, C, spread):
    rng = np.random.default_rng(n + S)
    cell, lam = 19.0, 3.0
    pos = rng.uniform(-spread, spread, (S, 2)) * cell / 2
    dirs = rng.uniform(-0.3, 0.3, (K, 2))
    vis = hermitian_vis(rng, K, C, S)
    want, dropped = O.station_xfft(n, pos, lam, cell, dirs, vis)
    want = np.stack([want[:, :, 0, 0].real, want[:, :, 1, 1].real, want[:, :, 0, 1].real, want[:, :, 0, 1].imag], 2)
    ctx = hai.hai_create(0)
    lay = hai.hai_vis_layout_create(ctx, pos, lam, cell, n, dirs)
    try:
        assert hai.hai_vis_layout_offgrid(lay) == dropped
        v = torch.from_numpy(vis).cuda()
        got = []
        for _ in range(3):
            img = torch.full((K * C, 4, n, n), float("nan"), device="cuda")
            hai.hai_xfft_station_image(ctx, lay, v, C, img)
            hai.hai_sync(ctx)
            got.append(img.cpu().numpy())
        assert rel_err_planes(got[0], want.reshape(K * C, 4, n, n)).max() < FP32_TOL
        assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    finally:
        hai.hai_vis_layout_destroy(lay)
        hai.hai_destroy(ctx)


def test_creating_a_large_layout_is_quick(hai):
    """2,048 stations (2.1 million pairs): 45 ms; building the lists on the host,
    pair by pair in several passes, took 560 ms."""
    rng = np.random.default_rng(1)
    pos = rng.uniform(-51.0, 51.0, (2048, 2)) * 19.0
    ctx = hai.hai_create(0)
    best = float("inf")
    for _ in range(3):
        t = time.perf_counter()
        lay = hai.hai_vis_layout_create(ctx, pos, 3.0, 19.0, 256, None)
        best = min(best, time.perf_counter() - t)
        hai.hai_vis_layout_destroy(lay)
    hai.hai_destroy(ctx)
    assert best < 0.2


def test_a_short_array_is_not_slow(hai):
    """256 stations within 57 m, 128 images: every pair on 49 cells.  0.28 ms;
    with one thread a cell 4.4 ms (by shared-memory atomics 1.1 ms)."""
    rng = np.random.default_rng(2)
    S, C, n = 256, 128, 256
    pos = rng.uniform(-1.5, 1.5, (S, 2)) * 19.0
    vis = torch.randint(-1000, 1000, (C, S * (S + 1) // 2, 2, 2, 2), device="cuda", dtype=torch.int32)
    img = torch.empty((C, 4, n, n), device="cuda")
    ctx = hai.hai_create(0)
    lay = hai.hai_vis_layout_create(ctx, pos, 3.0, 19.0, n, None)
    try:
        best = float("inf")
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            hai.hai_xfft_station_image(ctx, lay, vis, C, img)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        assert best < 1.0
    finally:
        hai.hai_vis_layout_destroy(lay)
        hai.hai_destroy(ctx)

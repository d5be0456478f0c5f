"""GPU parity of the inter-station XFFT imager at the grid sides, image counts,
buffer alignments and pair layouts where its kernels change form, against the
FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from tests.helpers import FP32_TOL, rel_err_planes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(hai):
    c = hai.hai_create(0)
    yield c
    hai.hai_destroy(c)


@pytest.mark.parametrize("n,S,K,C,extent,off_v,off_i", [
    (128, 40, 2, 3, 0.45, 0, 0),
    (256, 33, 1, 33, 0.30, 0, 0),      # one image more than a warp
    (64, 17, 3, 11, 0.60, 2, 1),       # pairs dropped; vis off 16 bytes, images off 4 bytes
    (32, 9, 1, 1, 0.45, 2, 0),
    (16, 6, 5, 13, 0.45, 0, 3),        # images of several beams in one warp
    (256, 1, 1, 2, 0.0, 0, 0),         # the auto alone
    (128, 24, 1, 2, -1.0, 0, 0),       # every station on a whole cell, many pairs on one cell
])
def test_station_xfft_forms(hai, ctx, n, S, K, C, extent, off_v, off_i):
    rng = np.random.default_rng(n + S + K)
    cell, lam = 19.0, 3.0
    if extent < 0:
        pos = rng.integers(-3, 4, (S, 2)) * cell
    else:
        pos = rng.uniform(-extent, extent, (S, 2)) * n * cell
    dirs = rng.uniform(-0.3, 0.3, (K, 2))
    nbl = S * (S + 1) // 2
    vis = rng.integers(-2**20, 2**20, (K, C, nbl, 2, 2, 2)).astype(np.int32)
    auto = [a * (a + 1) // 2 + a for a in range(S)]
    vis[:, :, auto, 0, 0, 1] = 0
    vis[:, :, auto, 1, 1, 1] = 0
    vis[:, :, auto, 1, 0, 0] = vis[:, :, auto, 0, 1, 0]
    vis[:, :, auto, 1, 0, 1] = -vis[:, :, auto, 0, 1, 1]
    want, dropped = O.station_xfft(n, pos, lam, cell, dirs, vis)
    want = np.stack([want[:, :, 0, 0].real, want[:, :, 1, 1].real, want[:, :, 0, 1].real, want[:, :, 0, 1].imag], 2)
    lay = hai.hai_vis_layout_create(ctx, pos, lam, cell, n, dirs)
    try:
        assert hai.hai_vis_layout_offgrid(lay) == dropped
        vb = torch.zeros(off_v + vis.size, dtype=torch.int32, device="cuda")
        vb[off_v:] = torch.from_numpy(vis).cuda().view(-1)
        ib = torch.full((off_i + want.size,), float("nan"), device="cuda")
        for _ in range(2):
            hai.hai_xfft_station_image(ctx, lay, vb[off_v:], C, ib[off_i:])
            hai.hai_sync(ctx)
            got = ib[off_i:].cpu().numpy().reshape(K * C, 4, n, n)
            assert rel_err_planes(got, want.reshape(K * C, 4, n, n)).max() < FP32_TOL
            first = got if _ == 0 else first
        assert np.array_equal(got, first) or rel_err_planes(got, first.astype(np.float64)).max() < FP32_TOL
    finally:
        hai.hai_vis_layout_destroy(lay)

"""GPU parity of the FP32 EPIC kernels of the 16^2 and 32^2 grids and of the
partial-image reduction, at the sizes where their phases, forms and splits
change, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_17804_gb300 import inputs as I
from tests.helpers import FP32_TOL, rel_err_planes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(hai):
    c = hai.hai_create(0)
    yield c
    hai.hai_destroy(c)


@pytest.mark.parametrize("n,P,bw,bh,ne,C,T,off", [
    (32, 1, 16, 16, 64, 1, 1024, 0),     # the usual box, many partial images of one channel
    (32, 2, 16, 16, 40, 3, 41, 1),       # ranges over two channels, buffers off 16 (volt) and 4 (img) bytes
    (32, 2, 32, 32, 200, 2, 9, 0),       # the whole grid
    (32, 2, 17, 15, 7, 160, 3, 0),       # one CTA per channel, 28-byte samples, phases of 3 of 4 samples
    (32, 1, 15, 17, 3, 5, 1, 3),         # one sample per channel, 6-byte samples
    (32, 2, 16, 16, 3000, 2, 6, 0),      # table in global memory
    (32, 2, 16, 16, 7000, 1, 5, 0),      # voltages too large for the phase: the general kernel
    (16, 1, 8, 8, 5, 2, 77, 0),
    (16, 2, 16, 16, 33, 170, 17, 1),     # 8-sample phases with one left over
    (16, 2, 9, 3, 1, 1, 8, 0),
])
def test_small_grid_forms(hai, ctx, n, P, bw, bh, ne, C, T, off):
    k = min(3, bw, bh)
    rng = np.random.default_rng(1000 * n + 100 * bw + ne)
    x0, y0 = n - bw, (n - bh) // 2
    ax = rng.integers(x0, x0 + bw - k + 1, ne)
    ay = rng.integers(y0, y0 + bh - k + 1, ne)
    if ne > 1:
        ax[0], ay[0], ax[-1], ay[-1] = x0, y0, x0 + bw - k, y0 + bh - k
    anchors = np.stack([ax, ay], 1).astype(np.int32)
    taps = rng.standard_normal((ne, k, k, 2)).astype(np.float32)
    volt = I.random_voltages((C, T, P, ne, 2), seed=bw + bh + ne)
    want = O.epic_image(n, anchors, taps, volt.numpy())
    lay = hai.hai_layout_create(ctx, anchors, taps, n, P)
    try:
        # `off` complex values into a larger buffer: 2 off bytes past 16-byte alignment
        vb = torch.empty(2 * off + volt.numel(), dtype=torch.int8, device="cuda")
        v = vb[2 * off:]
        v.copy_(volt.reshape(-1))
        ib = torch.full((off + want.size,), float("nan"), device="cuda")
        img = ib[off:]
        for rep in (1, 2):
            hai.hai_epic_image(ctx, lay, v, C, T, hai.HAI_PREC_FP32, img, rep - 1)
            hai.hai_sync(ctx)
            assert rel_err_planes(img.cpu().numpy().reshape(want.shape), rep * want).max() < FP32_TOL
    finally:
        hai.hai_layout_destroy(lay)

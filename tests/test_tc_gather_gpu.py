"""GPU parity of the tensor-core EPIC kernels of the 32^2, 64^2 and 128^2 grids
where their gridding and staging change form (odd element counts, buffers off 4
and 16 bytes, real and complex taps, zero weights, cells with very uneven lists),
against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_17804_gb300 import inputs as I
from tests.helpers import BF16_SPLIT_TOL, BF16_TOL, REDUCED_TOL, rel_err_planes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(hai):
    c = hai.hai_create(0)
    yield c
    hai.hai_destroy(c)


@pytest.mark.parametrize("n,ne,k,C,T,cplx,off,prec", [
    (64, 37, 3, 3, 7, False, 1, "FP16"),       # odd element count, volt off 4 bytes, a ragged step
    (64, 38, 3, 2, 5, False, 1, "FP16"),       # even count off 4 bytes: element by element
    (64, 38, 3, 160, 3, True, 2, "FP16"),      # even count on 4 bytes, one CTA per channel
    (64, 1, 1, 1, 1, False, 0, "BF16"),
    (64, 300, 2, 2, 9, False, 0, "FP16_SPLIT"),
    (32, 21, 3, 5, 11, True, 1, "BF16_SPLIT"),
    (32, 50, 3, 2, 6, False, 0, "FP16"),
    (128, 41, 1, 2, 5, True, 1, "FP16"),       # one tap, complex; odd count
    (128, 90, 3, 40, 3, False, 2, "BF16"),     # more channels than clusters
    (128, 400, 5, 1, 33, False, 0, "FP16"),
])
def test_tc_gather_forms(hai, ctx, n, ne, k, C, T, cplx, off, prec):
    rng = np.random.default_rng(1000 * n + ne)
    # half of the elements on a few cells, the rest over the box
    x0, y0 = n // 4 + 1, n // 4
    lo = rng.integers(0, n // 2 - k + 1, (ne, 2))
    lo[: ne // 2] = lo[: ne // 2] % 3 + 2
    anchors = (lo + [x0, y0]).astype(np.int32)
    anchors[:, 0] = np.minimum(anchors[:, 0], x0 + n // 2 - k)
    taps = rng.standard_normal((ne, k, k, 2)).astype(np.float32)
    if not cplx:
        taps[..., 1] = 0
    if ne > 30:
        taps[5:9] = 0                           # elements switched off
    volt = I.random_voltages((C, T, 2, ne, 2), seed=ne)
    want = O.epic_image(n, anchors, taps, volt.numpy())
    tol = {"FP16": REDUCED_TOL, "BF16": BF16_TOL, "FP16_SPLIT": REDUCED_TOL, "BF16_SPLIT": BF16_SPLIT_TOL}[prec]
    lay = hai.hai_layout_create(ctx, anchors, taps, n, 2)
    try:
        vb = torch.empty(2 * off + volt.numel(), dtype=torch.int8, device="cuda")
        v = vb[2 * off:]
        v.copy_(volt.reshape(-1))
        img = torch.full((C, 4, n, n), float("nan"), device="cuda")
        for rep in (1, 2):
            hai.hai_epic_image(ctx, lay, v, C, T, getattr(hai, "HAI_PREC_" + prec), img, rep - 1)
            hai.hai_sync(ctx)
            assert rel_err_planes(img.cpu().numpy(), rep * want).max() < tol
    finally:
        hai.hai_layout_destroy(lay)

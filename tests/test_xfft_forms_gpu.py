"""GPU parity of the correlator + FFT imager over kernel sides, tap types,
channel counts and buffer alignments where its gridding changes form, against
the FP64 oracle."""
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


@pytest.mark.parametrize("n,P,ne,k,C,cplx,off_v,off_i", [
    (64, 2, 40, 3, 33, False, 0, 0),     # one channel more than a warp
    (64, 2, 23, 5, 2, True, 2, 1),       # complex taps; vis off 16 bytes, images off 4
    (64, 1, 90, 1, 3, False, 0, 0),      # one tap, one pol
    (32, 2, 30, 2, 40, True, 0, 3),
    (32, 1, 17, 3, 1, True, 2, 0),
    (16, 2, 7, 15, 2, False, 0, 0),      # lags wrap round the grid
    (16, 1, 1, 9, 5, True, 0, 0),        # one element: its auto alone
    (64, 2, 130, 3, 1, False, 0, 0),     # many records on the patches around zero lag
])
def test_xfft_forms(hai, ctx, n, P, ne, k, C, cplx, off_v, off_i):
    rng = np.random.default_rng(n + ne + k)
    anchors = rng.integers(0, n - k + 1, (ne, 2)).astype(np.int32)
    if ne == 130:
        anchors = (anchors // 8 + 24).astype(np.int32)
    taps = rng.standard_normal((ne, k, k, 2)).astype(np.float32)
    if not cplx:
        taps[..., 1] = 0
    nbl = ne * (ne + 1) // 2
    vis = rng.integers(-2**18, 2**18, (C, nbl, P, P, 2)).astype(np.int32)    # autos' imaginary parts included
    want = O.xfft_as_epic_planes(O.xfft_image(n, anchors, taps, vis))
    lay = hai.hai_layout_create(ctx, anchors, taps, n, P)
    try:
        vb = torch.zeros(off_v + vis.size, dtype=torch.int32, device="cuda")
        vb[off_v:] = torch.from_numpy(vis).cuda().view(-1)
        ib = torch.full((off_i + want.size,), float("nan"), device="cuda")
        for rep in (1, 2):
            hai.hai_xfft_image(ctx, lay, vb[off_v:], C, ib[off_i:], rep - 1)
            hai.hai_sync(ctx)
            got = ib[off_i:].cpu().numpy().reshape(want.shape)
            assert rel_err_planes(got, rep * want).max() < FP32_TOL
    finally:
        hai.hai_layout_destroy(lay)

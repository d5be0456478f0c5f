"""GPU parity of the beamformer where its producers' order changes: fewer chunks
a unit than ring slots, a station change at every unit or within a block's
range, element and sample remainders, weights off 16 bytes: bit-exact."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_17804_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,C,T,K,N,P,off", [
    (400, 1, 3, 8, 8, 1, 0),       # one chunk a unit, a new station at every unit
    (500, 1, 1, 8, 72, 2, 2),      # four chunks, weights 2 bytes off
    (311, 1, 129, 8, 136, 1, 6),   # three chunks, two tiles a station
    (37, 9, 130, 16, 200, 2, 0),   # eight chunks, stations end within a block's range
    (1, 1, 1, 64, 64, 1, 0),       # one unit, most beams
])
def test_orders_bit_exact(hai, S, C, T, K, N, P, off):
    volt = I.random_voltages((S, C, T, P, N, 2), seed=S + N)
    w = I.random_voltages((S, K, P, N, 2), seed=K + N, lo=-128)
    want = O.beamform(volt.numpy(), w.numpy())
    ctx = hai.hai_create(0)
    try:
        buf = torch.empty(off + w.numel(), dtype=torch.int8, device="cuda")
        wd = buf[off:]
        wd.copy_(w.reshape(-1))
        beams = torch.full((S, C, T, K, P, 2), 99, dtype=torch.int32, device="cuda")
        hai.hai_beamform(ctx, volt.cuda(), wd, S, C, T, K, N, P, -1, beams, None)
        hai.hai_sync(ctx)
        assert np.array_equal(beams.cpu().numpy().astype(np.int64), want)
    finally:
        hai.hai_destroy(ctx)

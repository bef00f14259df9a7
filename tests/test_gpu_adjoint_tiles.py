"""The FP32 position adjoint on staged tiles against the oracle's adjoint where its sizes can go
wrong: the shortest line, remainders of the four-face blocks, lines at the switch from 128 to 64
columns a tile and at the longest that fits, partial tiles, both directions, whole-cell shifts;
on rough lines, which take every source of the limited value.  Tolerance: that of one FP32 sweep
(FP32 rounding away from flipped limiter branches, at most 2e-4 of the entries on them)."""
import numpy as np
import pytest

import oracle as O
from paper_2110_15867_gb300 import inputs as I
from test_gpu_adjoint import _compare, _dt_for, _lib, _rough_velocity_f

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfl", [0.8, 2.6])
@pytest.mark.parametrize("n,nu", [
    ((6, 7, 8), (4, 4, 4)),     # z: 64 columns a row; y: 512 columns, 128 a tile
    ((9, 6, 11), (4, 8, 12)),   # z: three tiles of 128
    ((37, 38, 6), (4, 4, 20)),  # 320 columns: the last tile of 128 half empty
    ((110, 4, 6), (4, 4, 4)),   # the longest line on tiles of 64 (x); y: lines of 4, one per thread
    ((116, 6, 4), (4, 4, 4)),   # too long for the tiles (x)
])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_position_adjoint_tiles(axis, n, nu, cfl):
    B = _lib()
    f0 = _rough_velocity_f(n, nu, np.float32)
    lam0 = np.random.default_rng(3).standard_normal(f0.shape).astype(np.float32)
    g = O.grid(n, nu, V=5.0)
    dt = _dt_for(g, axis, I.fourier_potential(n, seed=11), cfl)
    ref = lam0.astype(np.float64)
    O.sweep_adjoint(g, f0.astype(np.float64), ref, axis, dt, 1.0)
    f_in, lam = torch.from_numpy(f0).cuda(), torch.from_numpy(lam0).cuda()
    v = B.Vlasov(torch.zeros_like(f_in), V=5.0)
    v.sweep_adjoint(f_in, lam, axis, dt, 1.0)
    v.status()
    assert torch.equal(f_in.cpu(), torch.from_numpy(f0))
    _compare(lam.cpu().numpy(), ref, False, "axis %d lambda" % axis, axis=axis)
    v.close()

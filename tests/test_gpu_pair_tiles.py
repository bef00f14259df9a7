"""FP32 staged tiles of any line length, two lines per thread: bit for bit the streamed sweep, for
position lines with every remainder of the 4-face blocks and short to long rings, rows of
columns that do not fill the last tile, u_z lines whose signs mix within a warp, and u_x lines;
and against the FP64 oracle (relative L1 <= 1e-6, L_inf <= 1e-4 of the largest value)."""
import numpy as np
import pytest

import oracle as O
from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [((4, 5, 6), (8, 12, 20)), ((7, 9, 10), (12, 8, 12)), ((11, 13, 4), (20, 12, 4)), ((32, 6, 33), (8, 8, 8)),
          ((5, 47, 4), (24, 4, 28)), ((100, 4, 4), (8, 4, 12)), ((4, 4, 90), (40, 12, 12)), ((9, 8, 8), (128, 12, 12)),
          ((5, 4, 9), (8, 8, 12)), ((8, 7, 10), (16, 8, 12))]  # y lines of 4 and 7 with both signs in a warp


@pytest.mark.parametrize("n,nu", SHAPES)
def test_tiles_equal_the_streamed_sweep(n, nu):
    from paper_2110_15867_gb300 import binding as B
    B.load()
    V = 5.0
    f0 = I.initial_f(I.gaussian_field(n, 0.05, seed=41), I.fermi_dirac(nu, V), np.float32)
    phi32 = I.fourier_potential(n, seed=42).astype(np.float32)
    g = O.grid(n, nu, V=V)
    phi = torch.from_numpy(phi32).cuda()
    for ax in (0, 1, 2, 3):
        dt = 0.8 / O.max_abs_nu(g, ax, 1.0, 1.0, phi32.astype(np.float64))
        ref = f0.astype(np.float64)
        O.sweep(g, ref, ax, dt, 1.0, phi32.astype(np.float64))
        out = []
        for tiles in (True, False):
            f = torch.from_numpy(f0).cuda()
            v = B.Vlasov(f, V=V)
            v.set_position_tiles(tiles)
            v.sweep(ax, dt, 1.0, phi)
            v.status()
            v.close()
            out.append(f)
        assert torch.equal(out[0], out[1]), ax
        err = np.abs(out[0].cpu().numpy().astype(np.float64) - ref)
        assert err.sum() <= 1e-6 * np.abs(ref).sum() and err.max() <= 1e-4 * np.abs(ref).max(), ax

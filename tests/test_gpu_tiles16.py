"""16-bit staged tiles (two lines per thread) over the shapes their run-time sizes have to get
right: u_z lines of every accepted length (256 columns start inside a line for 24, 40 and
48), position lines with every remainder of the 4-face blocks, lines of the shortest and of
nearly the longest kind, u_x lines that the register-line kernel does not take.

Each sweep against the FP64 oracle's sweep of the same decoded input, with the codec bound
of the other 16-bit tests: relative L1 <= 2^-8 (BF16) / 2^-11 (FP16) + 1e-6, L_inf <= 1.5 x
twice that.  The tiles draw their own rounding streams: codes equal to the streamed sweep's
would show that the tiles did not run.
"""
import numpy as np
import pytest

import oracle as O
from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (n, nu): n_uz 16, 24, 40, 48, 32; position lines of 4..9, 13, 18, 35, 90 cells
SHAPES = [((9, 5, 6), (16, 16, 16)), ((4, 13, 7), (16, 16, 24)), ((18, 4, 8), (8, 16, 40)),
          ((5, 35, 4), (16, 4, 48)), ((90, 4, 5), (8, 32, 32)), ((4, 4, 6), (24, 32, 32)), ((4, 5, 4), (40, 16, 48))]


@pytest.mark.parametrize("fmt", ["bf16", "f16"])
@pytest.mark.parametrize("n,nu", SHAPES)
def test_sweeps_against_the_oracle(n, nu, fmt):
    from paper_2110_15867_gb300 import binding as B
    B.load()
    V = 5.0
    bound = {"bf16": 2.0 ** -8, "f16": 2.0 ** -11}[fmt]
    f0 = I.initial_f(I.gaussian_field(n, 0.05, seed=21), I.fermi_dirac(nu, V), np.float64)
    phi_np = I.fourier_potential(n, seed=22)
    g = O.grid(n, nu, V=V)
    phi = torch.from_numpy(phi_np.astype(np.float32)).cuda()
    phi64 = phi.cpu().numpy().astype(np.float64)
    codes0, scale0 = B.encode_lines(torch.from_numpy(f0).cuda(), {"bf16": torch.bfloat16, "f16": torch.float16}[fmt])
    axes = [0, 1, 2] + ([3] if nu[0] in (24, 40) else [])
    for ax in axes:
        dt = 0.8 / O.max_abs_nu(g, ax, 1.0, 0.9, phi64)
        ref = B.decode_lines(codes0, scale0).cpu().numpy()
        O.sweep(g, ref, ax, dt, 0.9, phi64)
        got = {}
        for tiles in (True, False):
            codes, scale = codes0.clone(), scale0.clone()
            v = B.Vlasov(codes, V=V, scale=scale)
            v.set_position_tiles(tiles)
            v.sweep(ax, dt, 0.9, phi)
            v.status()
            out = B.decode_lines(codes, scale).cpu().numpy()
            v.close()
            err = np.abs(out - ref)
            rl1, rinf = err.sum() / np.abs(ref).sum(), err.max() / np.abs(ref).max()
            assert rl1 <= bound + 1e-6 and rinf <= 1.5 * (2 * bound + 1e-6), (ax, tiles, rl1, rinf)
            assert torch.equal(scale, scale0)
            got[tiles] = codes
        assert not torch.equal(got[True], got[False]), ax

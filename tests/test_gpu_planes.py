"""D_uy and D_uz over staged (cell, j_x) planes of any size (FP32), one at a time and in one pass
of a kick, against the FP64 oracle: shortest and longest lines, rows whose length in 16-byte
units is odd and even, planes that do not fill a block and blocks that cross spatial cells
with different signs of the Courant number.  Tolerances of the per-sweep parity tests:
relative L1 <= 1e-6, L_inf <= 1e-4 of the largest value; a kick three times that.  The pass
of a kick equals the separate sweeps bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [((4, 5, 4), (4, 4, 4)), ((5, 4, 5), (8, 12, 20)), ((4, 4, 5), (12, 28, 20)), ((4, 4, 4), (4, 128, 8)),
          ((4, 4, 4), (4, 8, 72)), ((4, 4, 4), (4, 100, 68)), ((6, 5, 4), (24, 24, 24)), ((4, 4, 4), (8, 40, 40)),
          ((4, 5, 4), (4, 12, 32)), ((4, 5, 4), (20, 16, 16))]


@pytest.mark.parametrize("n,nu", SHAPES)
def test_planes(n, nu):
    from paper_2110_15867_gb300 import binding as B
    B.load()
    V = 5.0
    f0 = I.initial_f(I.gaussian_field(n, 0.05, seed=31), I.fermi_dirac(nu, V), np.float32)
    phi32 = I.fourier_potential(n, seed=32).astype(np.float32)
    phi64 = phi32.astype(np.float64)
    g = O.grid(n, nu, V=V)
    phi = torch.from_numpy(phi32).cuda()

    def close(f, ref, times):
        err = np.abs(f.cpu().numpy().astype(np.float64) - ref)
        assert err.sum() <= times * 1e-6 * np.abs(ref).sum() and err.max() <= times * 1e-4 * np.abs(ref).max()

    for ax in (4, 5):
        dt = 0.8 / O.max_abs_nu(g, ax, 1.0, 1.0, phi64)
        ref = f0.astype(np.float64)
        O.sweep(g, ref, ax, dt, 1.0, phi64)
        f = torch.from_numpy(f0).cuda()
        v = B.Vlasov(f, V=V)
        v.sweep(ax, dt, 1.0, phi)
        v.status()
        v.close()
        close(f, ref, 1)
    dt = 0.8 / max(O.max_abs_nu(g, ax, 1.0, 1.0, phi64) for ax in (3, 4, 5))
    ref = f0.astype(np.float64)
    for ax in (3, 4, 5):
        O.sweep(g, ref, ax, dt, 1.0, phi64)
    out = []
    for mode in (1, 0):
        f = torch.from_numpy(f0).cuda()
        v = B.Vlasov(f, V=V)
        v.set_fused_kick(mode)
        v.kick(dt, phi)
        v.status()
        v.close()
        close(f, ref, 3)
        out.append(f)
    assert torch.equal(out[0], out[1])


def test_rows_of_more_than_72_cells_are_refused():
    from paper_2110_15867_gb300 import binding as B
    B.load()
    with pytest.raises(B.VlasovError, match="axis 5"):
        B.Vlasov(torch.zeros((4, 4, 4, 4, 4, 76), device="cuda"), V=5.0)
    # and leave no error behind for the next call
    codes, scale = B.encode_lines(torch.rand((5, 16), device="cuda"), torch.bfloat16)
    assert (scale > 0).all()

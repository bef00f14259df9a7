"""Chained launches (a small grid's kernels may start while the one before still runs): many
steps queued without a wait, on grids below and above the size up to which launches are
chained, give the bits of the same steps with a synchronisation after each call, and work on
another stream ordered by events sees whole results."""
import numpy as np
import pytest

from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nu,dtype", [((8, 8, 8), (16, 16, 16), "f32"), ((6, 5, 7), (20, 24, 28), "f32"),
                                        ((8, 8, 8), (16, 16, 16), "bf16"), ((8, 6, 5), (8, 8, 8), "f64"),
                                        ((20, 20, 20), (16, 16, 16), "f32")])
def test_queued_steps_equal_synchronised_steps(n, nu, dtype):
    from paper_2110_15867_gb300 import binding as B
    B.load()
    f0 = I.initial_f(I.gaussian_field(n, 0.05, seed=51), I.fermi_dirac(nu, 5.0), np.float64)
    bg = torch.rand(n, dtype=torch.float64, device="cuda")
    out = []
    for wait in (True, False):
        f, scale = torch.from_numpy(f0).cuda(), None
        if dtype == "f32":
            f = f.float()
        elif dtype == "bf16":
            f, scale = B.encode_lines(f, torch.bfloat16)
        v = B.Vlasov(f, V=5.0, scale=scale)
        phi = torch.from_numpy(I.fourier_potential(n, seed=52).astype(np.float32)).cuda()
        phi2, rho = torch.empty_like(phi), torch.empty(n, dtype=torch.float64, device="cuda")
        side, copy = torch.cuda.Stream(), torch.empty_like(f)
        for _ in range(12):
            v.step(0.0004, 0.55, 0.56, phi, rho_bg=bg, phi_next=phi2, rho_nu=rho)
            phi, phi2 = phi2, phi
            if wait:
                torch.cuda.synchronize()
        done = torch.cuda.Event()
        done.record()
        side.wait_event(done)
        with torch.cuda.stream(side):
            copy.copy_(f)
        torch.cuda.synchronize()
        v.status()
        v.close()
        out.append((copy, phi, rho))
    for a, b in zip(*out):
        assert torch.equal(a, b)

"""Chained launches (a small grid's kernels may start while the one before still runs): many
steps queued without a wait, on grids below and above the size up to which launches are
chained, against the same steps made of single calls, and work on another stream ordered by events
sees whole results.

In the reference a kernel that started before the one ahead of it had finished would read the same
values all the same: every sweep is a call of its own with a synchronisation before and after it,
and calls of more than one kernel (the constants of a velocity sweep and the sweep, the five
launches of Poisson) are made twice, the first time on a scratch f, so that the arrays between their
kernels already hold what the second call writes there.  (FP32 and FP64; the moment is taken by its own
kernel.  A 16-bit kick draws streams by the number of sweeps before it, so its steps are compared
with the same steps, synchronised one by one.)"""
import numpy as np
import pytest

from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _step_by_calls(B, v, dt, a_half, a_full, phi, bg, phi2, rho):
    sync = torch.cuda.synchronize

    def kick(p):
        for ax in (3, 4, 5):
            scratch = v.f.clone()
            B.vlasov_set_f(v.ctx, scratch.data_ptr())
            v.sweep(ax, 0.5 * dt, 1.0, p)
            sync()
            B.vlasov_set_f(v.ctx, v.f.data_ptr())
            v.sweep(ax, 0.5 * dt, 1.0, p)
            sync()

    kick(phi)
    for ax in (2, 1, 0):
        v.sweep(ax, dt, a_half)
        sync()
    v.moment(rho)
    sync()
    for _ in range(2):
        v.poisson(rho, a_full, rho_bg=bg, phi=phi2)
        sync()
    kick(phi2)


@pytest.mark.parametrize("n,nu,dtype", [((8, 8, 8), (16, 16, 16), "f32"), ((6, 5, 7), (20, 24, 28), "f32"),
                                        ((8, 8, 8), (16, 16, 16), "bf16"), ((8, 6, 5), (8, 8, 8), "f64"),
                                        ((20, 20, 20), (16, 16, 16), "f32")])
def test_queued_steps_equal_single_calls(n, nu, dtype):
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
        v.set_fused_moment(False)
        phi = torch.from_numpy(I.fourier_potential(n, seed=52).astype(np.float32)).cuda()
        phi2, rho = torch.empty_like(phi), torch.empty(n, dtype=torch.float64, device="cuda")
        side, copy = torch.cuda.Stream(), torch.empty_like(f)
        for _ in range(12):
            if wait and dtype != "bf16":
                _step_by_calls(B, v, 0.0004, 0.55, 0.56, phi, bg, phi2, rho)
            else:
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

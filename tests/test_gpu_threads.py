"""Host threads, a context and a stream each, whose grids need different amounts of shared memory of
the same kernels: every call succeeds, and the results are those of one thread."""
import threading

import numpy as np
import pytest

from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# kernels of run-time sizes: pair tiles, whole-cell tiles, planes, adjoint tiles (FP32); streamed, whole-cell
# and transposing sweeps (FP64); the tiles of 16-bit codes
GRIDS = {"f32": (((12, 4, 5), (12, 8, 12)), ((5, 100, 6), (24, 20, 28))),
         "f64": (((6, 4, 5), (8, 8, 8)), ((40, 5, 4), (12, 8, 20))),
         "bf16": (((6, 4, 5), (8, 32, 32)), ((60, 4, 4), (24, 32, 32)))}


def _work(n, nu, dtype, calls, out, k):
    from paper_2110_15867_gb300 import binding as B
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            f, scale = torch.from_numpy(I.initial_f(I.gaussian_field(n, 0.05, seed=3), I.fermi_dirac(nu, 5.0), np.float64)).cuda(), None
            if dtype == "f32":
                f = f.float()
            elif dtype == "bf16":
                f, scale = B.encode_lines(f, torch.bfloat16)
            lam = torch.ones_like(f)
            v = B.Vlasov(f, V=5.0, scale=scale)
            phi = torch.from_numpy(I.fourier_potential(n, seed=4).astype(np.float32)).cuda()
            for i in range(calls):
                for ax in range(3):
                    v.sweep(ax, 0.1 / n[ax] / 5.0, 1.0)
                    if dtype != "bf16":
                        v.sweep(ax, 1.1 / n[ax] / 5.0, 1.0)
                v.kick(0.0005, phi)
                if dtype == "f32":
                    v.sweep_adjoint(f, lam, i % 3, 0.1 / n[i % 3] / 5.0, 1.0)
            v.status()
            torch.cuda.current_stream().synchronize()
            v.close()
            out[k] = f
    except Exception as e:  # noqa: BLE001 (shown by the caller)
        out[k] = e


@pytest.mark.parametrize("dtype", ["f32", "f64", "bf16"])
def test_two_threads(dtype):
    from paper_2110_15867_gb300 import binding as B
    B.load()
    got, ref, calls = [None, None], [None, None], 300
    threads = [threading.Thread(target=_work, args=g + (dtype, calls, got, k)) for k, g in enumerate(GRIDS[dtype])]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k, g in enumerate(GRIDS[dtype]):
        if isinstance(got[k], Exception):
            raise got[k]
        _work(*g, dtype, calls, ref, k)
        assert torch.equal(got[k], ref[k]), k


def test_short_calls_of_four_threads():
    # a limit that one thread set between another's set and launch failed 5 to 10 % of these
    from paper_2110_15867_gb300 import binding as B
    B.load()
    failed = []

    def work(n, nu):
        with torch.cuda.stream(torch.cuda.Stream()):
            v = B.Vlasov(torch.rand(n + nu, device="cuda"), V=5.0)
            dt = 0.1 / n[0] / 5.0
            try:
                for _ in range(5000):
                    B.vlasov_sweep(v.ctx, 0, dt, 1.0, None)
            except B.VlasovError as e:
                failed.append((n, str(e)))
            torch.cuda.current_stream().synchronize()
            v.close()

    threads = [threading.Thread(target=work, args=a) for a in (((12, 4, 4), (4, 8, 8)), ((100, 4, 4), (4, 4, 8)),
                                                               ((60, 4, 4), (4, 4, 8)), ((16, 4, 5), (4, 4, 8)))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed

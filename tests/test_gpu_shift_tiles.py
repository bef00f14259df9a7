"""FP32 position sweeps that shift whole cells on staged tiles, two lines per thread: bit for bit
the sweep of one line per thread, at the sizes where the tiles can go wrong (shortest and longest
line, partial tiles) and where the two lines of a pair shift by different numbers of cells, by as
many as a thread can hold back, and by more (lines marched in place and rotated); and, both, against
the FP64 oracle (relative L1 <= 1e-6, L_inf <= 1e-4 of the largest value)."""
import numpy as np
import pytest

import oracle as O
from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfl", [1.3, 8.9, 14.2])
@pytest.mark.parametrize("axis,n,nu", [
    (2, (4, 5, 12), (8, 4, 20)),  # the shortest line; adjacent columns of different shift
    (0, (47, 4, 5), (4, 8, 12)),      # partial last tile
    (1, (4, 110, 4), (8, 4, 4)),      # the longest line
    (0, (7, 4, 5), (20, 8, 12)),      # too short for the tiles: one line per thread both times
    (2, (4, 5, 130), (8, 12, 8)),     # too long for them
])
def test_whole_cell_tiles_match_one_line_per_thread(axis, n, nu, cfl):
    from paper_2110_15867_gb300 import binding as B
    rng = np.random.default_rng(5)
    f0 = I.initial_f(I.gaussian_field(n, 0.01, seed=2), I.fermi_dirac(nu, 5.0), np.float32)
    f0 *= (0.2 + rng.random(f0.shape)).astype(np.float32)
    out = []
    for tiles in (True, False):
        f = torch.from_numpy(f0).cuda()
        v = B.Vlasov(f, V=5.0)
        v.set_position_tiles(tiles)
        v.sweep(axis, cfl / n[axis] / 5.0, 1.0)
        v.status()
        out.append(f.cpu())
        v.close()
    assert torch.equal(out[0], out[1])
    assert not torch.equal(out[0], torch.from_numpy(f0))
    ref = f0.astype(np.float64)
    O.sweep(O.grid(n, nu, V=5.0), ref, axis, cfl / n[axis] / 5.0, 1.0, np.zeros(n))
    err = np.abs(out[0].numpy().astype(np.float64) - ref)
    assert err.sum() <= 1e-6 * np.abs(ref).sum() and err.max() <= 1e-4 * np.abs(ref).max()

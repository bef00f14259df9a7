"""16-bit staged tiles (two lines per thread) over the shapes their run-time sizes have to get
right: u_z lines of every accepted length (256 columns start inside a line for 24, 40 and
48), position lines with every remainder of the 4-face blocks, lines of the shortest and of
nearly the longest kind, u_x lines that the register-line kernel does not take.

Each sweep against the FP64 oracle's sweep of the same decoded input, with the codec bound
of the other 16-bit tests: relative L1 <= 2^-8 (BF16) / 2^-11 (FP16) + 1e-6, L_inf <= 1.5 x
twice that.  The tiles draw the rounding streams that the shape draws on its other kernel (the
streamed sweep; the register lines for u_x lines of 48), walked forward or backward: the same
codes but for FP32's last place.  Only position lines of 16, 24, 32, 48, 64 or 96 cells with n_uz = 32 and lines of
48 with n_uz = 48 draw one stream per column in the order of the walk, from the line's end where u < 0:
their codes are checked against a NumPy copy of that stream.
"""
import numpy as np
import pytest

import oracle as O
from paper_2110_15867_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (n, nu): n_uz 16, 24, 40, 48, 32; position lines of 4..9, 13, 18, 35, 90 cells; then lines that draw
# their own streams, beside others that do not
SHAPES = [((9, 5, 6), (16, 16, 16)), ((4, 13, 7), (16, 16, 24)), ((18, 4, 8), (8, 16, 40)),
          ((5, 35, 4), (16, 4, 48)), ((90, 4, 5), (8, 32, 32)), ((4, 4, 6), (24, 32, 32)), ((4, 5, 4), (40, 16, 48)),
          ((16, 5, 24), (8, 32, 32)), ((5, 48, 4), (48, 16, 48)), ((4, 4, 5), (48, 16, 32))]


def _own_streams(L, nuz, ax):
    return L == 48 if nuz == 48 else ax < 3 and nuz == 32 and L in (16, 24, 32, 48, 64, 96)


def _own_codes(values, scale, ax, seed, drift, fmt):
    """values (FP32, before rounding) as codes by one stream per column: 16 random bits a cell in
    walk order, the upper halves of x -> 1664525 x + 1013904223 from a hash (MurmurHash3's
    finalizer) of the column's first cell and the sweep's number.  drift: the sign of the
    Courant number, broadcastable over the columns."""
    M, u64 = np.uint64(0xffffffff), np.uint64
    first = np.take(np.arange(values.size, dtype=np.uint64).reshape(values.shape), 0, axis=ax)
    x = (first ^ u64(seed * 0x85ebca6b)) & M
    for shift, mul in ((16, 0x85ebca6b), (13, 0xc2b2ae35), (16, 1)):
        x ^= x >> u64(shift)
        x = (x * u64(mul)) & M
    draws = np.empty((values.shape[ax],) + first.shape, dtype=np.uint32)
    for d in draws:
        x = (x * u64(1664525) + u64(1013904223)) & M
        d[...] = x >> u64(16)
    draws = np.moveaxis(np.where(drift < 0, draws[::-1], draws), 0, ax)
    bits = (values * (np.float32(1) / scale)[..., None]).view(np.uint32)
    if fmt == "bf16":
        return ((bits + draws) >> np.uint32(16)).astype(np.uint16)
    up = (bits + (draws & np.uint32(0x1fff))).view(np.float32)
    h = up.astype(np.float16)  # toward zero
    return h.view(np.uint16) - (h.astype(np.float32) > up)


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
    axes = [0, 1, 2] + ([3] if nu[0] in (24, 40, 48) else [])
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
        if not _own_streams((n + nu)[ax], nu[2], ax):
            # (the streamed kernel's products of code and scale may be fused into its first sums: a few
            # units of FP32's last place, against the 2^16 (BF16) or 2^13 (FP16) of a code's step)
            assert (got[True].view(torch.int16) != got[False].view(torch.int16)).float().mean() <= 1e-3, ax
            continue
        f32 = B.decode_lines(codes0, scale0, torch.float32)
        v = B.Vlasov(f32, V=V)
        v.sweep(ax, dt, 0.9, phi)  # the same march, unrounded
        v.close()
        if ax < 3:
            drift = np.sign(np.arange(nu[ax]) + 0.5 - nu[ax] / 2).reshape([-1 if k == ax + 3 else 1 for k in range(6) if k != ax])
        else:
            drift = np.sign(-(8 * (np.roll(phi64, -1, 0) - np.roll(phi64, 1, 0)) - np.roll(phi64, -2, 0) + np.roll(phi64, 2, 0)))
            drift = drift[..., None, None]
        want = _own_codes(f32.cpu().numpy(), scale0.cpu().numpy(), ax, 1, drift, fmt)
        # (the kernel multiplies by a reciprocal that is off by up to 2 units in the last place)
        assert (want != got[True].view(torch.int16).cpu().numpy().view(np.uint16)).mean() <= 1e-3, ax

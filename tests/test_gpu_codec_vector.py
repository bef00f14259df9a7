"""The four-at-a-time codec kernels against the one-at-a-time ones, which arrays that are only
aligned to their elements still take: the same bits for every count of lanes per line, line
counts around a warp's and a block's, empty lines and the scalar-only lengths between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _shifted(t):
    """A copy of t at an address one element past an aligned one."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    out = buf[1:].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("fmt", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("src", [torch.float32, torch.float64])
@pytest.mark.parametrize("nuz", [4, 8, 12, 20, 32, 36, 64, 68, 128, 7])
def test_aligned_and_shifted_arrays_give_the_same_bits(fmt, src, nuz):
    from paper_2110_15867_gb300 import binding as B
    B.load()
    for nlines in (1, 7, 33, 4099):
        rng = np.random.default_rng(nuz + nlines)
        v = rng.random((nlines, nuz)) * np.exp(rng.uniform(-30, 5, size=(nlines, 1)))
        v[rng.random(nlines) < 0.1] = 0.0
        f = torch.from_numpy(v).cuda().to(src)
        c1, s1 = B.encode_lines(f, fmt)
        c2, s2 = B.encode_lines(_shifted(f), fmt, codes=_shifted(torch.zeros_like(c1)))
        assert torch.equal(c1.view(torch.int16), c2.view(torch.int16)) and torch.equal(s1, s2), nlines
        top = f.float().amax(-1)
        assert torch.equal(s1, top.clamp(min=2.0 ** -64) if fmt is torch.bfloat16 else top), nlines
        d1 = B.decode_lines(c1, s1, src)
        d2 = B.decode_lines(_shifted(c1), s1, src)
        assert torch.equal(d1, d2), nlines
        assert torch.equal(d1, (c1.to(torch.float64) * s1.to(torch.float64)[:, None]).to(src)), nlines

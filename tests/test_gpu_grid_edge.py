"""Pixels on the gridding radius: with a convolution function that does not vanish there
(a disc), a pixel takes a visibility when dx^2 + dy^2, in FP32 as fma(dx, dx, dy dy), is
below r_max^2, whatever the pixel's tile.  The other order, fma(dy, dy, dx dx), differs
by a last bit for some pairs; the visibilities here are such pairs, on all four sides
and in all tile positions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = 12.0
F = np.float32


def fma(a, b, c):
    """FP32 fused multiply-add of arrays (the product is exact in FP64; None of the pairs
    used rounds differently for the sum's second rounding)."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def edge_pairs(n, pix):
    """n offsets (dx, dy) of a visibility from a pixel whose two FP32 sums fall on either
    side of R^2, representable at coordinates up to `pix`."""
    rng = np.random.default_rng(5)
    step = 2.0 ** (np.ceil(np.log2(pix)) - 24)
    out = []
    while len(out) < n:
        dx = np.round(rng.uniform(0.5, R - 0.5, 200000) / step) * step
        dy = np.round(np.sqrt(R * R - dx * dx) / step) * step + step * rng.integers(-1, 2, dx.size)
        x, y = dx.astype(F), dy.astype(F)
        a, b = fma(x, x, y * y), fma(y, y, x * x)
        out += list(zip(dx[(a < R * R) != (b < R * R)], dy[(a < R * R) != (b < R * R)]))
    return np.array(out[:n]) * rng.choice([-1.0, 1.0], size=(n, 2))


@pytest.mark.parametrize("n_pol", [1, 4])
def test_pixels_on_the_radius(n_pol):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_5575_gb300 import Gridder, build
    build.build()
    n_pix, cell = 1000, 37
    side = n_pix // cell - 1
    d = edge_pairs(side * side, n_pix)
    k = np.arange(side * side)
    pix = cell * np.stack([k % side, k // side], axis=1) + 27
    xy = (pix - d).astype(F)
    assert np.array_equal(pix - xy.astype(np.float64), d)
    want = np.zeros((n_pix, n_pix), dtype=bool)
    for px, q in zip(pix, xy):
        x, y = (np.arange(px[i] - 25, px[i] + 26) for i in (0, 1))
        dx, dy = np.meshgrid(x.astype(F) - q[0], y.astype(F) - q[1])
        want[np.ix_(y, x)] |= fma(dx, dx, dy * dy) < F(R * R)
    for bin in (12, 24, 33):
        g = Gridder(n_pix, R, np.ones(2), bin=bin, n_pol=n_pol, max_vis=len(xy))
        out = g.run(torch.from_numpy(xy).cuda(), torch.ones((len(xy), n_pol), dtype=torch.complex64, device="cuda"))
        got = out.cpu().numpy()
        g.close()
        for pol in range(n_pol):
            np.testing.assert_array_equal(got[pol] != 0, want)

"""Ray counts and texel tables where FP32 stands in for FP64 (k_map.cu).

FP64 ray counts by FP32 rays: every ray near a bin edge takes the FP64
deflection, so counts, off-map and lost totals equal the oracle's.  FP16
codes by FP32 logarithms: equal to the FP64 logarithm rounded once, also on
either side of every rounding boundary.
"""
import numpy as np
import pytest

import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1511_01157_gb300 as m
    c = m.Context(0)
    yield c
    c.close()


# (s, q, L, npix, rays, X): maps narrower and wider than the bin window,
# ragged ray grids, a ray on each lens (s = 2, q = 1, X = 2.5: x = -1, 1),
# wide and tiny lenses, and sizes whose error bound sends every ray to FP64
@pytest.mark.parametrize("s,q,L,npix,rays,X", [
    (1.0, 1e-3, 2.0, 512, 1029, 3.0),
    (0.3, 0.1, 2.0, 127, 700, 3.0),
    (2.0, 1.0, 2.0, 129, 5, 2.5),
    (2.0, 1.0, 2.0, 64, 255, 2.5),
    (1.1, 1e-9, 2.0, 300, 513, 3.0),
    (3.0, 5.0, 1e-3, 256, 1025, 3.0),
    (0.9, 5e-4, 2.0, 2048, 777, 3.0),
    (1.0, 1e-2, 2.0, 2, 257, 3.0),
    (40.0, 0.5, 30.0, 500, 601, 45.0),
    (1.0, 1e-3, 2.0, 64, 300, 1e5),
    (1e9, 1e-3, 2.0, 64, 300, 3.0),
])
def test_fp64_counts_equal_oracle(ctx, s, q, L, npix, rays, X):
    mp = ctx.build_map(s, q, L, npix, rays, image_halfwidth=X,
                       deflect="fp64")
    c, off, lost = mp.counts()
    A_o, c_o, off_o, lost_o = orc.build_map(s, q, L, npix, rays, X)
    assert np.array_equal(c, c_o)
    assert (off, lost) == (off_o, lost_o)
    h, d = 2.0 * X / rays, 2.0 * L / npix
    f = (h * h) / (d * d)
    assert np.array_equal(mp.values(), (c.astype(np.float64) * f).astype(
        np.float32))
    mp.free()


def test_half_codes_at_rounding_boundaries(ctx):
    n = 512
    rng = np.random.default_rng(2)
    h = rng.integers(0, 0x4700, n * n).astype(np.uint16).view(np.float16)
    mid = (h.astype(np.float64) +
           np.nextafter(h, np.float16(np.inf)).astype(np.float64)) / 2
    mid *= rng.choice([-1.0, 1.0], n * n)
    A = np.float32(10.0 ** mid)
    k = rng.integers(-2, 3, n * n)  # a few ulps about the boundary
    A = (A.view(np.int32) + k.astype(np.int32)).view(np.float32)
    A = np.clip(A, np.float32(1e-9), np.float32(1e9)).reshape(n, n)
    A[0, :8] = [0.0, 1.0, 1e-6, 1e-5, 1e4, 1e-7, 1.0000001, 0.9999999]
    mp = ctx.map_from_host(A, 2.0)
    mp.set_lookup(True)
    codes, floor = mp.half()
    want = np.log10(np.maximum(A.astype(np.float64), floor)).astype(
        np.float16).view(np.uint16)
    assert np.array_equal(codes, want)
    mp.free()

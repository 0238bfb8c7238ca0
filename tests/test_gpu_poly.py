"""GPU parity of the polynomial map generator (§4.1: the lens polynomial
solved at every texel centre) against the oracle's poly_map.

* Texel values equal the oracle's FP64 point-source magnification at the
  texel centres, rounded to FP32, within 1e-6 relative away from caustics
  (the two solve the quintic differently: the GPU in the frame of the mass
  midpoint by the Aberth-Ehrlich iteration, the oracle in the centre-of-
  mass frame by Laguerre with deflation).  On a caustic the image count can
  differ between two correct solvers; at most 1e-3 of the texels may
  differ by more.
* A map made this way is searched like any other: chi^2 against the oracle
  on the same values within 1e-5.
"""
import numpy as np
import pytest

import oracle as orc
import synth

pytestmark = pytest.mark.gpu

NT = orc.threads_default()


@pytest.fixture(scope="module")
def m():
    import paper_1511_01157_gb300 as lib
    return lib


@pytest.fixture(scope="module")
def ctx(m):
    c = m.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("s,q,L,npix", [
    (1.0, 1e-3, 2.0, 128),
    (0.6, 0.2, 1.5, 96),
    (2.5, 5e-4, 2.0, 128),
    (1.1, 1.0, 1.2, 65),       # equal masses, odd size
    (0.95, 1e-5, 1.0, 128),    # low-mass planet next to the central caustic
])
def test_poly_map_matches_oracle(ctx, m, s, q, L, npix):
    mp = ctx.build_map(s, q, L, npix, 1, generator="poly")
    A = mp.values()
    P = orc.poly_map(s, q, L, npix, nthreads=NT)
    rel = np.abs(A.astype(np.float64) - P) / P
    # smooth texels: the image count is the same at the 8 neighbours
    d = 2 * L / npix
    cnt = np.array([[orc.images(s, q, -L + (i + 0.5) * d,
                                -L + (j + 0.5) * d)[0]
                     for i in range(npix)] for j in range(npix)])
    from scipy.ndimage import maximum_filter, minimum_filter
    smooth = maximum_filter(cnt, 3) == minimum_filter(cnt, 3)
    assert smooth.mean() > 0.8
    print(f"max rel (smooth) {rel[smooth].max():.2e}, texels > 1e-6: "
          f"{(rel > 1e-6).sum()} of {rel.size}")
    assert rel[smooth].max() <= 1e-6
    assert (rel > 1e-6).mean() <= 1e-3
    with pytest.raises(m.MorseError) as e:
        mp.counts()
    assert e.value.status == m.EINVAL


def test_poly_map_search_and_fp16(ctx, m):
    s, q, L, npix = 1.0, 1e-3, 2.0, 256
    mp = ctx.build_map(s, q, L, npix, 1, generator="poly", fp16log=True)
    A = mp.values()
    mp.set_lookup(False)
    c = synth.CFG0
    t = synth.epoch_times(300, 4, 0.0)
    At = orc.lightcurve_point(s, q, t, 0.0, 20.0, 0.05, 0.7)
    F, sig = synth.photometry(At + 0.3, 4)
    ev = ctx.event(t, F, sig)
    g = m.Grid.make(6, 12, 5, 5, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True, True,
                    8)
    og = orc.Grid(6, 12, 5, 5, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0)
    chi2, *_ = ctx.grid_chi2_dense(ev, mp, g)
    o, *_ = orc.grid_chi2(og, t, F, 1.0 / sig ** 2, A=A, L=L, nthreads=NT)
    assert np.max(np.abs(chi2 - o) / o) <= 1e-5
    mp.set_lookup(True)
    codes, floor = mp.half()
    assert floor == 1e-6
    assert np.abs(codes.astype(int) -
                  orc.log10_half(A, floor).astype(int)).max() <= 1


def test_sweep_with_polynomial_maps(ctx, m):
    t = synth.epoch_times(200, 6, 0.0)
    At = orc.lightcurve_point(0.9, 2e-3, t, 0.0, 15.0, 0.1, 1.0)
    F, sig = synth.photometry(At + 0.2, 6)
    ev = ctx.event(t, F, sig)
    g = m.Grid.make(5, 8, 4, 4, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True, True,
                    4)
    S, Q = [0.8, 0.9], [1e-3, 2e-3]
    sw = ctx.sweep(ev, S, Q, 2.0, 96, 1, g, generator="poly")
    for i in range(2):
        mp = ctx.build_map(S[i], Q[i], 2.0, 96, 1, generator="poly")
        one = ctx.grid_chi2(ev, mp, g)
        assert np.array_equal(sw[i]["idx"], one["idx"])
        assert np.array_equal(sw[i]["chi2"], one["chi2"])


@pytest.mark.parametrize("s,q,L,npix", [
    (1.0, 1e-8, 2.0, 64),      # the lightest lens of the fast form
    (0.05, 0.3, 2.0, 64),      # close: most texels left to the general form
    (1.0, 1e-3, 0.02, 96),     # about the central caustic
    (1.2, 5.0, 2.0, 96),       # the lighter lens on the left
    (1.0, 1e-9, 2.0, 48),      # general form alone
    (1.3, 0.06, 2.0, 33),      # a row that does not fill a block
])
def test_poly_map_fast_and_general_forms(ctx, s, q, L, npix):
    A = ctx.build_map(s, q, L, npix, 1, generator="poly").values()
    P = orc.poly_map(s, q, L, npix, nthreads=NT)
    assert np.isfinite(A).all() and (A >= 1.0 - 1e-6).all()
    rel = np.abs(A.astype(np.float64) - P) / P
    assert (rel > 1e-6).mean() <= 1e-3


# A next to a fold goes as the square root of the distance to it, so an error
# of a few ulps of the texel's place (4e-16 at |y| < 2) moves A by some
# 2e-14 A^2 of itself where the caustic's scale is 1e-2
def _near_caustic(ctx, s, q, L, npix, cols, rows):
    A = ctx.build_map(s, q, L, npix, 1, generator="poly").values()
    d = 2 * L / npix
    got = A[rows[0]:rows[1], cols[0]:cols[1]].astype(np.float64)
    P = np.array([[orc.mag_point(s, q, -L + (i + 0.5) * d, -L + (j + 0.5) * d)
                   for i in range(*cols)] for j in range(*rows)])
    assert np.isfinite(A).all()
    assert (np.abs(got - P) <= (1e-6 + 2e-14 * P ** 2) * P).all()


@pytest.mark.parametrize("s,q,L,col,row", [
    # FP32 iterations that do not converge, or meet away from the roots: a
    # pair of images must not be lost with them
    (5.782718165466182, 0.04254807934035008, 2.0082425727177124, 1813, 2048),
    (8.05, 0.235, 1.924, 447, 2048),
    (4.13, 0.867, 2.296, 482, 2047),
    (3.9046490442410478, 0.33909214800333815, 2.15438373784511, 1206, 2047),
])
def test_poly_map_keeps_every_image_pair(ctx, s, q, L, col, row):
    _near_caustic(ctx, s, q, L, 4096, (col - 3, col + 4), (row - 3, row + 4))


@pytest.mark.parametrize("s,q,L", [(4.0, 0.5, 1.6), (8.0, 0.3, 2.2),
                                   (20.0, 0.1, 2.0)])
def test_poly_map_about_a_wide_lens_caustic(ctx, s, q, L):
    """Every texel about the heavier lens' caustic, inside and outside."""
    e2 = q / (1 + q)
    col = int((-s * e2 + e2 / s + L) / (2 * L / 4096))
    assert 40 <= col < 4096 - 40
    _near_caustic(ctx, s, q, L, 4096, (col - 40, col + 40), (2028, 2068))


def test_poly_map_general_form_spreads_small_maps(ctx):
    """A 64^2 map by the general form alone has a sixteenth of the texels of
    a 256^2 one; it must not take as long (half as long would already mean
    that most of the chip waits)."""
    ms = {}
    for npix in (64, 256):
        t = []
        for _ in range(4):
            ctx.build_map(1.0, 1e-9, 2.0, npix, 1, generator="poly").free()
            t.append(ctx.kernel_ms(0))
        ms[npix] = min(t)
    assert ms[64] < 0.5 * ms[256]


@pytest.mark.parametrize("npix", [2, 11, 12, 197, 198])
def test_poly_map_tiles(ctx, npix):
    """Maps of less and more than a block's tile of texels, of tiles of one
    and of two texels per thread, and the general form alone."""
    for s, q in ((0.05, 0.3), (1.0, 1e-9)):
        A = ctx.build_map(s, q, 2.0, npix, 1, generator="poly").values()
        P = orc.poly_map(s, q, 2.0, npix, nthreads=NT)
        rel = np.abs(A.astype(np.float64) - P) / P
        assert (rel > 1e-6).mean() <= 1e-3


def test_poly_map_rounds_as_the_general_form(ctx):
    """Texels equal the oracle's FP64 magnification rounded to FP32, bit for
    bit, but for near ties: the general form's did in every one of 2.4e6, and
    where the FP64 steps stop early the fast form's would not in 1 of 6e4."""
    rng = np.random.default_rng(8)
    unlike = 0
    for _ in range(24):
        s = np.exp(rng.uniform(np.log(0.3), np.log(3.0)))
        q = np.exp(rng.uniform(np.log(1e-5), np.log(0.1)))
        A = ctx.build_map(s, q, 2.0, 256, 1, generator="poly").values()
        unlike += int((A != orc.poly_map(s, q, 2.0, 256, nthreads=NT)
                       .astype(np.float32)).sum())
    assert unlike <= 1

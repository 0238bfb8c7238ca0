"""The screened trajectory search (k_screen.cu) against the dense ranking.

The dense call evaluates every trajectory; the screened top-K must be its
smallest K by (chi2, index), bit for bit: at the epoch counts where the
subsets' sizes change, on light curves whose bounds discard nearly all, some
or none of the grid (the last searches the whole range), for ranges, cut
lines, FP16 tables, line grids and several K.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    import paper_1511_01157_gb300 as lib
    return lib


@pytest.fixture(scope="module")
def setup(m):
    ctx = m.Context(0)
    mp = ctx.build_map(1.1, 3e-3, 2.0, 301, 2100, image_halfwidth=3.0,
                       deflect="fp32")
    yield ctx, mp
    ctx.close()


def _event(ctx, n, kind, seed=5):
    t = synth.epoch_times(n, seed)
    if kind == "flat":      # no signal: no bound can discard anything
        f = np.full(n, 2.0)
    elif kind == "weak":
        f = 3.0 + 1.0 / np.sqrt(0.5 + (t / 60.0) ** 2)
    else:                   # high magnification, two bumps
        f = (0.4 + 1.0 / np.sqrt(2e-4 + (t / 15.0) ** 2) +
             3.0 * np.exp(-((t - 1.3) / 0.2) ** 2))
    F, sig = synth.photometry(f, seed, 0.01 if kind == "strong" else 0.0)
    return ctx.event(t, F, sig)


def _grid(m, top_k, a_min=0.0, n_tE=9):
    return m.Grid.make(12, 20, 11, n_tE, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0,
                       True, True, top_k, a_min)


def _best(chi2, k, first=0):
    idx = np.lexsort((np.arange(len(chi2)), chi2))[:k]
    idx = idx[np.isfinite(chi2[idx])]
    return idx + first, chi2[idx]


@pytest.mark.parametrize("kind", ["strong", "weak", "flat"])
@pytest.mark.parametrize("n", [127, 128, 639, 640, 1023, 1024, 2047, 2048,
                               3001])
def test_screened_equals_dense(m, setup, n, kind):
    ctx, mp = setup
    ev = _event(ctx, n, kind)
    for k in (1, 33):
        g = _grid(m, k)
        got = ctx.grid_chi2(ev, mp, g)
        chi2, fs, fb = ctx.grid_chi2_dense(ev, mp, g)
        idx, val = _best(chi2, k)
        assert np.array_equal(got["idx"], idx)
        assert np.array_equal(got["chi2"], val)
        assert np.array_equal(got["Fs"], fs[idx])
        assert np.array_equal(got["Fb"], fb[idx])


@pytest.mark.parametrize("kind", ["strong", "flat"])
def test_screened_forms(m, setup, kind):
    ctx, mp = setup
    ev = _event(ctx, 1500, kind)
    g = _grid(m, 700)
    chi2, *_ = ctx.grid_chi2_dense(ev, mp, g)
    idx, val = _best(chi2, 700)
    got = ctx.grid_chi2(ev, mp, g)
    assert np.array_equal(got["idx"], idx)
    assert np.array_equal(got["chi2"], val)
    # a range that starts and ends inside a line
    for first, count in ((1, g.size - 2), (1237, 17001)):
        r = ctx.grid_chi2_range(ev, mp, g, first, count)
        idx, val = _best(chi2[first:first + count], 700, first)
        assert np.array_equal(r["idx"], idx)
        assert np.array_equal(r["chi2"], val)
    # FP16 table
    mp.set_lookup(True)
    h16, *_ = ctx.grid_chi2_dense(ev, mp, g)
    got = ctx.grid_chi2(ev, mp, g)
    mp.set_lookup(False)
    idx, val = _best(h16, 700)
    assert np.array_equal(got["idx"], idx)
    assert np.array_equal(got["chi2"], val)
    # the minimum-magnification cut
    top = ctx.line_max(mp, g)
    cut = _grid(m, 700, float(np.median(top)))
    kept, *_ = ctx.grid_chi2_dense(ev, mp, cut)
    idx, val = _best(kept, 700)
    got = ctx.grid_chi2(ev, mp, cut)
    assert np.array_equal(got["idx"][:len(idx)], idx)
    assert np.array_equal(got["chi2"][:len(idx)], val)
    # the same lines as a line grid, an odd number of tE
    g = _grid(m, 20, n_tE=13)
    u0 = np.exp(np.linspace(np.log(1e-3), np.log(0.5), 12))
    lines = np.array([(u, 2 * np.pi * j / 20, 0.0) for u in u0
                      for j in range(20)])
    lg = m.Grid.make(len(lines), 1, 11, 13, 1.0, 1.0, -2.0, 2.0, 5.0, 80.0,
                     False, True, 20)
    a, b = ctx.grid_chi2_lines(ev, mp, lg, lines), ctx.grid_chi2(ev, mp, g)
    assert np.array_equal(a["idx"], b["idx"])
    np.testing.assert_allclose(a["chi2"], b["chi2"], rtol=1e-6)


def test_screened_batch_equals_single_searches(m, setup):
    """Light curves with one, three and four subsets, of strong and of no
    signal (pairs that fall back to the whole range), in one batch."""
    ctx, mp = setup
    other = ctx.build_map(0.7, 2e-2, 2.0, 301, 2100, image_halfwidth=3.0,
                          deflect="fp32")
    evs = [_event(ctx, n, kind) for n, kind in
           ((130, "strong"), (700, "weak"), (1500, "strong"),
            (1500, "flat"), (3000, "strong"), (3000, "flat"))]
    g = _grid(m, 40)
    for h16 in (False, True):
        mp.set_lookup(h16)
        other.set_lookup(h16)
        got = ctx.grid_chi2_batch(evs, [mp, other], g)
        for i, ev in enumerate(evs):
            for j, x in enumerate((mp, other)):
                assert np.array_equal(got[i, j], ctx.grid_chi2(ev, x, g))
    mp.set_lookup(False)
    other.free()


@pytest.mark.parametrize("n", [3, 33, 257, 3001])
@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (3, 7, 2, 3),
                                  (8, 16, 8, 8), (9, 16, 8, 8)])
def test_small_grid_equals_dense(m, setup, dims, n):
    """Up to 8192 trajectories every one is bounded over the whole light
    curve; just above, the unscreened search."""
    ctx, mp = setup
    g = m.Grid.make(*dims, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True, True, 37)
    for kind in ("strong", "flat"):
        ev = _event(ctx, n, kind)
        got = ctx.grid_chi2(ev, mp, g)
        chi2, fs, fb = ctx.grid_chi2_dense(ev, mp, g)
        idx, val = _best(chi2, 37)
        k = len(idx)
        assert np.array_equal(got["idx"][:k], idx)
        assert np.array_equal(got["chi2"][:k], val)
        assert np.array_equal(got["Fs"][:k], fs[idx])
        assert np.all(got["idx"][k:] == -1)
    if g.size > 100:
        cut = m.Grid.make(*dims, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True, True,
                          37, float(np.median(ctx.line_max(mp, g))))
        kept, *_ = ctx.grid_chi2_dense(ev, mp, cut)
        idx, val = _best(kept, 37)
        got = ctx.grid_chi2(ev, mp, cut)
        assert np.array_equal(got["idx"][:len(idx)], idx)
        r = ctx.grid_chi2_range(ev, mp, g, 5, 91)
        idx, val = _best(chi2[5:96], 37, 5)
        assert np.array_equal(r["idx"], idx)


@pytest.mark.parametrize("kind", ["strong", "weak"])
@pytest.mark.parametrize("n", [1024, 1027, 3001])
def test_listed_bounds_on_one_to_four_lanes(m, setup, n, kind):
    """409 600 trajectories: K from 1 to 4096 makes the list of the second
    bound from a few tiles, its trajectories on four lanes each, to more
    than there are blocks, on one."""
    ctx, mp = setup
    ev = _event(ctx, n, kind)
    dims = (40, 40, 16, 16, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True, True)
    chi2, *_ = ctx.grid_chi2_dense(ev, mp, m.Grid.make(*dims, 1))
    for h16 in (False, True):
        mp.set_lookup(h16)
        if h16:
            chi2, *_ = ctx.grid_chi2_dense(ev, mp, m.Grid.make(*dims, 1))
        for k in (1, 64, 1024, 4096):
            got = ctx.grid_chi2(ev, mp, m.Grid.make(*dims, k))
            idx, val = _best(chi2, k)
            assert np.array_equal(got["idx"][:len(idx)], idx)
            assert np.array_equal(got["chi2"][:len(idx)], val)
    mp.set_lookup(False)


def _curve(ctx, n, kind):
    t = synth.epoch_times(n, 9)
    f = {"flat": np.full(n, 2.0),
         "faint": 2.0 + 0.03 / np.sqrt(1.0 + (t / 20.0) ** 2),
         # no trajectory fits it: screened, and the lists come out too long
         "wave": 2.0 + 0.5 * np.sin(2 * np.pi * t / 7.0),
         "strong": 0.4 + 1.0 / np.sqrt(2e-4 + (t / 15.0) ** 2)}[kind]
    F, sig = synth.photometry(f, 9)
    return ctx.event(t, F, sig)


@pytest.mark.parametrize("n", [300, 1500, 3001])
def test_light_curves_the_bounds_cannot_use(m, setup, n):
    """Without a signal that the subsets can discard by, the search is the
    unscreened one (that of a light curve too short for subsets), not the
    screen and then all of it again."""
    ctx, mp = setup
    # (one subset: on large grids only)
    big = n < 1024
    g = m.Grid.make(40, 40, 25 if big else 5, 15 if big else 5, 1e-3, 0.5,
                    -2.0, 2.0, 5.0, 80.0, True, True, 33)

    def launches(ev):
        ctx.grid_chi2(ev, mp, g)
        a = ctx.launch_count()
        ctx.grid_chi2(ev, mp, g)
        return ctx.launch_count() - a

    plain = launches(_curve(ctx, 100, "strong"))
    assert launches(_curve(ctx, n, "strong")) > plain
    assert launches(_curve(ctx, n, "wave")) > plain
    for kind in ("flat", "faint"):
        assert launches(_curve(ctx, n, kind)) == plain
    for kind in ("wave", "faint"):
        ev = _curve(ctx, n, kind)
        for k in (1, 33):
            chi2, *_ = ctx.grid_chi2_dense(ev, mp, _grid(m, k))
            idx, val = _best(chi2, k)
            got = ctx.grid_chi2(ev, mp, _grid(m, k))
            assert np.array_equal(got["idx"], idx)
            assert np.array_equal(got["chi2"], val)


def test_batch_of_weak_and_strong_light_curves(m, setup):
    ctx, mp = setup
    other = ctx.build_map(0.7, 2e-2, 2.0, 301, 2100, image_halfwidth=3.0,
                          deflect="fp32")
    g = _grid(m, 40)
    for kinds in (("strong", "flat", "wave", "faint", "strong", "flat"),
                  ("flat", "faint", "flat"), ("flat", "strong", "wave")):
        evs = [_curve(ctx, n, kind) for n, kind in
               zip((130, 700, 1500, 900, 3000, 5000), kinds)]
        got = ctx.grid_chi2_batch(evs, [mp, other], g)
        for i, ev in enumerate(evs):
            for j, x in enumerate((mp, other)):
                assert np.array_equal(got[i, j], ctx.grid_chi2(ev, x, g))
    other.free()


def test_no_list_where_a_sample_says_it_would_be_long(m, setup):
    """300 000 trajectories that all miss the light curve: the screen must end
    before the second and third subsets of the whole grid (half as much again
    as the search of a flat light curve, which is not screened)."""
    ctx = setup[0]
    mp = ctx.build_map(1.0, 1e-3, 2.0, 1024, 4000, image_halfwidth=3.0,
                       deflect="fp32")
    g = m.Grid.make(30, 40, 25, 10, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True,
                    True, 16)
    ms = {}
    for kind in ("flat", "wave"):
        ev = _curve(ctx, 1100, kind)
        got = [ctx.grid_chi2(ev, mp, g) for _ in range(2)][-1]
        t = []
        for _ in range(7):
            ctx.grid_chi2(ev, mp, g)
            t.append(ctx.kernel_ms(2))
        ms[kind] = min(t)
        chi2, *_ = ctx.grid_chi2_dense(ev, mp, g)
        idx, val = _best(chi2, 16)
        assert np.array_equal(got["idx"], idx)
        assert np.array_equal(got["chi2"], val)
    mp.free()
    print(f"wave {ms['wave']:.3f} ms, flat {ms['flat']:.3f} ms")
    assert ms["wave"] < 1.35 * ms["flat"]


def test_subsets_cost_little_of_an_event(m, setup):
    """Light curves of 2^20 epochs have subsets, longer ones none: what they
    add to making the event."""
    import time
    ctx = setup[0]
    t = synth.epoch_times((1 << 20) + 1, 9)
    f = 0.4 + 1.0 / np.sqrt(2e-4 + (t / 15.0) ** 2)
    F, sig = synth.photometry(f, 9)
    best = []
    for n in (1 << 20, (1 << 20) + 1):
        w = []
        for _ in range(9):
            t0 = time.perf_counter()
            ctx.event(t[:n], F[:n], sig[:n]).free()
            w.append(time.perf_counter() - t0)
        best.append(min(w))
    print(f"with subsets {best[0]:.4f} s, without {best[1]:.4f} s")
    assert best[0] < 1.45 * best[1]

"""Device memory of the handles and the workspace.

* Freed maps and events: the memory is the next handle's only when every
  stream has finished with it, and what the context keeps of it is bounded at
  once, not only by its later calls.
* On a GPU that others have filled a search whose screen does not fit is the
  unscreened one.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def m():
    import paper_1511_01157_gb300 as lib
    return lib


def _event(ctx, n, seed=3):
    t = synth.epoch_times(n, seed)
    F, sig = synth.photometry(0.3 + 1.0 / np.sqrt(0.03 + (t / 18.0) ** 2),
                              seed)
    return ctx.event(t, F, sig)


def test_freed_memory_is_given_back(m):
    """3.3 GB of maps, freed: 2 GB at most stay with the context at once, 256
    MB after its next synchronous call."""
    import torch
    ctx = m.Context(0)
    small = ctx.build_map(1.0, 1e-3, 2.0, 64, 200, deflect="fp32")
    small.values()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info(0)[0]
    held = [ctx.build_map(1.0, 1e-3, 2.0, 4096, 4096, deflect="fp32")
            for _ in range(8)]
    assert before - torch.cuda.mem_get_info(0)[0] > 3000 * MB
    for x in held:
        x.free()
    assert before - torch.cuda.mem_get_info(0)[0] <= 2048 * MB
    small.values()
    assert before - torch.cuda.mem_get_info(0)[0] <= 288 * MB
    ctx.close()


def test_a_map_is_freed_after_every_streams_work(m):
    """A captured gradient replayed on a stream of its own: freeing the map
    and the event waits for the replays, and the next maps do not get their
    memory before."""
    import torch
    lib_stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = m.Context(0, stream=lib_stream)
    rng = np.random.default_rng(5)
    n = 20000
    th = np.stack([rng.uniform(-1, 1, n), 20 * np.exp(rng.uniform(-.3, .3, n)),
                   .3 * np.exp(rng.uniform(-.5, .5, n)),
                   rng.uniform(-.2, .2, n)], axis=1)
    ev = _event(ctx, 3000)
    mp = ctx.build_map(1.0, 1e-3, 2.0, 512, 4000, image_halfwidth=3.0,
                       deflect="fp32")
    ref, gref, *_ = ctx.chi2_grad(ev, mp, th)
    theta = torch.tensor(th, device="cuda")
    chi2 = torch.zeros(n, dtype=torch.float64, device="cuda")
    grad = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=lib_stream):
        ctx.chi2_grad_dev(ev, mp, theta, chi2, grad)
    with torch.cuda.stream(other):
        for _ in range(100):
            graph.replay()
        done = torch.cuda.Event()
        done.record()
    assert not done.query()
    mp.free()
    assert done.query()
    ev.free()
    more = [ctx.build_map(0.3, 0.5, 2.0, 512, 4000, image_halfwidth=3.0,
                          deflect="fp32") for _ in range(3)]
    evs = [_event(ctx, 3000, 8 + k) for k in range(3)]
    torch.cuda.synchronize()
    assert np.array_equal(chi2.cpu().numpy(), ref)
    assert np.array_equal(grad.cpu().numpy(), gref)
    for x in more + evs:
        x.free()
    ctx.close()


def _fill(left):
    """Takes the GPU's free memory but for `left` bytes."""
    import torch
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info(0)[0]
    x = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    assert torch.cuda.mem_get_info(0)[0] <= left + 8 * MB
    return x


@pytest.fixture
def empty_torch():
    import torch
    yield
    torch.cuda.empty_cache()


def test_searches_whose_screen_does_not_fit(m, empty_torch):
    kw = dict(image_halfwidth=3.0, deflect="fp32")
    g = m.Grid.make(64, 128, 64, 32, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True,
                    True, 16)                       # 116 MB with the screen
    gb = m.Grid.make(40, 72, 25, 40, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True,
                     True, 16)                      # 8 pairs, 20 MB of scratch each
    small = m.Grid.make(10, 20, 10, 10, 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0, True,
                        True, 16)

    def calls(ctx, grids):
        ev = [_event(ctx, 200, s) for s in range(4)]
        mp = [ctx.build_map(s, 1e-3, 2.0, 256, 1500, **kw) for s in (1., 1.2)]
        return lambda: (ctx.grid_chi2(ev[0], mp[0], grids[0]),
                        ctx.grid_chi2_batch(ev, mp, grids[1]))

    with m.Context(0) as other:
        f = calls(other, (g, gb))
        ref = f()
        del f
    ctx = m.Context(0)
    ctx.batch_tuning(False)
    calls(ctx, (small, small))()  # (the kernels are loaded)
    f = calls(ctx, (g, gb))
    held = _fill(100 * MB)
    got = f()
    del held
    for a, b in zip(got, ref):
        for k in ("idx", "chi2", "Fs", "Fb"):
            assert np.array_equal(a[k], b[k]), k
    ctx.close()

"""Contexts of their own on several host threads, whose launches of the same
kernels differ in shared memory (top_k, epochs, source radius): a kernel's
limit belongs to the process, so no launch may depend on who set it last.
"""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_threads_with_launches_of_different_sizes():
    import paper_1511_01157_gb300 as m

    def work(n_ep, top_k, rho, out, errors, start):
        try:
            with m.Context(0) as ctx:
                ctx.batch_tuning(False)
                t = synth.epoch_times(n_ep, 3)
                F, sig = synth.photometry(
                    0.3 + 1.0 / np.sqrt(0.03 + (t / 18.0) ** 2), 3)
                ev = ctx.event(t, F, sig)
                mp = ctx.build_map(1.0, 1e-3, 2.0, 256, 1500,
                                   image_halfwidth=3.0, deflect="fp32")
                g = m.Grid.make(12, 20, 10, 10, 1e-3, 0.5, -2.0, 2.0, 5.0,
                                80.0, True, True, top_k)
                start.wait()
                for k in range(60):
                    got = (ctx.grid_chi2(ev, mp, g).tobytes(),
                           ctx.grid_chi2_batch([ev], [mp], g).tobytes(),
                           mp.finite_source(rho).values().tobytes())
                    if k == 0:
                        out.append(got)
                    elif got != out[0]:
                        raise AssertionError("results differ between calls")
                mp.free()
                ev.free()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    errors = []
    shapes = [(200, 4, 0.1), (3000, 600, 0.6), (130, 1, 1.1)]
    start = threading.Barrier(len(shapes))
    outs = [[] for _ in shapes]
    threads = [threading.Thread(target=work, args=(*s, o, errors, start))
               for s, o in zip(shapes, outs)]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    assert not errors, errors
    # each the same as alone
    for s, o in zip(shapes, outs):
        alone = []
        work(*s, alone, errors, threading.Barrier(1))
        assert not errors and alone[0] == o[0]

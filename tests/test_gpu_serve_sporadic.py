"""Requests sent one at a time to a server of several workers.

Whichever worker wakes takes the idle slot, and replays the launch sequences captured
there: a request after the slot's first ones captures nothing.
"""
import time

import numpy as np
import pytest

from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_later_requests_capture_nothing():
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(4, 4, 2)
    act = I.slab_actuation(mesh, seed=11)
    diag = float(np.linalg.norm(mesh.rest.max(0) - mesh.rest.min(0)))
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        with fsim.Server(ctx, workers=4) as sv:
            counts, times, first = [], [], None
            for _ in range(16):
                c0, t0 = ctx.capture_count(), time.perf_counter()
                rc, x, _, _, _ = sv.wait(sv.submit(m, act.fiber, act.stretch, precision=fsim.MIXED))
                counts.append(ctx.capture_count() - c0)
                times.append(1e3 * (time.perf_counter() - t0))
                assert rc == 0
                first = x if first is None else first
                assert np.abs(x - first).max() <= 1e-6 * diag
            print("captures", counts, "ms", [round(t, 1) for t in times])
    assert counts[0] > 0
    # (two requests: the buffers a frame swaps may end it either way round)
    assert sum(counts[2:]) == 0, counts

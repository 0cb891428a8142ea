"""A server counts what a batch's frames grow by.

The frames of a batch start with reduced-system buffers for 64 contact vertices; those
that need more take larger ones, which are part of the bytes in use and so of what
the memory budget sees.
"""
import time

import numpy as np
import pytest

from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_grown_buffers_are_in_use():
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(8, 8, 2)
    acts = [I.slab_actuation(mesh, seed=s) for s in range(20, 24)]
    still = np.ones(mesh.T)                   # no stretch: the slabs stay apart
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        with fsim.Server(ctx, workers=1, batch_frames=len(acts)) as sv:
            rc, _, st, _, _ = sv.wait(sv.submit(m, acts[0].fiber, still, precision=fsim.MIXED))
            assert rc == 0 and st["n_c_max"] <= 64
            before = sv.info()["bytes_in_use"]
            got = [sv.wait(t) for t in [sv.submit(m, a.fiber, a.stretch, precision=fsim.MIXED)
                                        for a in acts]]
            assert all(g[0] == 0 for g in got)
            # B-check alone, (3 n_c)^2 doubles a frame (the frames share len(acts) places)
            grown = max(72 * g[2]["n_c_max"] ** 2 for g in got)
            assert grown > 72 * 128 ** 2
            end = time.time() + 5.0           # (counted when the batch runs out of requests)
            while sv.info()["bytes_in_use"] < before + grown and time.time() < end:
                time.sleep(0.01)
            assert sv.info()["bytes_in_use"] >= before + grown

"""The CCD step bound is one number, whichever form a pair's march takes.

The solver marches a pair with a whole warp or in one lane, by how many pairs of its
warp still march, which depends on the order of an atomically filled list.
fsim_ccd_noalloc marches every pair in a lane.  Both round every operation
alike, so the bounds agree to the bit, and so do repeated calls.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _edges(tris):
    e = np.concatenate([tris[:, [0, 1]], tris[:, [1, 2]], tris[:, [2, 0]]], axis=0)
    return np.unique(np.sort(e, axis=1), axis=0).astype(np.int32)


@pytest.mark.parametrize("moving", [1, 3, None])
def test_bound_repeats_and_does_not_depend_on_the_form(moving):
    torch = pytest.importorskip("torch")
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(6, 6, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    free = mesh.pinned == 0
    p = fsim.params_for(mesh)
    dev = torch.device("cuda", 0)
    tris = torch.tensor(mesh.proxy_tris.astype(np.int32), device=dev)
    edges = torch.tensor(_edges(mesh.proxy_tris), device=dev)
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(p)
        m.set_actuation(act.fiber, act.stretch)
        for seed in range(24):
            rng = np.random.default_rng(seed)
            x = mesh.rest.copy()
            x[free] += 1e-4 * rng.standard_normal((int(free.sum()), 3))
            top = (mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free
            x[top, 2] -= 0.003
            if moving:
                low = np.nonzero(top)[0]
                low = low[np.argsort(x[low, 2])[:moving]]
                top = np.isin(np.arange(len(x)), low)
            dx = np.zeros_like(x)
            dx[top] = (0.002, 0.0, -0.003)
            dx[top] += 3e-4 * rng.standard_normal((int(top.sum()), 3))
            bounds = {m.eval_ccd(x, dx) for _ in range(4)}
            s = torch.tensor(m.eval_proxy(x), device=dev)
            ds = torch.tensor(m.eval_proxy(dx), device=dev)
            alpha = torch.zeros(1, dtype=torch.float64, device=dev)
            torch.cuda.synchronize()
            rc = ctx.lib.fsim_ccd_noalloc(
                C.c_void_p(s.data_ptr()), C.c_void_p(ds.data_ptr()), s.shape[0],
                C.c_void_p(tris.data_ptr()), tris.shape[0], C.c_void_p(edges.data_ptr()),
                edges.shape[0], p.dhat, p.ccd_s, p.accd_max_iters, C.c_void_p(alpha.data_ptr()), None)
            assert rc == fsim.FSIM_OK
            assert 0.0 < alpha.item() < 1.0, seed
            assert bounds == {alpha.item()}, (seed, bounds, alpha.item())

"""The grid form of the reduced system at the edges of its blocks.

Two slabs pressed together put every facing vertex in contact, so the slab
size sets n_c and with it the padding of the 32-wide blocks of S (n_c) and N
(3 n_c).  In float64 the grid form serves every n_c: 8 (less than a block), 18,
32 (whole blocks of S and of N), 36 and 98.  Its step is held to the same bound as
the other float64 steps (1e-9 relative to the oracle's direct solve).  A batch of
frames with n_c > 128 runs its systems side by side: each frame's result is that
of the frame alone to 1e-9 of the diagonal.
"""
import numpy as np
import pytest

from oracle import solver as S
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsim():
    from paper_2312_02999_gb300 import build, fsim as f
    build.build()
    return f


def _pressed(mesh, seed):
    rng = np.random.default_rng(seed)
    x = mesh.rest.copy()
    free = mesh.pinned == 0
    x[free] += 1e-4 * rng.standard_normal((int(free.sum()), 3))
    x[(mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free, 2] -= 0.0033
    return x


@pytest.mark.parametrize("nx,ny,n_c", [(1, 1, 8), (2, 2, 18), (3, 3, 32), (2, 5, 36), (6, 6, 98)])
def test_float64_step_at_block_edges(fsim, nx, ny, n_c):
    mesh = I.two_slabs(nx, ny, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    x = _pressed(mesh, 9)
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        m.set_actuation(act.fiber, act.stretch)
        _, clist, _ = m.eval_barrier(x)
        assert abs(len(clist) - n_c) <= 1
        dx = m.eval_global_step(x, precision=fsim.FP64)
        kappa = m.info()["kappa"]
    pr = S.Problem(mesh.rest, mesh.tets, mesh.pinned, mesh.proxy_tris, mesh.W_rowptr, mesh.W_col,
                   mesh.W_val, S.Params(dhat=mesh.dhat, tol_abs=mesh.tol_abs, kappa=kappa))
    pr.set_actuation(act.fiber, act.stretch)
    ev = pr.evaluate(x)
    g = pr.gradient(x, ev).ravel()[pr.free_dofs]
    ref = np.zeros_like(x)
    ref.reshape(-1)[pr.free_dofs] = pr.global_step_direct(g, pr.free_part(pr.barrier_hessian(ev)))
    assert np.abs(dx - ref).max() <= 1e-9 * np.abs(ref).max()


def test_batched_systems_beside_each_other(fsim):
    mesh = I.two_slabs(8, 8, 2)                      # n2 = 162: every frame passes n_c = 128
    acts = [I.slab_actuation(mesh, seed=s) for s in range(20, 25)]
    diag = np.linalg.norm(mesh.rest.max(0) - mesh.rest.min(0))
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        rc, xs, st = fsim.solve_batch(ctx, [(m, a.fiber, a.stretch, None) for a in acts],
                                      max_frames=len(acts))
        assert rc == 0
        assert all(s["reduced_steps"][fsim.REDUCED_COOPERATIVE] > 0 for s in st), st
        for a, x in zip(acts, xs):
            m.set_actuation(a.fiber, a.stretch)
            m.solve_frame(mesh.rest, precision=fsim.MIXED)
            assert np.abs(m.positions() - x).max() <= 1e-9 * diag

"""x1 of a mixed step with n_c > 128: sums over the contact forces that keep what cancels.

x1 = bx1 + Phi[:, c] v, and the forces v of a pressed pair nearly cancel in it.  The
rounding of Phi's entries and of bx1, both float32, leaves about 0.45 u32 of the
largest contact-free step at these states (median of the worst entry); sums in
float32 made it 0.7.  The bar of 0.6 lies between, 40 states each, where a median of
values that vary by 40 % is good to 8 %.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle import solver as S
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,closest", [(8, 0.02), (9, 0.02)])     # n_c = 162, 200
def test_error_of_x1(nx, closest):
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(nx, nx, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    free = mesh.pinned == 0
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        m.set_actuation(act.fiber, act.stretch)
        pr = S.Problem(mesh.rest, mesh.tets, mesh.pinned, mesh.proxy_tris, mesh.W_rowptr, mesh.W_col,
                       mesh.W_val, S.Params(dhat=mesh.dhat, tol_abs=mesh.tol_abs,
                                            kappa=m.info()["kappa"],
                                            weight_scale=mesh.weight_scale), region=mesh.region)
        pr.set_actuation(act.fiber, act.stretch)
        lu = spla.splu(pr.H.tocsc())
        i1, _ = pr.split_dofs()
        errs = []
        for seed in range(40):
            rng = np.random.default_rng(seed)
            x = mesh.rest.copy()
            x[free] += 3e-4 * rng.standard_normal((int(free.sum()), 3))
            top = (mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free
            x[top, 2] -= 0.0035
            for _ in range(8):
                x[top, 2] -= pr.evaluate(x)["C"][3].min() - closest * mesh.dhat
            ev = pr.evaluate(x)
            g = pr.gradient(x, ev).ravel()[pr.free_dofs]
            ref = spla.spsolve((pr.H + pr.free_part(pr.barrier_hessian(ev))).tocsc(), -g)
            dx = m.eval_global_step(x, precision=fsim.MIXED)
            err = np.abs(dx.ravel()[pr.free_dofs] - ref)[i1].max()
            errs.append(err / np.abs(lu.solve(g)).max())
    median = float(np.median(errs))
    print("x1", nx, closest, median * 2.0 ** 24, "u32")
    assert median <= 0.6 * 2.0 ** -24

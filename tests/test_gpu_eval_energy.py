"""eval_energy in both precisions against the oracle.

The elastic gradient of either form is within 1e-9 of its largest entry of the
oracle's, entry by entry, and the barrier's far closer, so the norm over the 3 n
entries is within sqrt(3 n) 1e-9 of that entry; the energy is within 1e-10.
"""
import numpy as np
import pytest

from oracle import solver as S
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name", ["FP64", "MIXED"])
@pytest.mark.parametrize("pressed", [False, True])
def test_energy_and_gradient_norm(prec_name, pressed):
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(4, 4, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    rng = np.random.default_rng(9)
    x = mesh.rest.copy()
    free = mesh.pinned == 0
    x[free] += 1e-4 * rng.standard_normal((int(free.sum()), 3))
    if pressed:
        x[(mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free, 2] -= 0.0033
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        m.set_actuation(act.fiber, act.stretch)
        energy, norm = m.eval_energy(x, precision=getattr(fsim, prec_name))
        kappa = m.info()["kappa"]
    pr = S.Problem(mesh.rest, mesh.tets, mesh.pinned, mesh.proxy_tris, mesh.W_rowptr, mesh.W_col,
                   mesh.W_val, S.Params(dhat=mesh.dhat, tol_abs=mesh.tol_abs, kappa=kappa))
    pr.set_actuation(act.fiber, act.stretch)
    ev = pr.evaluate(x)
    assert (ev["C"][0].size > 0) == pressed
    g = pr.gradient(x, ev).ravel()[pr.free_dofs]
    want = float(np.linalg.norm(g))
    assert abs(energy - pr.energy(x)) <= 1e-10 * abs(pr.energy(x))
    assert abs(norm - want) <= np.sqrt(g.size) * 1e-9 * np.abs(g).max()

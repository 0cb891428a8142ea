"""The float32 eigen-solve of the one-warp pair form is as good as the one-lane form's.

Both forms project the same pair Hessians in float32, so over many states a mixed step
is as far from the oracle's direct step with one as with the other: the geometric
means of the two errors over the same states differ by sampling only.  Per state the
errors of the two agree or differ by some 30 %, so the mean of 40 is good to 5 %
and the bar of 1.12 leaves more than twice that.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle import solver as S
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _state(mesh, pr, seed, closest):
    rng = np.random.default_rng(seed)
    x = mesh.rest.copy()
    free = mesh.pinned == 0
    x[free] += 3e-4 * rng.standard_normal((int(free.sum()), 3))
    top = (mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free
    x[top, 2] -= 0.0035
    for _ in range(8):
        x[top, 2] -= pr.evaluate(x)["C"][3].min() - closest * mesh.dhat
    return x


@pytest.mark.parametrize("closest", [0.3, 0.1])
def test_mixed_step_errors_of_the_two_forms(closest):
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(5, 5, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    with fsim.Context(0) as ctx:
        forms = []
        for lanes in (0, 1):
            m = ctx.upload(mesh)
            m.prefactor(fsim.params_for(mesh, barrier_lane_per_pair=lanes))
            m.set_actuation(act.fiber, act.stretch)
            forms.append(m)
        pr = S.Problem(mesh.rest, mesh.tets, mesh.pinned, mesh.proxy_tris, mesh.W_rowptr, mesh.W_col,
                       mesh.W_val, S.Params(dhat=mesh.dhat, tol_abs=mesh.tol_abs,
                                            kappa=forms[0].info()["kappa"],
                                            weight_scale=mesh.weight_scale), region=mesh.region)
        pr.set_actuation(act.fiber, act.stretch)
        logs = []
        for seed in range(40):
            x = _state(mesh, pr, seed, closest)
            ev = pr.evaluate(x)
            g = pr.gradient(x, ev).ravel()[pr.free_dofs]
            ref = spla.spsolve((pr.H + pr.free_part(pr.barrier_hessian(ev))).tocsc(), -g)
            errs = [np.abs(m.eval_global_step(x, precision=fsim.MIXED).ravel()[pr.free_dofs] - ref).max()
                    for m in forms]
            logs.append(np.log(errs))
    ratio = float(np.exp(np.mean([a - b for a, b in logs])))
    print("warp / lane", closest, ratio)
    assert ratio <= 1.12, ratio

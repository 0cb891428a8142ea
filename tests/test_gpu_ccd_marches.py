"""The CCD step bound where few pairs of a warp march, where many do, and where the
pairs slide.

A marching pair takes a whole warp or a lane, by how many of its warp march, and
every march ends at the smallest time of impact found so far.  The bound is the
oracle's up to rounding: a distance of d between points of size |x| carries a few
eps |x| / d, here below 2e-16 * 1e5, and t adds up advances proportional to such
distances, so 1e-10 leaves a factor of five.
"""
import numpy as np
import pytest

from oracle import contact as OC
from oracle import solver as S
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def state():
    mesh = I.two_slabs(6, 6, 2, gap=0.004)
    rng = np.random.default_rng(9)
    x = mesh.rest.copy()
    free = mesh.pinned == 0
    x[free] += 1e-4 * rng.standard_normal((int(free.sum()), 3))
    x[(mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free, 2] -= 0.003
    pr = S.Problem(mesh.rest, mesh.tets, mesh.pinned, mesh.proxy_tris, mesh.W_rowptr, mesh.W_col,
                   mesh.W_val, S.Params(dhat=mesh.dhat, kappa=1.0, weight_scale=mesh.weight_scale),
                   region=mesh.region)
    return mesh, pr, x


@pytest.fixture(scope="module")
def fsim_ctx():
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh, pr, x = state()
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        act = I.slab_actuation(mesh, seed=11)
        m.set_actuation(act.fiber, act.stretch)
        yield mesh, m, pr, x


@pytest.mark.parametrize("fall, slide, jitter, only", [
    (0.004, 0.0, 0.0, None),        # every pair of the gap at once
    (0.02, 0.0, 3e-4, None),        # far past it
    (0.004, 0.0, 3e-4, 1),          # the pairs of one vertex
    (0.004, 0.0, 3e-4, 3),
    (0.0005, 0.05, 0.0, None),      # along the gap, hardly closing
    (0.0, 0.02, 0.0, None),         # no impact
])
def test_step_bound_against_the_oracle(fsim_ctx, fall, slide, jitter, only):
    mesh, m, pr, x = fsim_ctx
    rng = np.random.default_rng(4)
    dx = np.zeros_like(x)
    free = mesh.pinned == 0
    top = (mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free
    if only:
        low = np.nonzero(top)[0]
        low = low[np.argsort(x[low, 2])[:only]]
        top = np.isin(np.arange(len(x)), low)
    dx[top] = (slide, 0.3 * slide, -fall)
    dx[top] += jitter * rng.standard_normal((int(top.sum()), 3))
    a = m.eval_ccd(x, dx)
    ao = OC.ccd_step_bound(pr.W @ x, pr.W @ dx, pr.tris, pr.edges, mesh.dhat)
    assert 0 < ao <= 1
    assert abs(a - ao) <= 1e-10 * ao

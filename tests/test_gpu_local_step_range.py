"""The local step's rotation over the whole range of deformation gradients.

Both precisions take a short Newton iteration where det(F A) is well positive
and a Jacobi SVD elsewhere, so the cases sit on both sides of that line:
ordinary and extreme stretches, nearly flat tets around the switch, inverted
tets, and scales whose squares leave float32.  The projections p = R A are
compared per tet with the oracle.  The rotation of M = F A has condition
s1 / (s2 + s3) (s3 carrying the sign of det M): the float64 form is held to
64 eps times it (p sums three products of entries near 1 after two
corrections that leave rounding), the mixed form to the float32 rotation's
error squared (2e-7 times the condition, squared, times 8) plus 2^-43 of the
double-float products times the condition.  The mixed form works with
F = I + Du Dm^-1 in double-float, so an F that is itself tiny carries the
rounding of 1, not its own: the tiny scale is compared in float64 only.
"""
import numpy as np
import pytest

from oracle import fem as OF
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROT = np.array([[0.36, 0.48, -0.8], [-0.8, 0.6, 0.0], [0.48, 0.64, 0.6]])
CASES = {
    "rest": (np.eye(3), 0.0),
    "rotated": (ROT, 2e-3),
    "stretched": (np.diag([2.0, 0.6, 1.1]) @ ROT, 3e-3),
    "flat_0.2": (np.diag([1.0, 0.2, 1.0]), 0.0),
    "flat_0.06": (np.diag([1.0, 1.2, 0.06]) @ ROT, 0.0),
    "flat_0.01": (np.diag([1.0, 1.0, 0.01]), 0.0),
    "inverted": (np.diag([1.0, -0.5, 1.2]) @ ROT, 0.0),
    "noisy": (np.eye(3), 3e-2),
    "tiny": (1e-5 * ROT, 0.0),
    "huge": (3e4 * ROT, 0.0),
}


@pytest.fixture(scope="module")
def setup():
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(3, 3, 2)
    act = I.slab_actuation(mesh, seed=5, lo=0.5)
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        m.set_actuation(act.fiber, act.stretch)
        _, gradN, _ = OF.tet_rest_data(mesh.rest, mesh.tets, mesh.weight_scale)
        yield mesh, m, OF.gradient_operators(gradN), OF.actuation_matrices(act.fiber, act.stretch)


@pytest.mark.parametrize("prec,name", [(p, n) for p in (0, 1) for n in sorted(CASES)
                                       if (p, n) != (1, "tiny")])
def test_projection_of_every_kind_of_tet(setup, prec, name):
    mesh, m, G, A = setup
    B, noise = CASES[name]
    rng = np.random.default_rng(3)
    x = mesh.rest @ B.T + noise * rng.standard_normal(mesh.rest.shape)
    _, _, P = m.eval_elastic(x, precision=prec, want_proj=True)
    F = OF.deformation_gradients(x, mesh.tets, G).reshape(-1, 3, 3)
    _, Po = OF.local_step(F, A)
    sig = np.linalg.svd(F @ A, compute_uv=False)
    sig[:, 2] *= np.sign(np.linalg.det(F))
    cond = sig[:, 0] / np.maximum(sig[:, 1] + sig[:, 2], 1e-12 * sig[:, 0])
    err = np.abs(P - Po.reshape(-1, 9)).max(axis=1)
    if prec == 0:
        bound = 64 * np.finfo(float).eps * cond
    else:
        bound = 8 * (2e-7 * cond) ** 2 + 2.0 ** -43 * cond
    ok = cond < 1e3      # beyond, the closest rotation itself is not determined
    assert ok.mean() > 0.9
    assert (err[ok] <= bound[ok]).all(), (err[ok] / bound[ok]).max()

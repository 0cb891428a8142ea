"""The float64 pair projection over the whole range of barrier stiffness.

The 5 x 5 eigen-solve takes its rotation angles through float32, so entries
outside that range are scaled first.  The barrier is linear in kappa: gradient
and B-check at any kappa are those at 1 times kappa, up to rounding (eigenvalues
that cancel to 0 may leave a few eps of the largest entry of their block: 1e-12 of
the largest entry is a thousand times that).
"""
import numpy as np
import pytest

from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def terms():
    from paper_2312_02999_gb300 import build, fsim
    build.build()
    mesh = I.two_slabs(4, 4, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    rng = np.random.default_rng(9)
    x = mesh.rest.copy()
    free = mesh.pinned == 0
    x[free] += 3e-4 * rng.standard_normal((int(free.sum()), 3))
    x[(mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free, 2] -= 0.0035
    with fsim.Context(0) as ctx:
        def at(kappa):
            m = ctx.upload(mesh)
            p = fsim.params_for(mesh)
            p.kappa = kappa
            m.prefactor(p)
            m.set_actuation(act.fiber, act.stretch)
            return m.eval_barrier(x)
        yield at


@pytest.mark.parametrize("kappa", [1e-60, 1e-28, 1e-12, 1e6, 1e24, 1e60])
def test_barrier_is_linear_in_kappa(terms, kappa):
    g1, c1, B1 = terms(1.0)
    g, c, B = terms(kappa)
    assert len(c1) > 20 and np.array_equal(c, c1)
    assert np.abs(g / kappa - g1).max() <= 1e-12 * np.abs(g1).max()
    assert np.abs(B / kappa - B1).max() <= 1e-12 * np.abs(B1).max()

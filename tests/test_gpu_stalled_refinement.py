"""Mixed global steps at pairs too close for a float32 reduced factor.

With a pair below about 1e-3 d0 the reduced system's cond(N) passes a few 1e6 and a
float32 factor no longer refines its solve, while all of its pivots stay positive.
Such a step is taken with float64 factors.  Steps at states of that kind, made on
slabs through every form of the reduced system and reached by frames of a pressed
face, are compared with the oracle's direct solve; whole frames of that face, alone
and in a batch, with the float64 frame.

Bound of a step.  The parts of a mixed step outside the reduced system (factor of
K11, Sigma^-1, their products, all float32) leave at most C u32 cond(H) max|dx_free|
with dx_free = -H^-1 g the contact-free step and C = 32 for the accumulations; the
reduced system's accepted residual rho, |rho| <= 1e-5 |y2|, reaches the step as
(Sigma + B)^-1 rho, so at most |rho| / lambda_min(H).
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle import solver as S
from paper_2312_02999_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
ACCEPTED = 1e-5          # |rho| / |y2|
# frames of the face from rest whose first twenty steps come to 5e-4 .. 2e-3 d0
FACE = dict(vertices=3212, index=23, seeds=[825331000 + i for i in (1, 3, 6, 7, 14, 15, 18, 20)])


@pytest.fixture(scope="module")
def fsim():
    from paper_2312_02999_gb300 import build, fsim as f
    build.build()
    return f


def _problem(mesh, act, kappa):
    pr = S.Problem(mesh.rest, mesh.tets, mesh.pinned, mesh.proxy_tris, mesh.W_rowptr, mesh.W_col,
                   mesh.W_val, S.Params(dhat=mesh.dhat, tol_abs=mesh.tol_abs, kappa=kappa,
                                        weight_scale=mesh.weight_scale), region=mesh.region)
    pr.set_actuation(act.fiber, act.stretch)
    return pr


def _check_step(fsim, m, pr, x):
    dx, path = m.eval_global_step(x, precision=fsim.MIXED, want_path=True)
    ev = pr.evaluate(x)
    g = pr.gradient(x, ev).ravel()[pr.free_dofs]
    H = pr.H.tocsc()
    ref = pr.global_step_direct(g, pr.free_part(pr.barrier_hessian(ev)))
    free = -spla.splu(H).solve(g)
    lmax = float(spla.eigsh(H, k=1, return_eigenvectors=False)[0])
    lmin = float(spla.eigsh(H, k=1, sigma=0.0, return_eigenvectors=False)[0])
    i1, i2 = pr.split_dofs()
    y2 = -g[i2] + H[i2][:, i1] @ spla.splu(H[i1][:, i1].tocsc()).solve(g[i1])
    bound = 32.0 * U32 * lmax / lmin * np.abs(free).max() + ACCEPTED * np.linalg.norm(y2) / lmin
    err = float(np.abs(dx.ravel()[pr.free_dofs] - ref).max())
    print("step", path, "err", err, "bound", bound, "max|dx|", np.abs(ref).max())
    assert err <= bound, (path, err, bound)
    return path


@pytest.mark.parametrize("closest", [1e-3, 2e-4])
@pytest.mark.parametrize("nx,one_cta_max", [(4, 0), (4, 32), (6, 0), (8, 0)])
def test_step_on_each_form(fsim, nx, one_cta_max, closest):
    # n_c = 50 on one CTA and on the cluster, 98 on the cluster, 162 in the grid form;
    # the slabs are pressed until the closest pair lies at the given part of d0
    mesh = I.two_slabs(nx, nx, 2, gap=0.004)
    act = I.slab_actuation(mesh, seed=11)
    rng = np.random.default_rng(9)
    x = mesh.rest.copy()
    free = mesh.pinned == 0
    x[free] += 3e-4 * rng.standard_normal((int(free.sum()), 3))
    top = (mesh.rest[:, 2] > mesh.rest[:, 2].mean()) & free
    x[top, 2] -= 0.0035
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh, reduced_one_cta_max=one_cta_max))
        m.set_actuation(act.fiber, act.stretch)
        pr = _problem(mesh, act, m.info()["kappa"])
        for _ in range(8):
            x[top, 2] -= pr.evaluate(x)["C"][3].min() - closest * mesh.dhat
        assert abs(pr.evaluate(x)["C"][3].min() / mesh.dhat - closest) <= 1e-2 * closest
        _check_step(fsim, m, pr, x)


@pytest.fixture(scope="module")
def face(fsim):
    mesh = I.face_shell(n_target=FACE["vertices"])
    field = I.bump_field(mesh, seed=2)
    acts = [I.bump_actuation(field, I.keyframe_coeffs(seed=s)[FACE["index"]]) for s in FACE["seeds"]]
    return mesh, acts


@pytest.mark.parametrize("frame,iterate", [(1, 12), (1, 17), (2, 12), (2, 13)])
def test_step_at_iterates_of_a_face(fsim, face, frame, iterate):
    mesh, acts = face
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh, max_iters=iterate))
        m.set_actuation(acts[frame].fiber, acts[frame].stretch)
        rc, _ = m.solve_frame(mesh.rest, precision=fsim.FP64, check=False)
        assert rc == fsim.FSIM_ENOT_CONVERGED
        _check_step(fsim, m, _problem(mesh, acts[frame], m.info()["kappa"]), m.positions())


def test_frames_end_where_the_float64_frame_does(fsim, face):
    # energies within 1e-9, positions within the mixed form's 1e-6 of the diagonal,
    # iterations within 2: steps that are wrong cost iterations before anything else
    mesh, acts = face
    diag = float(np.linalg.norm(mesh.rest.max(0) - mesh.rest.min(0)))
    with fsim.Context(0) as ctx:
        m = ctx.upload(mesh)
        m.prefactor(fsim.params_for(mesh))
        rc, xb, sb = fsim.solve_batch(ctx, [(m, a.fiber, a.stretch, None) for a in acts],
                                      max_frames=len(acts))
        assert rc == 0
        float64_steps = 0
        for i, a in enumerate(acts):
            m.set_actuation(a.fiber, a.stretch)
            _, s64 = m.solve_frame(mesh.rest, precision=fsim.FP64)
            x64 = m.positions()
            _, sm = m.solve_frame(mesh.rest, precision=fsim.MIXED)
            xm = m.positions()
            for how, x, s in (("alone", xm, sm), ("batch", xb[i], sb[i])):
                print(how, i, s["iterations"], s64["iterations"], s["fp64_steps"])
                assert abs(s["iterations"] - s64["iterations"]) <= 2, (how, i)
                assert abs(s["energy"] - s64["energy"]) <= 1e-9 * abs(s64["energy"]), (how, i)
                assert np.abs(x - x64).max() <= 1e-6 * diag, (how, i)
                float64_steps += s["fp64_steps"]
    assert float64_steps > 0       # the states this is about were met

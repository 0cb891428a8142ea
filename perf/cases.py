"""Performance cases of the actuated-face solver: what its users have it do.

A case is a dict of plain values.  ``listed()`` names the standing cases and
``draw(rng)`` gives further ones of the same ranges; ``prepare`` builds what a
caller holds before the call (a context with a prefactored mesh, a server,
actuations, start positions), ``run`` is one pass through the public Python
entry points, ``work`` the bytes and operations no implementation can avoid
and ``exact`` the same outputs in plain float64 numpy / torch.

Kinds of case
  frame    set_actuation + solve_frame + positions: one frame, host arrays
  batch    solve_batch: frames of one mesh in lock step, host arrays
  served   Server: requests with device inputs and outputs, all in flight
  elastic  eval_elastic: the local step alone (energy and forces)
  contact  eval_contacts + eval_barrier: constraint set, gradient, B-check
  step     eval_global_step + eval_ccd: one step and its collision bound
"""
import math
import weakref

import numpy as np
import torch

from paper_2312_02999_gb300 import fsim
from paper_2312_02999_gb300 import inputs

# iterations of Algorithm 1 a frame takes (about 90 on every workload here);
# only the estimates of work() use it
ITERATIONS = 90
# muscle directions and bump centres belong to the mesh, as in the benchmark
FIELD_SEED = 2


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # the smallest frame there is (the smoke test's mesh): all latency
        frame("slabs small frame float64", slabs(3, 3, 2), "float64"),
        # the two-slab lip-contact workload at its full size
        frame("slabs frame mixed", slabs(10, 10, 3), "mixed"),
        # one frame of a small face from the rest pose: interactive preview
        frame("face 5k frame mixed", face(5000), "mixed", index=20),
        # the next frame of a sequence on the full face, lips in contact:
        # single-sequence playback, warm-started from the frame before
        frame("face 30k frame mixed", face(30000), "mixed", index=21, warm=True),
        # the same in the reference precision
        frame("face 30k frame float64", face(30000), "float64", index=21, warm=True),
        # offline batches from rest: many poses of one small face ...
        batch("face 5k batch", face(5000), 16, index=20),
        # ... and a few of a detailed one
        batch("face 60k batch", face(60000), 8, index=20),
        # the serving workload: 96 sequences in lock-step batches of 32
        served("face 30k served", face(30000), 96, workers=3, batch_frames=32, index=21),
        # the local step alone, for a caller with its own outer loop
        elastic("face 30k local step mixed", face(30000), "mixed"),
        elastic("face 15k local step float64", face(15000), "float64"),
        # contact terms of pressed lips, for a caller with its own solver
        contact("face 30k contact terms", face(30000), 14.0),
        # one step with its collision bound, odd mesh size
        step("face 12k step float64", face(12347), 16.0),
    ]


def slabs(nx, ny, nz):
    return {"mesh": "slabs", "nx": nx, "ny": ny, "nz": nz, "embedded": 0}


def face(vertices):
    return {"mesh": "face", "vertices": vertices}


def frame(name, mesh, precision, index=0, warm=False, mollifier=False):
    return dict(mesh, name=name, kind="frame", precision=precision, index=index, warm=warm,
                mollifier=mollifier)


def batch(name, mesh, frames, index):
    return dict(mesh, name=name, kind="batch", precision="mixed", frames=frames, index=index,
                warm=False, mollifier=False)


def served(name, mesh, frames, workers, batch_frames, index):
    return dict(mesh, name=name, kind="served", precision="mixed", frames=frames, workers=workers,
                batch_frames=batch_frames, index=index, warm=True, mollifier=False)


def elastic(name, mesh, precision):
    return dict(mesh, name=name, kind="elastic", precision=precision, mollifier=False)


def contact(name, mesh, width):
    return dict(mesh, name=name, kind="contact", precision="float64", width=width, mollifier=False)


def step(name, mesh, width):
    return dict(mesh, name=name, kind="step", precision="float64", width=width, mollifier=False)


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def slab_mesh():
        m = slabs(rng.randint(3, 11), rng.randint(3, 11), rng.randint(2, 4))
        m["embedded"] = rng.choice([0, 0, 0, 1])   # sometimes a finer embedded proxy surface
        return m

    kind = rng.choice(["frame", "frame", "frame", "batch", "batch", "served", "elastic", "contact",
                       "step"])
    if kind == "frame":
        prec = rng.choice(["mixed", "mixed", "float64"])
        if rng.random() < 0.35:
            c = frame("", slab_mesh(), prec, mollifier=rng.random() < 0.2)
        else:
            c = frame("", face(spread(2000, 60000 if prec == "mixed" else 40000)), prec,
                      index=rng.randint(8, 28), warm=rng.random() < 0.5)
    elif kind == "batch":
        v = spread(2000, 60000)
        c = batch("", face(v), spread(2, min(40, 1000000 // v)), index=rng.randint(8, 28))
    elif kind == "served":
        v = spread(2000, 40000)
        n = spread(4, min(128, 2000000 // v))
        bf = rng.choice([0, 8, 16, 32])
        c = served("", face(v), n, workers=rng.randint(2, 8) if bf == 0 else rng.randint(1, 3),
                   batch_frames=bf, index=rng.randint(8, 28))
    elif kind == "elastic":
        c = elastic("", face(spread(2000, 60000)), rng.choice(["mixed", "float64"]))
    elif kind == "contact":
        c = contact("", face(spread(2000, 60000)), rng.uniform(5.0, 26.0))
    else:
        c = step("", face(spread(2000, 40000)), rng.uniform(5.0, 26.0))
    del c["name"]
    return c


# ----------------------------------------------------------------------------
# what a caller keeps: the mesh, its context and (served) its server
# ----------------------------------------------------------------------------
def build_mesh(case):
    if case["mesh"] == "slabs":
        m = inputs.two_slabs(case["nx"], case["ny"], case["nz"])
        return inputs.embed_finer_surface(m, levels=case["embedded"], relief=0.02) \
            if case["embedded"] else m
    return inputs.face_shell(n_target=case["vertices"])


class Program:
    """A long-running caller's handles: they outlive any single frame."""

    def __init__(self, case):
        self.mesh = build_mesh(case)
        self.field = inputs.bump_field(self.mesh, seed=FIELD_SEED) if case["mesh"] == "face" else None
        self.ctx = fsim.Context(0)
        self.handle = self.ctx.upload(self.mesh)
        self.handle.prefactor(fsim.params_for(self.mesh, ee_mollifier=int(case["mollifier"])))
        self.server = None
        if case["kind"] == "served":
            self.server = fsim.Server(self.ctx, workers=case["workers"],
                                      batch_frames=case["batch_frames"])

    def __del__(self):
        if getattr(self, "server", None) is not None:
            self.server.close()
        if getattr(self, "ctx", None) is not None:
            self.ctx.close()

    def actuation(self, case, seed, offset=0):
        if self.field is None:
            return inputs.slab_actuation(self.mesh, seed=seed)
        coeffs = inputs.keyframe_coeffs(seed=seed)
        return inputs.bump_actuation(self.field, coeffs[case["index"] + offset])


_programs = weakref.WeakValueDictionary()   # live programs, shared by the states of one case


def program(case):
    key = repr(sorted((k, case[k]) for k in ("mesh", "nx", "ny", "nz", "embedded", "vertices",
                                             "mollifier", "kind", "workers", "batch_frames")
                      if k in case))
    p = _programs.get(key)
    if p is None:
        p = _programs[key] = Program(case)
    return p


def precision(case):
    return fsim.MIXED if case["precision"] == "mixed" else fsim.FP64


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def deformed(mesh, seed):
    """A smooth expression-sized deformation (a few millimetres) with some noise."""
    rng = np.random.default_rng([seed, 1])
    x = mesh.rest.copy()
    for _ in range(8):
        c = mesh.rest[rng.integers(mesh.n)]
        bump = np.exp(-((mesh.rest - c) ** 2).sum(1) / (2.0 * rng.uniform(0.01, 0.03) ** 2))
        x += bump[:, None] * rng.uniform(-0.004, 0.004, 3)
    x += 2e-5 * rng.standard_normal(x.shape)
    x[mesh.pinned != 0] = mesh.rest[mesh.pinned != 0]
    return x


def pressed(mesh, width, seed):
    """Lips closed to a fraction of dhat over |phi| <= width degrees."""
    rng = np.random.default_rng([seed, 2])
    g = mesh.grid
    x = mesh.rest + 0.02 * mesh.dhat * rng.standard_normal(mesh.rest.shape)
    ids = {(i, j, k): v for v, (i, j, k) in enumerate(zip(g["gi"].tolist(), g["gj"].tolist(),
                                                          g["gk"].tolist()))}
    for i, phi in enumerate(np.linspace(-80.0, 80.0, g["nphi"])):
        if abs(phi) > width:
            continue
        for k in range(3):                       # the layers the slit cuts through
            lo, up = ids.get((i, g["jm"], k)), ids.get((i, g["jm"] + 1, k))
            if lo is None or up is None:
                continue
            d = x[up] - x[lo]
            gap = mesh.dhat * rng.uniform(0.35, 0.85)
            shift = 0.5 * (1.0 - gap / np.linalg.norm(d)) * d
            x[lo] += shift
            x[up] -= shift
    x[mesh.pinned != 0] = mesh.rest[mesh.pinned != 0]
    return x


def prepare(case, seed):
    p = program(case)
    state = {"case": case, "program": p}
    kind = case["kind"]
    if kind == "elastic":
        a = inputs.bump_actuation(p.field, inputs.keyframe_coeffs(seed=seed)[20])
        p.handle.set_actuation(a.fiber, a.stretch)
        state.update(act=a, x=deformed(p.mesh, seed))
    elif kind in ("contact", "step"):
        a = inputs.bump_actuation(p.field, inputs.keyframe_coeffs(seed=seed)[20])
        p.handle.set_actuation(a.fiber, a.stretch)
        state.update(act=a, x=pressed(p.mesh, case["width"], seed))
    elif kind == "frame":
        state["act"] = p.actuation(case, seed)
        state["x_init"] = p.mesh.rest
        if case["warm"]:                         # the sequence's frame before, already solved
            b = p.actuation(case, seed, offset=-1)
            p.handle.set_actuation(b.fiber, b.stretch)
            p.handle.solve_frame(p.mesh.rest, precision=precision(case), check=False)
            state["x_init"] = p.handle.positions()
    elif kind == "batch":
        state["requests"] = []
        for i in range(case["frames"]):
            a = p.actuation(case, 1000 * seed + i)
            state["requests"].append((p.handle, a.fiber, a.stretch, None))
    else:                                        # served: device-resident inputs and outputs
        fiber = torch.from_numpy(p.field.fiber).cuda()
        rest = torch.from_numpy(p.mesh.rest).cuda()
        n = case["frames"]
        stretch, before = ([torch.from_numpy(p.actuation(case, 1000 * seed + i, offset=o).stretch)
                            .cuda() for i in range(n)] for o in (0, -1))
        x_init = [torch.empty_like(rest) for _ in range(n)]
        torch.cuda.synchronize()
        tickets = [p.server.submit_dev(p.handle, fiber.data_ptr(), before[i].data_ptr(),
                                       rest.data_ptr(), x_init[i].data_ptr(), precision(case))
                   for i in range(n)]
        for t in tickets:
            p.server.wait(t)
        state.update(fiber=fiber, stretch=stretch, x_init=x_init,
                     x_out=[torch.empty_like(rest) for _ in range(n)])
        torch.cuda.synchronize()
    return state


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def run(state):
    case, p = state["case"], state["program"]
    kind, prec = case["kind"], precision(case)
    if kind == "frame":
        a = state["act"]
        p.handle.set_actuation(a.fiber, a.stretch)
        status, st = p.handle.solve_frame(state["x_init"], precision=prec, check=False)
        return {"x": p.handle.positions(), "energy": st["energy"], "status": status}
    if kind == "batch":
        status, x, st = fsim.solve_batch(p.ctx, state["requests"], max_frames=len(state["requests"]))
        return {"x": np.stack(x), "energy": np.array([s["energy"] for s in st]), "status": status}
    if kind == "served":
        tickets = [p.server.submit_dev(p.handle, state["fiber"].data_ptr(), s.data_ptr(),
                                       x0.data_ptr(), x1.data_ptr(), prec)
                   for s, x0, x1 in zip(state["stretch"], state["x_init"], state["x_out"])]
        got = [p.server.wait(t) for t in tickets]
        return {"x": torch.stack(state["x_out"]), "energy": np.array([g[2]["energy"] for g in got]),
                "status": np.array([g[0] for g in got])}
    if kind == "elastic":
        a = state["act"]
        p.handle.set_actuation(a.fiber, a.stretch)
        energy, grad = p.handle.eval_elastic(state["x"], precision=prec)
        return {"energy": energy, "grad": grad}
    if kind == "contact":
        pairs, energy = p.handle.eval_contacts(state["x"])
        grad, clist, bcheck = p.handle.eval_barrier(state["x"])
        return {"pairs": pairs, "energy": energy, "grad": grad, "clist": clist, "bcheck": bcheck}
    a = state["act"]
    p.handle.set_actuation(a.fiber, a.stretch)
    dx = p.handle.eval_global_step(state["x"], precision=prec)
    return {"dx": dx, "alpha": p.handle.eval_ccd(state["x"], dx)}


# ----------------------------------------------------------------------------
# what no implementation can avoid
# ----------------------------------------------------------------------------
def work(case):
    if case["mesh"] == "slabs":
        cells = 2 * case["nx"] * case["ny"] * case["nz"]
        n = 2.0 * (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        tets = 6.0 * cells
        n2 = 2.0 * (case["nx"] + 1) * (case["ny"] + 1)
    else:
        n = float(case["vertices"])
        tets, n2 = 4.95 * n, 0.048 * n
    factor = 18.0 * n * math.log2(n)             # stored entries of the sparse factor
    # per iteration: polar rotation, products, energy and forces of a tet
    # (about 700 operations); both substitutions for three right-hand sides;
    # the dense Schur inverse times three right-hand sides
    local, solve = 700.0 * tets, 12.0 * factor + 6.0 * n2 * n2
    mesh = tets * (16 + 80) + n * 24             # connectivity, rest shapes and weights, rest positions
    actuation, positions = tets * 32, n * 24
    entry = 4 if case["precision"] == "mixed" else 8
    kind = case["kind"]
    if kind == "elastic":
        return {"bytes": mesh + actuation + 2 * positions, "flops": local}
    if kind == "contact":
        nc = contact_vertices(case)
        return {"bytes": 2 * positions + 8 * 9 * nc * nc, "flops": 30.0 * nc * 2000}
    if kind == "step":
        nc = contact_vertices(case)
        return {"bytes": mesh + actuation + 2 * positions + entry * (factor + n2 * n2),
                "flops": local + solve + 14.0 * nc ** 3}
    frames = case.get("frames", 1)
    return {"bytes": mesh + frames * (actuation + 2 * positions) + entry * (factor + n2 * n2),
            "flops": frames * ITERATIONS * (local + solve)}


def contact_vertices(case):
    # vertices of both lips over 2 x width degrees, three layers deep
    nphi = math.sqrt(case["vertices"] / 7.0 * 80.0 / 54.0)
    return 6.0 * max(1.0, 2.0 * case["width"] / 160.0 * nphi)


# ----------------------------------------------------------------------------
# the same outputs in plain float64
# ----------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind not in ("elastic", "contact", "step"):
        # a whole frame: ninety factorisations of the contact system, minutes on the host
        return None
    mesh = build_mesh(case)
    field = inputs.bump_field(mesh, seed=FIELD_SEED)
    act = inputs.bump_actuation(field, inputs.keyframe_coeffs(seed=seed)[20])
    if kind == "elastic":
        energy, grad, _, _ = elastic_terms(mesh, act, deformed(mesh, seed))
        return {"energy": energy, "grad": grad}
    x = pressed(mesh, case["width"], seed)
    _, egrad, grads, weight = elastic_terms(mesh, act, x)
    free = np.nonzero(mesh.pinned == 0)[0]
    diag = np.bincount(mesh.tets.ravel(), weights=(weight[:, None] * (grads ** 2).sum(2)).ravel(),
                       minlength=mesh.n)
    kappa = diag[free].mean()
    # the proxy of the face meshes selects mesh vertices
    vert = mesh.W_col.astype(np.int64)
    groups = active_pairs(x[vert], mesh.proxy_tris.astype(np.int64), mesh.dhat)
    energy, bgrad, blocks = 0.0, np.zeros((mesh.n, 3)), []
    for dist, idx in groups:
        y = torch.from_numpy(x[vert[idx]].reshape(len(idx), 12))

        def term(v, dist=dist):
            d = dist(v.reshape(4, 3))
            return -kappa * (d - mesh.dhat) ** 2 * torch.log(d / mesh.dhat)

        energy += float(torch.func.vmap(term)(y).sum())
        np.add.at(bgrad, vert[idx].reshape(-1),
                  torch.func.vmap(torch.func.grad(term))(y).numpy().reshape(-1, 3))
        if kind == "step":
            lam, q = torch.linalg.eigh(torch.func.vmap(torch.func.hessian(term))(y))
            blocks.append((vert[idx], ((q * lam.clamp(min=0.0)[:, None, :]) @ q.mT).numpy()))
    bgrad[mesh.pinned != 0] = 0.0
    if kind == "contact":
        return {"pairs": None, "energy": energy, "grad": bgrad, "clist": None, "bcheck": None}
    if len(free) > 14000:                        # the dense factorisation below
        return None
    return {"dx": contact_step(mesh, free, grads, weight, egrad + bgrad, blocks), "alpha": None}


def elastic_terms(mesh, act, x):
    """Energy, gradient (zero at pinned vertices), shape gradients and weights of the tets."""
    t = mesh.tets
    dm = np.swapaxes(mesh.rest[t[:, 1:]] - mesh.rest[t[:, :1]], 1, 2)
    inv = np.linalg.inv(dm)
    weight = mesh.weight_scale * np.linalg.det(dm) / 6.0
    grads = np.concatenate([-inv.sum(1, keepdims=True), inv], axis=1)      # (T, 4, 3)
    f = np.swapaxes(x[t[:, 1:]] - x[t[:, :1]], 1, 2) @ inv
    fib = act.fiber / np.linalg.norm(act.fiber, axis=1, keepdims=True)
    ff = fib[:, :, None] * fib[:, None, :]
    a = act.stretch[:, None, None]
    amat = a * ff + (np.eye(3) - ff) / np.sqrt(a)
    u, _, vt = np.linalg.svd(f @ amat)
    u[:, :, 2] *= np.sign(np.linalg.det(u @ vt))[:, None]
    d = f - u @ vt @ amat
    energy = float(0.5 * (weight * (d ** 2).sum((1, 2))).sum())
    force = weight[:, None, None] * (grads @ np.swapaxes(d, 1, 2))
    grad = np.stack([np.bincount(t.ravel(), weights=force[:, :, c].ravel(), minlength=mesh.n)
                     for c in range(3)], axis=1)
    grad[mesh.pinned != 0] = 0.0
    return energy, grad, grads, weight


def point_point(y):
    return torch.linalg.vector_norm(y[0] - y[1])


def point_line(y):
    e = y[2] - y[1]
    return torch.linalg.vector_norm(torch.linalg.cross(y[0] - y[1], e)) / torch.linalg.vector_norm(e)


def point_plane(y):
    n = torch.linalg.cross(y[2] - y[1], y[3] - y[1])
    return torch.abs(((y[0] - y[1]) * n).sum()) / torch.linalg.vector_norm(n)


def line_line(y):
    n = torch.linalg.cross(y[1] - y[0], y[3] - y[2])
    return torch.abs(((y[2] - y[0]) * n).sum()) / torch.linalg.vector_norm(n)


def segment_parameter(p, a, b):
    e = b - a
    return np.clip(((p - a) * e).sum(1) / (e * e).sum(1), 0.0, 1.0)


def active_pairs(s, tris, dhat):
    """Pairs closer than dhat by closest feature: (distance function, (k, 4) proxy vertices)."""
    edges = np.unique(np.sort(np.concatenate([tris[:, [0, 1]], tris[:, [1, 2]], tris[:, [2, 0]]]), 1),
                      axis=0)

    def boxes(prims):
        c = s[prims]
        return c.min(1), c.max(1)

    def overlapping(a, b):
        (alo, ahi), (blo, bhi) = a, b
        near = np.ones((len(alo), len(blo)), dtype=bool)
        for c in range(3):
            near &= alo[:, c, None] - dhat <= bhi[None, :, c]
            near &= blo[None, :, c] - dhat <= ahi[:, c, None]
        return np.nonzero(near)

    found = {point_point: [], point_line: [], point_plane: [], line_line: []}

    def put(dist, mask, *cols):
        # a feature of fewer than four vertices: the rest repeat the first and have no weight
        cols = list(cols) + [cols[0]] * (4 - len(cols))
        found[dist].append(np.stack(cols, 1)[mask])

    # point-triangle
    v, t = overlapping((s, s), boxes(tris))
    own = (tris[t] == v[:, None]).any(1)
    v, t = v[~own], tris[t[~own]]
    p, a, b, c = s[v], s[t[:, 0]], s[t[:, 1]], s[t[:, 2]]
    m = np.stack([b - a, c - a], 2)
    lam = np.linalg.solve(np.swapaxes(m, 1, 2) @ m, np.swapaxes(m, 1, 2) @ (p - a)[:, :, None])[:, :, 0]
    inside = (lam[:, 0] > 0) & (lam[:, 1] > 0) & (lam.sum(1) < 1)
    plane = np.linalg.norm(p - a - (m @ lam[:, :, None])[:, :, 0], axis=1)
    put(point_plane, inside & (plane < dhat), v, t[:, 0], t[:, 1], t[:, 2])
    sides = [(0, 1), (1, 2), (2, 0)]
    par = np.stack([segment_parameter(p, s[t[:, i]], s[t[:, j]]) for i, j in sides], 1)
    dist = np.stack([np.linalg.norm(p - s[t[:, i]] - par[:, k, None] * (s[t[:, j]] - s[t[:, i]]), axis=1)
                     for k, (i, j) in enumerate(sides)], 1)
    side = dist.argmin(1)
    rows = np.arange(len(v))
    hit = ~inside & (dist[rows, side] < dhat)
    q = par[rows, side]
    ends = np.array(sides)[side]
    e0, e1 = t[rows, ends[:, 0]], t[rows, ends[:, 1]]
    put(point_line, hit & (q > 0) & (q < 1), v, e0, e1)
    put(point_point, hit & (q == 0), v, e0)
    put(point_point, hit & (q == 1), v, e1)
    # edge-edge
    i, j = overlapping(boxes(edges), boxes(edges))
    keep = (i < j) & ~(edges[i][:, :, None] == edges[j][:, None, :]).any((1, 2))
    ea, eb = edges[i[keep]], edges[j[keep]]
    p0, p1, q0, q1 = s[ea[:, 0]], s[ea[:, 1]], s[eb[:, 0]], s[eb[:, 1]]
    d1, d2, r = p1 - p0, q1 - q0, p0 - q0
    aa, bb, cc = (d1 * d1).sum(1), (d1 * d2).sum(1), (d2 * d2).sum(1)
    den = aa * cc - bb * bb
    sp = ((bb * (d2 * r).sum(1)) - cc * (d1 * r).sum(1)) / np.where(den > 0, den, 1.0)
    tp = (bb * sp + (d2 * r).sum(1)) / cc
    inner = (den > 1e-10 * aa * cc) & (sp > 0) & (sp < 1) & (tp > 0) & (tp < 1)
    lines = np.linalg.norm(p0 + sp[:, None] * d1 - q0 - tp[:, None] * d2, axis=1)
    put(line_line, inner & (lines < dhat), ea[:, 0], ea[:, 1], eb[:, 0], eb[:, 1])
    quads = [(ea[:, 0], eb), (ea[:, 1], eb), (eb[:, 0], ea), (eb[:, 1], ea)]
    par = np.stack([segment_parameter(s[v], s[e[:, 0]], s[e[:, 1]]) for v, e in quads], 1)
    dist = np.stack([np.linalg.norm(s[v] - s[e[:, 0]] - par[:, k, None] * (s[e[:, 1]] - s[e[:, 0]]), axis=1)
                     for k, (v, e) in enumerate(quads)], 1)
    best = dist.argmin(1)
    for k, (v, e) in enumerate(quads):
        hit = ~inner & (best == k) & (dist[:, k] < dhat)
        put(point_line, hit & (par[:, k] > 0) & (par[:, k] < 1), v, e[:, 0], e[:, 1])
        put(point_point, hit & (par[:, k] == 0), v, e[:, 0])
        put(point_point, hit & (par[:, k] == 1), v, e[:, 1])
    got = [(f, np.concatenate(idx)) for f, idx in found.items()]
    return [(f, idx) for f, idx in got if len(idx)]


def contact_step(mesh, free, grads, weight, grad, blocks):
    """dx of (K x I3 + B) dx = -grad: dense factor of K, then the contact vertices' system."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    pos = -np.ones(mesh.n, dtype=np.int64)
    pos[free] = np.arange(len(free))
    local = weight[:, None, None] * (grads @ np.swapaxes(grads, 1, 2))
    rows, cols = np.repeat(pos[mesh.tets], 4, axis=1).ravel(), np.tile(pos[mesh.tets], (1, 4)).ravel()
    ok = (rows >= 0) & (cols >= 0)
    k = torch.zeros(len(free) ** 2, dtype=torch.float64, device=dev)
    k.index_add_(0, torch.from_numpy(rows[ok] * len(free) + cols[ok]).to(dev),
                 torch.from_numpy(local.ravel()[ok]).to(dev))
    chol = torch.linalg.cholesky(k.view(len(free), len(free)))
    rhs = torch.from_numpy(-grad[free]).to(dev)
    dx = torch.cholesky_solve(rhs, chol)
    touched = sorted({int(v) for vs, _ in blocks for v in vs.ravel() if pos[v] >= 0})
    if touched:
        place = {v: c for c, v in enumerate(touched)}
        nc = len(touched)
        b = np.zeros((nc, 3, nc, 3))
        for vs, hs in blocks:
            for v4, h in zip(vs, hs.reshape(-1, 4, 3, 4, 3)):
                for i in range(4):
                    for j in range(4):
                        if int(v4[i]) in place and int(v4[j]) in place:
                            b[place[int(v4[i])], :, place[int(v4[j])], :] += h[i, :, j, :]
        b = torch.from_numpy(b.reshape(3 * nc, 3 * nc)).to(dev)
        c = torch.from_numpy(pos[touched]).to(dev)
        sel = torch.zeros(len(free), nc, dtype=torch.float64, device=dev)
        sel[c, torch.arange(nc, device=dev)] = 1.0
        kinv = torch.cholesky_solve(sel, chol)                       # K^-1[:, c]
        s = torch.kron(kinv[c], torch.eye(3, dtype=torch.float64, device=dev))
        v = torch.linalg.solve(torch.eye(3 * nc, dtype=torch.float64, device=dev) + b @ s,
                               b @ dx[c].reshape(-1))
        dx = dx - kinv @ v.reshape(nc, 3)
    out = np.zeros((mesh.n, 3))
    out[free] = dx.cpu().numpy()
    return out

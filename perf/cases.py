"""Performance cases: what a user of this framework has it do, through its public entry points.

A case is one call or a short run of calls on one robot (or one batch of robots), with the positions left on the GPU:

* ``contacts``: the allocation-free contact check of a control loop (``casim_contacts_noalloc``);
* ``run``: a whole simulation, reset to the initial shape and ``step(n)``;
* ``adjoint``: gradient of a loss on tip positions with respect to the chamber ratios, forward and reverse pass
  through ``actuation_to_positions``.

Robots are the pneumatic fingers, the gripper, the batch and the beam of ``synth``.  A ``run`` starts either from the
rest shape or from a seeded contact-bearing shape (``contact``): the teeth of every finger swollen into their
neighbours by a fraction of a voxel plus a little noise, as they are after the first iterations of an actuation.

In MIXED precision a contact decision on a computed position can fall either way within the solver's tolerance, and the
trajectories that follow differ by more than rounding; runs of many iterations with contacts are therefore listed at
the sizes where these differences stay small, and the larger robots with one iteration from a contact-bearing shape,
where every decision is taken on given positions.  The adjoint runs in FP64: a MIXED gradient is only as good as the
solver's tolerance, about 1e-4.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2203_02054_gb300 import casim, synth

H = 0.5  # voxel edge of every synthetic robot, cm


# ------------------------------------------------------------------ the cases
def _finger(name, nx, ny, nz, n_ch, n, **kw):
    c = dict(name=name, kind="run", robot="finger", nx=nx, ny=ny, nz=nz, n_ch=n_ch, n=n, fp64=False, contact=False,
             trees=False)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: one contact check of a small finger inside a control loop that may not allocate.
        dict(name="contacts_20x4x4", kind="contacts", nx=20, ny=4, nz=4, n_ch=4),
        # The cantilever beam, all FP64, no collision, its 50 iterations: a small accurate solve, latency only.
        dict(name="beam_fp64_50it", kind="run", robot="beam", nx=20, ny=4, nz=4, n=50, fp64=True, contact=False,
             trees=False),
        # The small finger of the tests, MIXED with self collision: a short interactive run, latency and launches.
        _finger("finger_20x4x4_10it", 20, 4, 4, 4, 10),
        # The bending finger (51,840 tets), 50 iterations from rest: the ordinary single-robot simulation.
        _finger("finger_60x12x12_50it", 60, 12, 12, 8, 50),
        # A ragged mid-size finger (odd cross-section), as a user's own robot would be.
        _finger("finger_45x9x11_contact", 45, 9, 11, 5, 1, contact=True),
        # One collision-laden iteration of the three-finger gripper with plate and sphere (193,920 tets).
        dict(name="gripper_contact", kind="run", robot="gripper", n=1, fp64=False, contact=True, trees=False),
        # The largest single robot (983,040 tets), one collision-laden iteration.
        _finger("finger_160x32x32_contact", 160, 32, 32, 16, 1, contact=True),
        # A batch of 24 uneven fingers in one simulation (about 0.9 million tets), one collision-laden iteration.
        dict(name="batch24_contact", kind="run", robot="batch", robots=24, mix=1004, n=1, fp64=False, contact=True,
             trees=False),
        # The bending finger in FP64 with self collision: the accurate mode, three iterations with springs kept,
        # re-targeted and released.
        _finger("finger_60x12x12_fp64_3it", 60, 12, 12, 8, 3, fp64=True, contact=True),
        # The paper's own broad phase (AABB trees, refitted) with a rigid tetrahedral obstacle at the tip.
        _finger("finger_60x12x12_trees", 60, 12, 12, 8, 1, contact=True, trees=True),
        # Gradient of a tip-position loss with respect to 16 chamber ratios through four iterations, FP64, on the
        # 20,736-tet copy of the adjoint workload.
        dict(name="adjoint_96x6x6_fp64", kind="adjoint", nx=96, ny=6, nz=6, n_ch=16, n=4, every=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_finger(rng, max_voxels):
    """A finger of the listed proportions with a ragged cross-section: 20..160 voxels long, 4..32 wide and high."""
    while True:
        nx = _log_int(rng, 20, 160)
        ny = max(4, min(32, int(nx * rng.uniform(0.12, 0.24))))
        nz = max(4, min(32, ny + rng.randint(-1, 2)))
        top = synth.max_chambers(nx, ny, nz)
        if nx * ny * nz <= max_voxels and top >= 2:
            return dict(nx=nx, ny=ny, nz=nz, n_ch=rng.randint(2, min(top, 16)))


def draw(rng):
    kind = rng.choice(["contacts", "beam", "finger", "finger", "contact", "contact", "contact", "batch", "fp64",
                       "trees", "adjoint"])
    if kind == "contacts":
        return dict(kind="contacts", **_draw_finger(rng, 10000))
    if kind == "beam":
        return dict(kind="run", robot="beam", nx=rng.randint(10, 20), ny=rng.randint(3, 4), nz=rng.randint(3, 4),
                    n=rng.randint(10, 50), fp64=True, contact=False, trees=False)
    if kind == "finger":
        return dict(kind="run", robot="finger", n=rng.randint(5, 20), fp64=False, contact=False, trees=False,
                    **_draw_finger(rng, 8640))
    if kind == "contact":
        return dict(kind="run", robot="finger", n=1, fp64=False, contact=True, trees=False,
                    **_draw_finger(rng, 163840))
    if kind == "batch":
        return dict(kind="run", robot="batch", robots=_log_int(rng, 2, 24), mix=rng.randint(1, 9999), n=1,
                    fp64=False, contact=True, trees=False)
    if kind == "fp64":
        return dict(kind="run", robot="finger", n=rng.randint(1, 3), fp64=True, contact=True, trees=False,
                    **_draw_finger(rng, 8640))
    if kind == "trees":
        return dict(kind="run", robot="finger", n=1, fp64=False, contact=True, trees=True,
                    **_draw_finger(rng, 8640))
    return dict(kind="adjoint", n=rng.randint(2, 4), every=rng.randint(1, 3), **_draw_finger(rng, 3456))


# ------------------------------------------------------------------- inputs
def _swell(rest, nx, ny, nz, n_ch, amount):
    """Displacement along the finger that swells every tooth by ``amount`` at its tip, so that it enters its neighbours
    across the slits (none at the spine)."""
    lay = synth.finger_layout(nx, ny, nz, n_ch)
    x, z = np.rint(rest[:, 0] / H), np.rint(rest[:, 2] / H)
    second = np.arange(rest.shape[0]) >= (nx + 1) * (ny + 1) * (nz + 1)  # the far side's copies of slit vertices
    edges = np.array([0] + lay["slits"] + [nx], dtype=np.float64)
    tooth = np.zeros(rest.shape[0], dtype=np.int64)
    for p in lay["slits"]:
        tooth += (x > p) | (second & (x == p))
    mid, half = (edges[tooth] + edges[tooth + 1]) / 2, (edges[tooth + 1] - edges[tooth]) / 2
    up = np.clip((z - lay["s"]) / (nz - lay["s"]), 0.0, 1.0)
    return amount * up * (x - mid) / half


def _contact_shape(meshes, case, rng):
    """Seeded contact-bearing positions of the robots (rest + swollen teeth + noise of 1/50 voxel)."""
    out = []
    for m in meshes:
        X = m.rest.copy()
        if case["robot"] == "gripper":
            local = synth.finger_mesh(60, 12, 12, 8)[0]
            k = local.shape[0]
            for f in range(3):  # the fingers hang: their length runs along -z
                X[f * k:(f + 1) * k, 2] -= _swell(local, 60, 12, 12, 8, rng.uniform(0.1, 0.25) * H)
        else:
            n = np.rint(m.rest.max(axis=0) / H).astype(int)
            X[:, 0] += _swell(m.rest, n[0], n[1], n[2], m.n_groups, rng.uniform(0.1, 0.25) * H)
        X += rng.uniform(-0.02 * H, 0.02 * H, size=X.shape)
        fixed = m.fixed.astype(bool)
        X[fixed] = m.rest[fixed]
        out.append(X)
    return np.concatenate(out)


def _scene(case, seed):
    """(meshes, batch, initial positions or None) of a case: the robots with seeded ratios, and where they start."""
    rng = np.random.default_rng([2203, int(seed)])
    key = int(rng.integers(1 << 62))
    robot = case.get("robot", "finger")
    if robot == "batch":
        meshes = synth.config4_batch(n_robots=case["robots"], seed=case["mix"])  # the mix of sizes
        for m in meshes:
            m.alpha = rng.uniform(1.2, 2.5, size=m.n_groups)
    elif robot == "gripper":
        m = synth.config3_gripper(seed=key)
        m.spheres[:, :2] *= 1.0 + 0.3 / np.linalg.norm(m.spheres[0, :2])  # the finger has closed onto the sphere
        meshes = [m]
    elif robot == "beam":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        m = synth.config1_beam()
        m.rest, m.tets, m.group, m.fixed = synth._voxel_kuhn(
            nx, ny, nz, H, group_of_voxel=lambda i, j, k: 0 if k == nz - 1 else -1)
        m.alpha = np.array([rng.uniform(1.2, 1.4)])
        meshes = [m]
    else:
        meshes = [synth.config2_finger(case["nx"], case["ny"], case["nz"], case["n_ch"], seed=key)]
    m = meshes[0]
    if case.get("trees"):
        top = m.rest.max(axis=0)
        m.obstacle_X, m.obstacle_tets = synth.box_obstacle(
            4, 8, 4, H, top * (0.85, 0.5, 1.0) - (0.0, 1.0, 0.4 * H), dtype=np.float32)
        m.collision = synth.COLLISION_SELF_OBSTACLE
    fp64 = case.get("fp64", case["kind"] == "adjoint")
    for q in meshes:
        q.precision = synth.PRECISION_FP64 if fp64 else synth.PRECISION_MIXED
    X0 = None
    if case.get("contact") or case["kind"] == "contacts":
        X0 = _contact_shape(meshes, dict(case, robot=robot), rng)
        if not fp64:
            X0 = X0.astype(np.float32).astype(np.float64)
    return meshes, robot == "batch", X0


def _tips(m, seed):
    """Loss vertices (the tip face) and their seeded targets."""
    tips = np.nonzero(m.rest[:, 0] == m.rest[:, 0].max())[0]
    return tips, m.rest[tips] + np.random.default_rng([64, int(seed)]).normal(size=(tips.size, 3))


def prepare(case, seed):
    meshes, batch, X0 = _scene(case, seed)
    m = meshes[0]
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "contacts":
        bnd = _Body(meshes).query.cpu().numpy()
        xyz = torch.tensor(X0, dtype=torch.float32, device="cuda")
        return dict(kind="contacts", m=m, xyz=xyz, tets=torch.tensor(m.tets, dtype=torch.int32, device="cuda"),
                    query=torch.tensor(bnd, dtype=torch.int32, device="cuda"), stream=stream)
    sim = casim.Sim(meshes if batch else m, stream=stream, broad_phase=1 if case.get("trees") else None)
    if X0 is not None:
        sim.set_positions(X0)
    st = dict(kind=case["kind"], sim=sim, n=case["n"])
    if case["kind"] == "adjoint":
        tips, targets = _tips(m, seed)
        st.update(alpha=m.alpha, tips=torch.from_numpy(tips), targets=torch.from_numpy(targets), every=case["every"])
    return st


# --------------------------------------------------------------------- runs
def run(state):
    if state["kind"] == "contacts":
        m, q = state["m"], state["query"]
        count = torch.empty(q.numel(), dtype=torch.int32, device="cuda")
        tets = torch.full((q.numel(), 8), -1, dtype=torch.int32, device="cuda")
        rc = casim.casim_contacts_noalloc(m.n_verts, state["xyz"].data_ptr(), m.n_tets, state["tets"].data_ptr(),
                                          q.numel(), q.data_ptr(), m.cell_size, 8, count.data_ptr(), tets.data_ptr(),
                                          state["stream"])
        if rc != casim.CASIM_OK:
            raise RuntimeError("contact check: %d" % rc)
        return {"count": count, "tets": tets}
    sim = state["sim"]
    if state["kind"] == "adjoint":
        alpha = torch.tensor(state["alpha"], requires_grad=True)
        X = casim.actuation_to_positions(sim, alpha, state["n"], state["every"])
        ((X[state["tips"]] - state["targets"]) ** 2).sum().backward()
        return {"x": X.detach(), "grad": alpha.grad}
    sim.reset()
    sim.step(state["n"])
    n_v = sim.sizes["n_verts"]
    x = torch.empty((n_v, 3), device="cuda",
                    dtype=torch.float64 if sim.params.precision == casim.CASIM_FP64 else torch.float32)
    casim.casim_get_positions(sim.h, n_v, x.data_ptr())
    return {"x": x}


def work(case):
    """Bytes: element records (4 indices, the centred rest shape, weight, volume, norm, group), the matrix (about 12
    off-diagonals a row), initial and final positions, each once.  Operations of one iteration: about 1,200 per
    element (rotation, target, scatter) and one matrix-vector product; a reverse iteration about twice that."""
    n_t, n_v = _sizes(case)
    if case["kind"] == "contacts":
        return {"bytes": 16 * n_t + 12 * n_v + 36 * n_v / 2, "flops": 100.0 * n_t}
    w = 8 if case.get("fp64", case["kind"] == "adjoint") else 4
    per_it = 1200.0 * n_t + 6 * 13 * n_v
    return {"bytes": n_t * (16 + 16 * w) + n_v * (12 * (4 + w) + 6 * w),
            "flops": per_it * case["n"] * (4 if case["kind"] == "adjoint" else 1)}


def _sizes(case):
    """Tets and vertices of a case (without the slits' second copies; the mean robot of a batch)."""
    robot = case.get("robot", "finger")
    if robot == "gripper":
        return 193920, 41789
    if robot == "batch":  # (20k, 4k, 4k) voxels, k ~ U{1..4}: 1,920 k^3 tets
        return 48000 * case["robots"], 10500 * case["robots"]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return 6 * nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1)


# ---------------------------------------------------- the loop in 64-bit torch
class _Body:
    """One mesh (or a batch of robots as one mesh) in FP64 torch: rest data, boundary, Laplacian."""

    FACES = ((1, 2, 3), (0, 3, 2), (0, 1, 3), (0, 2, 1))  # outward faces of a positively oriented tet

    def __init__(self, meshes, dev="cuda"):
        off = np.cumsum([0] + [m.n_verts for m in meshes])
        goff = np.cumsum([0] + [m.n_groups for m in meshes])
        t64 = dict(dtype=torch.float64, device=dev)
        self.rest = torch.tensor(np.concatenate([m.rest for m in meshes]), **t64)
        self.tets = torch.tensor(np.concatenate([m.tets + o for m, o in zip(meshes, off)]), dtype=torch.long, device=dev)
        self.group = torch.tensor(np.concatenate([np.where(m.group >= 0, m.group + o, -1)
                                                  for m, o in zip(meshes, goff)]), dtype=torch.long, device=dev)
        self.fixed = torch.tensor(np.concatenate([m.fixed for m in meshes]), device=dev).bool()
        self.alpha = torch.tensor(np.concatenate([m.alpha for m in meshes]), **t64)
        self.robot = torch.tensor(np.repeat(np.arange(len(meshes)), [m.n_tets for m in meshes]), device=dev)
        n_v, n_t = self.rest.shape[0], self.tets.shape[0]
        E = self.rest[self.tets]
        self.Tc = E - E.mean(1, keepdim=True)
        self.vol = _volume(E)
        mean = torch.zeros(len(meshes), **t64).index_add_(0, self.robot, self.vol) / torch.bincount(self.robot)
        self.omega = self.vol / mean[self.robot]
        # boundary faces, ordered by (tet, local face)
        f = torch.stack([self.tets[:, list(k)] for k in self.FACES], 1).reshape(-1, 3)
        key = f.sort(1).values
        _, inv, cnt = torch.unique((key[:, 0] * n_v + key[:, 1]) * n_v + key[:, 2], return_inverse=True,
                                   return_counts=True)
        keep = cnt[inv] == 1
        self.faces = f[keep]
        self.face_robot = self.robot.repeat_interleave(4)[keep]
        surf = torch.zeros(n_v, dtype=torch.bool, device=dev)
        surf[self.faces.reshape(-1)] = True
        self.query = torch.nonzero(surf & ~self.fixed)[:, 0]
        vrobot = torch.zeros(n_v, dtype=torch.long, device=dev)
        vrobot[self.tets.reshape(-1)] = self.robot.repeat_interleave(4)
        self.vert_robot = vrobot
        # Laplacian 3/4 w on the diagonal, -1/4 w per element edge
        a = self.tets.repeat_interleave(4, 1).reshape(-1)
        b = self.tets.repeat(1, 4).reshape(-1)
        v = self.omega.repeat_interleave(16) * torch.where(a == b, 0.75, -0.25).to(torch.float64)
        L = torch.sparse_coo_tensor(torch.stack([a, b]), v, (n_v, n_v)).coalesce()
        i, j = L.indices()
        self.diag = torch.zeros(n_v, **t64).index_add_(0, i[i == j], L.values()[i == j])
        ptr = torch.zeros(n_v + 1, dtype=torch.long, device=dev)
        ptr[1:] = torch.cumsum(torch.bincount(i, minlength=n_v), 0)
        self.L = torch.sparse_csr_tensor(ptr, j, L.values(), size=(n_v, n_v))


def _volume(E):
    return ((E[:, 1] - E[:, 0]) * torch.linalg.cross(E[:, 2] - E[:, 0], E[:, 3] - E[:, 0])).sum(-1) / 6


def _inside(P, X, tets, skip, step=256):
    """Index pairs (point, tet) with the point strictly inside; ``skip(points, tets)`` drops candidates."""
    E = X[tets]
    lo, hi = E.amin(1), E.amax(1)
    qi, ti = [], []
    for s in range(0, P.shape[0], step):
        p = P[s:s + step]
        c = torch.ones(p.shape[0], tets.shape[0], dtype=torch.bool, device=P.device)
        for k in range(3):
            c &= (p[:, None, k] > lo[None, :, k]) & (p[:, None, k] < hi[None, :, k])
        a, b = torch.nonzero(c, as_tuple=True)
        qi.append(a + s)
        ti.append(b)
    qi, ti = torch.cat(qi), torch.cat(ti)
    ok = ~skip(qi, ti)
    qi, ti = qi[ok], ti[ok]
    T, p = E[ti], P[qi]
    ok = torch.ones(qi.shape[0], dtype=torch.bool, device=P.device)
    for k in range(4):
        Q = T.clone()
        Q[:, k] = p
        ok &= _volume(Q) > 0
    return qi[ok], ti[ok]


def _closest(P, A, B, C):
    """Closest points of triangles (A, B, C) to P: (squared distance, weights of B and C)."""
    e1, e2, r = B - A, C - A, P - A
    d11, d12, d22 = (e1 * e1).sum(-1), (e1 * e2).sum(-1), (e2 * e2).sum(-1)
    r1, r2 = (r * e1).sum(-1), (r * e2).sum(-1)
    den = d11 * d22 - d12 * d12
    b1, b2 = (d22 * r1 - d12 * r2) / den, (d11 * r2 - d12 * r1) / den
    inside = (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1)
    best = torch.where(inside, ((r - b1[..., None] * e1 - b2[..., None] * e2) ** 2).sum(-1), torch.inf)
    for k, (u, v) in enumerate(((A, B), (B, C), (C, A))):
        e = v - u
        s = ((P - u) * e).sum(-1).div((e * e).sum(-1)).clamp(0, 1)
        d = ((P - u - s[..., None] * e) ** 2).sum(-1)
        better = ~inside & (d < best)
        best = torch.where(better, d, best)
        b1 = torch.where(better, (s, 1 - s, torch.zeros_like(s))[k], b1)
        b2 = torch.where(better, (torch.zeros_like(s), s, 1 - s)[k], b2)
    return best, b1, b2


def _face_point(X, faces, f, b1, b2):
    A, B, C = (X[faces[f, k]] for k in range(3))
    n = torch.linalg.cross(B - A, C - A)
    n = n / n.norm(dim=-1, keepdim=True)
    return (1 - b1 - b2)[:, None] * A + b1[:, None] * B + b2[:, None] * C, n


def _cast(body, X, v, normal, step=64):
    """Faces and weights that the vertices v correspond to: the first exit face along -normal, else the closest face.
    Weights of a hit carry their dependence on X, those of a closest point do not."""
    n_f = body.faces.shape[0]
    face = torch.empty(v.shape[0], dtype=torch.long, device=X.device)
    hit = torch.empty(v.shape[0], dtype=torch.bool, device=X.device)
    cb = torch.zeros(v.shape[0], 2, dtype=torch.float64, device=X.device)
    Xd = X.detach()
    A, B, C = (Xd[body.faces[:, k]][None] for k in range(3))
    for s in range(0, v.shape[0], step):
        w = v[s:s + step]
        o, d = Xd[w][:, None], -normal.detach()[s:s + step][:, None]
        no = (body.faces[None] == w[:, None, None]).any(-1) | (body.face_robot[None] != body.vert_robot[w][:, None])
        e1, e2 = B - A, C - A
        pv = torch.linalg.cross(d.expand(-1, n_f, -1), e2.expand(w.shape[0], -1, -1))
        det = (e1 * pv).sum(-1)
        tv = o - A
        qv = torch.linalg.cross(tv, e1.expand(w.shape[0], -1, -1))
        b1, b2, t = (tv * pv).sum(-1) / det, (d * qv).sum(-1) / det, (e2 * qv).sum(-1) / det
        good = ~no & ((d * torch.linalg.cross(e1, e2)).sum(-1) > 0) & (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1) & (t > 0)
        t, f = torch.where(good, t, torch.inf).min(1)
        hit[s:s + step] = torch.isfinite(t)
        miss = ~torch.isfinite(t)
        if miss.any():
            d2, c1, c2 = _closest(o[miss], A, B, C)
            g = torch.where(no[miss], torch.inf, d2).argmin(1)
            f[miss] = g
            at = torch.nonzero(miss)[:, 0] + s
            cb[at, 0], cb[at, 1] = c1.gather(1, g[:, None])[:, 0], c2.gather(1, g[:, None])[:, 0]
        face[s:s + step] = f
    # weights of the hits from their planes: x + t d with t = n.(q0 - x) / n.d
    q0, q1, q2 = (X[body.faces[face, k]] for k in range(3))
    x, d = X[v], -normal
    e1, e2 = q1 - q0, q2 - q0
    n = torch.linalg.cross(e1, e2)
    r = x + ((n * (q0 - x)).sum(-1) / (n * d).sum(-1))[:, None] * d - q0
    d11, d12, d22 = (e1 * e1).sum(-1), (e1 * e2).sum(-1), (e2 * e2).sum(-1)
    r1, r2 = (r * e1).sum(-1), (r * e2).sum(-1)
    den = d11 * d22 - d12 * d12
    hb = torch.stack([(d22 * r1 - d12 * r2) / den, (d11 * r2 - d12 * r1) / den], 1)
    return face, torch.where(hit[:, None], hb, cb)


class _Solve(torch.autograd.Function):
    """Free rows of A^-1 b, A = L + diag(extra), by conjugate gradients to 1e-14; its own adjoint."""

    @staticmethod
    def cg(body, extra, b, x):
        free = (~body.fixed)[:, None].to(torch.float64)
        idg = free / (body.diag + extra)[:, None]
        mul = lambda y: free * (body.L @ y + extra[:, None] * y)  # noqa: E731
        r = free * b - mul(x)
        z = idg * r
        p, g = z.clone(), (z * r).sum()
        stop = 1e-28 * ((free * b) ** 2).sum()
        for k in range(20000):
            q = mul(p)
            a = g / (p * q).sum()
            x, r = x + a * p, r - a * q
            if k % 16 == 0 and (r * r).sum() <= stop:
                break
            z = idg * r
            g, old = (z * r).sum(), g
            p = z + (g / old) * p
        return x

    @staticmethod
    def forward(ctx, body, extra, b, x):
        ctx.body, ctx.extra = body, extra
        return _Solve.cg(body, extra, b, x)

    @staticmethod
    def backward(ctx, g):
        return None, None, _Solve.cg(ctx.body, ctx.extra, g, torch.zeros_like(g)), None


def _rotation(D):
    """Nearest rotation of every D (det > 0), by Newton's iteration for the polar factor."""
    R = D / (D * D).sum((1, 2), keepdim=True).sqrt() * 3 ** 0.5
    for _ in range(25):
        C = torch.stack([torch.linalg.cross(R[:, (k + 1) % 3], R[:, (k + 2) % 3]) for k in range(3)], 1)
        R = 0.5 * (R + C / (R[:, 0] * C[:, 0]).sum(-1)[:, None, None])
    return R


def _local(body, X, alpha, knots):
    """Weighted element targets gathered on the vertices."""
    E = X[body.tets]
    Xc = E - E.mean(1, keepdim=True)
    R = _rotation(Xc.transpose(1, 2) @ body.Tc)
    RT = body.Tc @ R.transpose(1, 2)
    mis = ((Xc - RT) ** 2).sum((1, 2)) / (body.Tc ** 2).sum((1, 2))
    eps = torch.where(mis > 0, mis, 1e-300).sqrt()
    e, w = (torch.tensor([k[c] for k in knots], dtype=torch.float64, device=X.device) for c in (0, 1))
    i = torch.bucketize(eps.detach(), e, right=True).clamp(1, len(knots) - 1)
    wt = (w[i - 1] + (eps - e[i - 1]) * (w[i] - w[i - 1]) / (e[i] - e[i - 1])).clamp(float(w.min()), float(w.max()))
    B = (1 - wt)[:, None, None] * Xc + wt[:, None, None] * RT
    vb = _volume(B)
    ok = vb > 1e-3 * body.vol
    s = torch.where(ok, body.vol / torch.where(ok, vb, 1.0), 1.0) ** (1.0 / 3.0)
    chamber = body.group >= 0
    s = torch.where(chamber, alpha[body.group.clamp(min=0)] ** (1.0 / 3.0), s)
    P = s[:, None, None] * torch.where(chamber[:, None, None], RT, B)
    out = torch.zeros_like(X)
    return out.index_add(0, body.tets.reshape(-1), (body.omega[:, None, None] * P).reshape(-1, 3))


def _springs(body, m, X, old):
    """Spring targets on the query vertices after one collision check; ``old`` and the result: (active, kind, face,
    weights), kind 0 self, 1 sphere, 2 tetrahedral obstacle."""
    q = body.query
    x, n_q, eps = X[q], body.query.shape[0], m.eps
    Xd = X.detach()
    active, kind, face, bary = (t.clone() for t in old)
    target = torch.zeros_like(x)
    own = lambda a, b: ((body.tets[b] == q[a][:, None]).any(1)  # noqa: E731
                        | (body.robot[b] != body.vert_robot[q[a]]))
    paired = torch.zeros(n_q, dtype=torch.bool, device=X.device)
    paired[_inside(Xd[q], Xd, body.tets, own)[0]] = True
    F = [X[body.faces[:, k]] for k in range(3)]
    fn = torch.linalg.cross(F[1] - F[0], F[2] - F[0])
    vn = torch.zeros_like(X)
    for k in range(3):
        vn = vn.index_add(0, body.faces[:, k], fn)
    new = torch.zeros(n_q, dtype=torch.bool, device=X.device)
    if m.collision >= 2 and len(m.spheres):
        S = torch.tensor(m.spheres, dtype=torch.float64, device=X.device)
        d = (Xd[q][:, None] - S[None, :, :3]).norm(dim=-1) - S[None, :, 3]
        d, j = d.min(1)
        new = d < 0
        kind[new], face[new] = 1, j[new]
    if m.collision >= 2 and m.obstacle_X is not None:
        O = torch.tensor(m.obstacle_X, dtype=torch.float64, device=X.device)
        ot = torch.tensor(m.obstacle_tets, dtype=torch.long, device=X.device)
        inob = torch.zeros_like(new)
        inob[_inside(Xd[q], O, ot, lambda a, b: torch.zeros_like(a, dtype=torch.bool))[0]] = True
        f = torch.stack([ot[:, list(k)] for k in _Body.FACES], 1).reshape(-1, 3)
        key = f.sort(1).values
        _, inv, cnt = torch.unique(key, dim=0, return_inverse=True, return_counts=True)
        f = f[cnt[inv] == 1]
        d2, c1, c2 = _closest(Xd[q][inob][:, None], *(O[f[:, k]][None] for k in range(3)))
        g = d2.argmin(1, keepdim=True)
        p, nf = _face_point(O, f, g[:, 0], c1.gather(1, g)[:, 0], c2.gather(1, g)[:, 0])
        target[inob] = p + eps * nf
        kind[inob], face[inob] = 2, g[:, 0]
        new = new | inob
    cast = paired & ~new
    if cast.any():
        vv = vn[q[cast]]
        f, b = _cast(body, X, q[cast], vv / vv.norm(dim=-1, keepdim=True))
        kind[cast], face[cast] = 0, f
        bary = bary.index_put((cast,), b)
    kept = active & ~new & ~cast
    active = new | cast | kept
    one = active & (kind == 1)
    if one.any():
        c, r = S[face[one], :3], S[face[one], 3]
        u = x[one] - c
        nu = u.norm(dim=-1)
        target = target.index_put((one,), c + ((r + eps) / nu)[:, None] * u)
        gone = kept[one] & ((nu - r) > eps)
        active[torch.nonzero(one)[:, 0][gone]] = False
    self_ = active & (kind == 0)
    if self_.any():
        p, nf = _face_point(X, body.faces, face[self_], bary[self_, 0], bary[self_, 1])
        target = target.index_put((self_,), p + eps * nf)
        gone = kept[self_] & (((x[self_] - p) * nf).sum(-1) > eps)
        active[torch.nonzero(self_)[:, 0][gone]] = False
    return (active, kind, face, bary), target


def _loop(body, m, X, alpha, n):
    dev, n_q = X.device, body.query.shape[0]
    sp = (torch.zeros(n_q, dtype=torch.bool, device=dev), torch.zeros(n_q, dtype=torch.long, device=dev),
          torch.full((n_q,), -1, dtype=torch.long, device=dev), torch.zeros(n_q, 2, dtype=torch.float64, device=dev))
    fixed = torch.where(body.fixed[:, None], X.detach(), 0.0)
    for _ in range(n):
        b = _local(body, X, alpha, m.w_knots) - body.L @ fixed
        extra = torch.zeros_like(body.diag)
        if m.collision >= 1:
            sp, target = _springs(body, m, X, sp)
            on = sp[0]
            extra[body.query[on]] = m.k_spring
            b = b.index_add(0, body.query[on], m.k_spring * target[on])
        y = _Solve.apply(body, extra, b, torch.where(body.fixed[:, None], 0.0, X.detach()))
        X = fixed + torch.where(body.fixed[:, None], 0.0, y)
    return X


def exact(case, seed):
    """The loop in 64-bit torch: a dense all-pairs contact check, dense ray casts, Newton polar factors, CG to 1e-14.
    None for MIXED runs of several iterations with contacts, whose decisions have no 64-bit counterpart, and for the
    contact check, whose outputs are whole numbers."""
    if case["kind"] == "contacts" or (case["kind"] == "run" and not case["fp64"] and case["n"] > 1):
        return None
    meshes, _, X0 = _scene(case, seed)
    body, m = _Body(meshes), meshes[0]
    X = body.rest if X0 is None else torch.tensor(X0, dtype=torch.float64, device="cuda")
    if case["kind"] == "run":
        x = _loop(body, m, X, body.alpha, case["n"])
        return {"x": x}
    alpha = body.alpha.clone().requires_grad_(True)
    x = _loop(body, m, X, alpha, case["n"])
    tips, targets = _tips(m, seed)
    ((x[torch.from_numpy(tips).cuda()] - torch.from_numpy(targets).cuda()) ** 2).sum().backward()
    return {"x": x.detach().cpu(), "grad": alpha.grad.cpu()}

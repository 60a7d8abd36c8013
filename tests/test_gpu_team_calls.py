"""Calls around the team PCG: several handles in one process, batches of very many
robots, robots without a free vertex, and solves that need no iteration."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import global_step, local, loop, springs as osprings

pytestmark = pytest.mark.gpu

FP64, MIXED = synth.PRECISION_FP64, synth.PRECISION_MIXED
BAR = {FP64: 1e-9, MIXED: 1e-5}


def _want(m, X0, collision):
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    return loop.iterate(prep, X0, osprings.SpringState.empty(prep.query.shape[0]), m.alpha, m.spheres, m.w_knots,
                        m.k_spring, m.eps, collision)[0]


def _fingers(precision, sizes):
    return [synth.small_finger(*s, seed=5 + k, n_iters=1, precision=precision) for k, s in enumerate(sizes)]


# (each pair runs on one kernel instance: FP64 and MIXED with one row per thread,
# MIXED batches of 93,000 and 70,000 rows with three)
@pytest.mark.parametrize("precision,first,second", [
    (FP64, [(60, 12, 12, 8)], [(30, 9, 9, 4)]),
    (MIXED, [(60, 12, 12, 8)], [(30, 9, 9, 4)]),
    (MIXED, [(40, 19, 18, 4)] * 6, [(36, 19, 18, 4)] * 5),
])
def test_an_upload_leaves_other_handles_alone(precision, first, second):
    """Eager launches (stats 2) and a first capture of a handle after another one
    has uploaded a smaller mesh."""
    runs = []
    for other in (False, True):
        ms = _fingers(precision, first)
        a = [casim.Sim(ms if len(ms) > 1 else ms[0], stats=s) for s in (1, 2)]
        assert a[0].stats().pcg_kernel == 5
        b = None
        if other:
            mb = _fingers(precision, second)
            b = casim.Sim(mb if len(mb) > 1 else mb[0])
        for s in a:
            s.step(2)
            assert s.sync() == 0
            runs.append(s.positions())
        for s in a + [b] * other:
            s.close()
    for X in runs[1:]:
        assert np.array_equal(X, runs[0])


def test_batch_of_very_many_robots():
    n = 11000
    rest, tets, group, fixed = synth._voxel_kuhn(1, 1, 2, 0.5, group_of_voxel=lambda i, j, k: 0)
    m = synth.config1_beam()
    m.rest, m.tets, m.group, m.fixed = rest, tets, group, fixed
    m.precision, m.collision = MIXED, synth.COLLISION_OFF
    robots = []
    for r in range(n):
        q = synth.Mesh(**vars(m)) if r else m
        q.alpha = np.array([1.1 + 0.5 * r / n])
        robots.append(q)
    sim = casim.Sim(robots)
    assert sim.stats().pcg_kernel == 5
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions().reshape(n, m.n_verts, 3)
    sim.close()
    for r in (0, 1, n // 2, n - 1):
        want = _want(robots[r], m.rest, 0)
        assert np.abs(X[r] - want).max() <= BAR[MIXED] * m.bbox_diag()


@pytest.mark.parametrize("precision", [FP64, MIXED])
@pytest.mark.parametrize("at", [0, 1, 2])
def test_a_robot_without_free_vertices(precision, at):
    ms = _fingers(precision, [(20, 4, 4, 4), (12, 4, 4, 2), (23, 5, 5, 3)])
    ms[at].fixed = np.ones_like(ms[at].fixed)
    dtype = np.float64 if precision == FP64 else np.float32
    X0 = [m.rest.copy() if k == at else synth.perturbed_positions(m, 0.25, seed=60 + k, dtype=dtype)
          for k, m in enumerate(ms)]
    sim = casim.Sim(ms)
    assert sim.stats().pcg_kernel == 5
    sim.set_positions(np.concatenate(X0))
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions()
    sim.close()
    o = np.cumsum([0] + [m.n_verts for m in ms])
    for k, m in enumerate(ms):
        want = X0[k] if k == at else _want(m, X0[k], m.collision)
        assert np.abs(X[o[k]:o[k + 1]] - want).max() <= BAR[precision] * m.bbox_diag()


@pytest.mark.parametrize("n_robots", [1, 3])
def test_a_solve_without_iterations_returns_where_its_residual_was_tested(n_robots):
    """With a loose tolerance the extrapolated start soon meets it.  The positions
    returned then have a residual within the tolerance, the ones the iteration
    came from had not (several times above it along this trajectory)."""
    tol = 5e-5
    ms = [synth.small_finger(20, 4, 4, 4, seed=7 + r, n_iters=30) for r in range(n_robots)]
    for m in ms:
        m.collision = synth.COLLISION_OFF
    preps = [loop.prepare(m.rest, m.tets, m.group, m.fixed) for m in ms]
    o = np.cumsum([0] + [m.n_verts for m in ms])

    def residual(k, Xi, X):
        """of the global step of robot k that starts from Xi, at X"""
        m, p = ms[k], preps[k]
        P = local.local_step(Xi, p.tets, p.T_c, p.vol0, p.group, m.alpha, m.w_knots)[0]
        A, b = global_step.assemble(p.tets, p.omega, P, p.n_verts, [], np.zeros((0, 3)), m.k_spring)
        free = ~p.fixed.astype(bool)
        rhs = b[free] - A[free][:, ~free] @ X[~free]
        return np.linalg.norm(rhs - A[free][:, free] @ X[free]) / np.linalg.norm(rhs)

    sim = casim.Sim(ms if n_robots > 1 else ms[0], pcg_tol=tol)
    assert sim.stats().pcg_kernel == 5
    X = np.concatenate([m.rest for m in ms])
    none = 0
    for _ in range(30):
        Xi = X.astype(np.float64)
        sim.step(1)
        assert sim.sync() == 0
        X = sim.positions().astype(np.float64)
        if sim.history()[-1]["pcg_iters"] == 0:
            none += 1
            for k in range(n_robots):
                s = slice(o[k], o[k + 1])
                assert residual(k, Xi[s], Xi[s]) > tol
                # (5 %: FP32 targets are within 1e-6 of the right-hand side)
                assert residual(k, Xi[s], X[s]) <= 1.05 * tol
    sim.close()
    assert none > 0  # (premise: such solves occurred)

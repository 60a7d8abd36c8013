"""Calls around the team PCG: several handles in one process, batches of very many
robots, and robots without a free vertex."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import loop, springs as osprings

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

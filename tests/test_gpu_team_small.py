"""Robots of a few free vertices, and free vertices that hardly touch one another:
their residuals fall by many digits within one CG iteration.  One outer iteration
against the FP64 oracle, held to the bars of the other replays."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import loop, springs as osprings

pytestmark = pytest.mark.gpu

FP64, MIXED = synth.PRECISION_FP64, synth.PRECISION_MIXED
BAR = {FP64: 1e-9, MIXED: 1e-5}


def _block(n, precision, free):
    """An n^3-voxel block of which only the vertices free(grid indices) move."""
    m = synth.config1_beam()
    m.rest, m.tets, m.group, m.fixed = synth._voxel_kuhn(n, n, n, 0.5,
                                                         group_of_voxel=lambda i, j, k: 0 if (i + j + k) % 2 else -1)
    m.fixed = (~free(np.rint(m.rest / 0.5).astype(int))).astype(np.uint8)
    m.alpha = np.array([1.3])
    m.precision, m.collision = precision, synth.COLLISION_OFF
    return m


def _check(m, X):
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    want = loop.iterate(prep, m.rest, osprings.SpringState.empty(prep.query.shape[0]), m.alpha, m.spheres, m.w_knots,
                        m.k_spring, m.eps, m.collision)[0]
    assert np.abs(X - want).max() <= BAR[m.precision] * m.bbox_diag()


def _first(rows):
    def free(g):
        f = np.zeros(len(g), bool)
        f[np.argsort(-g[:, 2] - 1e-3 * g[:, 1] - 1e-6 * g[:, 0], kind="stable")[:rows]] = True
        return f
    return free


def _apart(g):
    return (g % 2 == 0).all(1)


@pytest.mark.parametrize("precision", [FP64, MIXED])
@pytest.mark.parametrize("rows", [1, 2, 3, 5, 9, 17, 31, 33, 64, 127, 128, 129])
def test_few_rows(precision, rows):
    m = _block(8, precision, _first(rows))
    sim = casim.Sim(m)
    assert sim.stats().pcg_kernel == 5 and sim.sizes["n_free"] == rows
    sim.step(1)
    assert sim.sync() == 0
    assert sim.history()[-1]["pcg_iters"] <= max(rows, 4) + 2
    _check(m, sim.positions())
    sim.close()


@pytest.mark.parametrize("precision", [FP64, MIXED])
@pytest.mark.parametrize("n_robots", [1, 3])
def test_rows_apart(precision, n_robots):
    ms = [_block(12, precision, _apart) for _ in range(n_robots)]
    if n_robots > 1:
        ms[1] = _block(8, precision, _first(3))
    sim = casim.Sim(ms if n_robots > 1 else ms[0])
    assert sim.stats().pcg_kernel == 5
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions()
    sim.close()
    o = np.cumsum([0] + [m.n_verts for m in ms])
    for k, m in enumerate(ms):
        _check(m, X[o[k]:o[k + 1]])

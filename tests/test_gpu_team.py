"""The team PCG (one thread-block team per robot, vectors on chip) at the sizes
where its plans change: a few rows, one part, parts that end in the middle of a
warp, two and three rows per thread, more parts than blocks.  One
outer iteration from a contact-bearing state against the FP64 oracle, held to
the bars of the other replays (1e-9 of the diagonal in FP64, 1e-5 in MIXED)."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import loop, springs as osprings

pytestmark = pytest.mark.gpu

FP64, MIXED = synth.PRECISION_FP64, synth.PRECISION_MIXED
BAR = {FP64: 1e-9, MIXED: 1e-5}


def _robot(nx, ny, nz, n_ch, seed, precision):
    return synth.small_finger(nx, ny, nz, n_ch, seed=seed, n_iters=1, precision=precision)


def _start(m, seed):
    dtype = np.float64 if m.precision == FP64 else np.float32
    return synth.perturbed_positions(m, 0.25, seed=seed, dtype=dtype)


def _check(m, X0, X):
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    want = loop.iterate(prep, X0, osprings.SpringState.empty(prep.query.shape[0]), m.alpha, m.spheres, m.w_knots,
                        m.k_spring, m.eps, m.collision)[0]
    assert np.abs(X - want).max() <= BAR[m.precision] * m.bbox_diag()


@pytest.mark.parametrize("precision,shape", [
    (FP64, (3, 3, 2, 1)),        # 36 rows: a part of one warp and one of four rows
    (FP64, (20, 4, 4, 4)),       # a row count that ends inside a warp
    (FP64, (48, 19, 20, 6)),     # 2 rows per thread
    (FP64, (100, 19, 20, 6)),    # 3 rows per thread
    (MIXED, (3, 3, 2, 1)),
    (MIXED, (31, 5, 7, 3)),
    (MIXED, (60, 11, 13, 8)),
])
@pytest.mark.parametrize("precond", [0, 1])
def test_one_iteration_matches_oracle(precision, shape, precond):
    if precond and shape[0] > 60:
        pytest.skip("covered by the smaller sizes")
    m = _robot(*shape, seed=41, precision=precision)
    X0 = _start(m, 9)
    sim = casim.Sim(m, pcg_precond=precond)
    assert sim.stats().pcg_kernel == 5
    sim.set_positions(X0)
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions()
    sim.close()
    _check(m, X0, X)


@pytest.mark.parametrize("precision,n_robots", [
    (FP64, 3),       # one part per block
    (FP64, 45),      # more parts than blocks
    (MIXED, 3),
    (MIXED, 45),     # 3 rows per thread
    (MIXED, 160),    # 3 rows per thread, more parts than blocks
])
def test_batches_match_each_robots_oracle(precision, n_robots):
    shapes = [(20, 8, 9, 2), (23, 5, 5, 3), (16, 10, 11, 2), (12, 4, 4, 2)]
    batch = [_robot(*shapes[r % 4], seed=r, precision=precision) for r in range(n_robots)]
    X0s = [_start(m, 50 + r) for r, m in enumerate(batch)]
    sim = casim.Sim(batch)
    assert sim.stats().pcg_kernel == 5
    sim.set_positions(np.concatenate(X0s))
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions()
    sim.close()
    at = np.cumsum([0] + [m.n_verts for m in batch])
    for r in sorted({0, 1, 2, n_robots // 2, n_robots - 1}):
        _check(batch[r], X0s[r], X[at[r]:at[r + 1]])


def test_coarse_correction_cuts_the_iterations():
    """From rest (no springs) and with contacts, in both precisions: its whole
    purpose (a wrong coarse matrix or inverse would only cost iterations)."""
    for precision in (FP64, MIXED):
        m = synth.config2_finger()
        m.precision = precision
        its = []
        for precond in (0, 1):
            sim = casim.Sim(m, pcg_precond=precond)
            sim.step(4)
            assert sim.sync() == 0
            its.append([h["pcg_iters"] for h in sim.history()])
            sim.close()
        assert its[0][0] < 0.5 * its[1][0] and its[0][3] < 0.6 * its[1][3], its


@pytest.mark.parametrize("unit", [1e-7, 1e6])
@pytest.mark.parametrize("shape", [(20, 4, 4, 4), (60, 11, 13, 8)])
def test_mixed_in_other_units(shape, unit):
    # squared residuals near FP32's range; one cluster and one team of blocks
    m = _robot(*shape, seed=23, precision=MIXED)
    X0 = _start(m, 4) * unit
    X0 = X0.astype(np.float32).astype(np.float64)
    m.rest = m.rest * unit
    m.collision = synth.COLLISION_OFF
    sim = casim.Sim(m)
    sim.set_positions(X0)
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions()
    sim.close()
    _check(m, X0, X)

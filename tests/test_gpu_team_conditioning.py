"""Bodies whose soft modes are far softer than their elements, where the coarse
correction's FP32 inverse is not good enough: the solves still converge, within the
iterations that they are given.  The residual of the returned positions, formed by
the oracle's own system, is within the solver's tolerance and the rounding of that
formula."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import global_step, local, loop

pytestmark = pytest.mark.gpu

FP64, MIXED = synth.PRECISION_FP64, synth.PRECISION_MIXED


def _bar(nx, ny, nz, precision):
    m = synth.config1_beam()
    m.rest, m.tets, m.group, m.fixed = synth._voxel_kuhn(nx, ny, nz, 0.5,
                                                         group_of_voxel=lambda i, j, k: 0 if k == nz - 1 else -1)
    m.alpha = np.array([1.3])
    m.precision, m.collision = precision, synth.COLLISION_OFF
    return m


def _check(m, Xi, X, tol):
    """Residual at X of the global step that starts from Xi."""
    p = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    P = local.local_step(Xi, p.tets, p.T_c, p.vol0, p.group, m.alpha, m.w_knots)[0]
    A, b = global_step.assemble(p.tets, p.omega, P, p.n_verts, [], np.zeros((0, 3)), m.k_spring)
    free = ~p.fixed.astype(bool)
    F, C = A[free][:, free], A[free][:, ~free]
    rhs = b[free] - C @ X[~free]
    # (64 roundings of each term: about 20 of them in a row, the targets' and the right-hand side's)
    size = abs(F) @ np.abs(X[free]) + abs(C) @ np.abs(X[~free]) + np.abs(b[free])
    bound = tol * np.linalg.norm(rhs) + 64 * 2.0 ** -53 * np.linalg.norm(size)
    assert np.linalg.norm(rhs - F @ X[free]) <= bound


@pytest.mark.parametrize("precision,nx", [(FP64, 300), (FP64, 1500), (FP64, 2000), (MIXED, 1500), (MIXED, 3000)])
def test_long_bodies_converge(precision, nx):
    m = _bar(nx, 2, 2, precision)
    sim = casim.Sim(m)
    assert sim.stats().pcg_kernel == 5
    X = m.rest
    for _ in range(3):
        Xi = X
        sim.step(1)
        assert sim.sync() == 0
        X = sim.positions().astype(np.float64)
        if precision == FP64:
            _check(m, Xi, X, sim.params.pcg_tol)
    sim.close()


@pytest.mark.parametrize("precision", [FP64, MIXED])
def test_a_long_body_in_a_batch(precision):
    ms = [_bar(20, 4, 4, precision), _bar(2500, 2, 2, precision), _bar(31, 5, 4, precision)]
    sim = casim.Sim(ms)
    assert sim.stats().pcg_kernel == 5
    sim.step(1)
    assert sim.sync() == 0
    X = sim.positions().astype(np.float64)
    sim.close()
    o = np.cumsum([0] + [m.n_verts for m in ms])
    if precision == FP64:
        for k, m in enumerate(ms):
            _check(m, m.rest, X[o[k]:o[k + 1]], 1e-12)


def _layered(nx, ny, nz, precision, thickness):
    """A bar with a layer of thin elements across it: its far side hangs on that
    fraction of an element's stiffness, a mode that no part's functions contain."""
    m = _bar(nx, ny, nz, precision)
    layer = np.rint(m.rest[:, 0] / 0.5) >= 5
    m.rest = m.rest.copy()
    m.rest[layer, 0] -= 0.5 * (1.0 - thickness)
    return m


@pytest.mark.parametrize("thickness", [1e-3, 1e-4, 1e-5, 1e-6])
@pytest.mark.parametrize("precision", [FP64, MIXED])
def test_a_thin_layer_converges(precision, thickness):
    m = _layered(40, 8, 8, precision, thickness)
    sim = casim.Sim(m)
    assert sim.stats().pcg_kernel == 5
    X = m.rest
    for _ in range(4):
        Xi = X
        sim.step(1)
        assert sim.sync() == 0
        X = sim.positions().astype(np.float64)
        if precision == FP64:
            _check(m, Xi, X, sim.params.pcg_tol)
    sim.close()


# (FP64 in one cluster and in a batch; MIXED with the linear functions, one row per
# thread in a batch and three)
@pytest.mark.parametrize("precision,shape,thickness", [
    (FP64, (16, 4, 4), 1e-7), (FP64, (40, 8, 8), 1e-5), (MIXED, (40, 8, 8), 1e-6), (MIXED, (150, 20, 20), 1e-5)])
def test_thin_layers_in_batches_and_large_bodies(precision, shape, thickness):
    ms = [_layered(*shape, precision, thickness)]
    if shape[0] == 40:
        ms.append(_bar(20, 4, 4, precision))
    sim = casim.Sim(ms if len(ms) > 1 else ms[0])
    assert sim.stats().pcg_kernel == 5
    for _ in range(3):
        sim.step(1)
        assert sim.sync() == 0
    sim.close()


@pytest.mark.parametrize("precision", [FP64, MIXED])
@pytest.mark.parametrize("k_spring", [1e-3, 1.0, 1e3, 1e5])
def test_spring_weights(precision, k_spring):
    """The two-level preconditioner against Jacobi over contact-bearing iterations:
    far from stiff springs it saves iterations, with them it costs few."""
    its = []
    for precond in (0, 1):
        m = synth.small_finger(40, 8, 8, 5, seed=2, n_iters=1, precision=precision)
        m.k_spring = k_spring
        X0 = synth.perturbed_positions(m, 0.25, seed=7, dtype=np.float64 if precision == FP64 else np.float32)
        sim = casim.Sim(m, pcg_precond=precond)
        assert sim.stats().pcg_kernel == 5
        sim.set_positions(X0)
        sim.step(3)
        assert sim.sync() == 0
        h = sim.history()
        assert all(r["n_springs"] > 0 for r in h)
        its.append(sum(r["pcg_iters"] for r in h))
        sim.close()
    # (in FP64 the first stops at 1/32 of the second's tolerance, a tenth more iterations)
    assert its[0] <= (1.25 if k_spring > 1 else 0.9) * its[1], its

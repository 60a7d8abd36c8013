"""FP64 rotation fit of the local step (FP32 SVD, two Newton steps, the FP64 SVD
where they do not apply) on elements near the edges of its tests: small and large
strains, inverted and flattened elements, elements almost collapsed onto a line,
and a robot measured in other units.  Targets against the oracle's LAPACK fit.
Tolerance: either fit is accurate to a few units of 1e-16 times s1 / (s2 + s3), the
fit's condition; elements conditioned worse than 1e5 are left out, which gives
1e-10 of an element's size, and a factor 10 is allowed on it."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import local, loop

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["small", "large", "flat", "line", "mirror", "mixed"])
@pytest.mark.parametrize("unit", [1.0, 1e-6, 1e5])
def test_targets_equal_oracle(kind, unit):
    m = synth.small_finger(nx=12, ny=3, nz=4, n_ch=2, seed=5, n_iters=1, precision=synth.PRECISION_FP64)
    rng = np.random.default_rng(8)
    X = synth.perturbed_positions(m, {"small": 0.02, "large": 1.2}.get(kind, 0.2), seed=3, dtype=np.float64)
    if kind == "flat":
        X[:, 2] *= 1e-3
    elif kind == "line":
        X[:, 1:] *= 1e-4
    elif kind == "mirror":
        X[:, 0] *= -1.0
    elif kind == "mixed":
        X *= np.where(rng.random((len(X), 1)) < 0.1, 3.0, 1.0)
    m.rest, X = m.rest * unit, X * unit
    m.collision = synth.COLLISION_OFF
    sim = casim.Sim(m)
    sim.set_positions(X)
    sim.step(1)
    sim.sync()
    got = sim.targets()
    sim.close()
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    want = local.local_step(X, prep.tets, prep.T_c, prep.vol0, prep.group, m.alpha, m.w_knots)[0]
    P = X[prep.tets]
    Xc = P - P.mean(axis=1, keepdims=True)
    R = m.rest[prep.tets]
    Tc = R - R.mean(axis=1, keepdims=True)
    D = np.einsum("eki,ekj->eij", Xc, Tc)
    s = np.linalg.svd(D, compute_uv=False)
    gap = s[:, 1] + np.sign(np.linalg.det(D)) * s[:, 2]
    ok = gap > 1e-5 * s[:, 0]
    assert ok.mean() > 0.5
    size = np.maximum(np.abs(Xc).max(axis=(1, 2)), np.abs(Tc).max(axis=(1, 2)))
    err = np.abs(got - want).reshape(len(size), -1).max(axis=1) / size
    assert err[ok].max() <= 1e-9

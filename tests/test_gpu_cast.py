"""Ray casts, four vertices to a warp behind FP32 reject tests, over the hash of the
faces and over their tree: cast counts that leave teams and warps idle, both precisions, and
positions far from the origin (where the FP32 test's bound of an FP64 position is
at its widest).  Hit faces equal the oracle's exactly; targets and barycentrics
agree to 1e-9, the bar of the other replays."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import loop, springs as osprings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [synth.PRECISION_FP64, synth.PRECISION_MIXED])
@pytest.mark.parametrize("shape,amp,shift", [
    ((8, 3, 3, 1), 0.45, 0.0),
    ((20, 4, 4, 4), 0.3, 0.0),
    ((20, 4, 4, 4), 0.45, 40.0),
    ((31, 5, 7, 3), 0.4, 3.0),
])
@pytest.mark.parametrize("broad", [0, 1])
def test_hits_equal_oracle(precision, shape, amp, shift, broad):
    m = synth.small_finger(*shape, seed=17, n_iters=1, precision=precision)
    dtype = np.float64 if precision == synth.PRECISION_FP64 else np.float32
    X0 = synth.perturbed_positions(m, amp, seed=5, dtype=np.float64) + shift * m.bbox_diag() * np.array([1.0, -0.7, 0.4])
    X0 = X0.astype(dtype).astype(np.float64)
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    _, st, _, ps, _ = loop.iterate(prep, X0, osprings.SpringState.empty(prep.query.shape[0]), m.alpha, m.spheres,
                                   m.w_knots, m.k_spring, m.eps, m.collision)
    sim = casim.Sim(m, broad_phase=broad)
    sim.set_positions(X0)
    sim.step(1)
    assert sim.sync() in (0, casim.CASIM_W_PCG_MAXIT)
    sp = sim.springs()
    assert ps.shape[0] > 0
    assert np.array_equal(sim.contacts()[0], ps)
    sim.close()
    assert np.array_equal(sp["active"], st.active)
    assert np.array_equal(sp["kind"][st.active], st.kind[st.active])
    assert np.array_equal(sp["face"][st.active], st.face[st.active])
    assert np.allclose(sp["target"], st.target, rtol=0.0, atol=1e-9)
    assert np.allclose(sp["bary"], st.bary, rtol=0.0, atol=1e-9)

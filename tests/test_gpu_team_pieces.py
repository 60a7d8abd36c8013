"""Small MIXED robots: row counts at the edges of one cluster of 96-row parts (up to
1,536 rows), of parts of two and of three such pieces, and of the sizes beyond them.
One outer iteration from a contact-bearing state against the FP64 oracle, held to
the bar of the other MIXED replays, and the coarse correction's effect."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import loop, springs as osprings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1536, 1537, 1921, 3072, 3073, 3400, 4096, 4097])
def test_small_robots_at_the_edges_of_their_plans(rows):
    m = synth.small_finger(44, 9, 9, 5, seed=12, n_iters=1)
    # clamped from the base on until that many rows are free
    m.fixed = np.ones_like(m.fixed)
    m.fixed[np.argsort(m.rest[:, 0], kind="stable")[-rows:]] = 0
    X0 = synth.perturbed_positions(m, 0.25, seed=4, dtype=np.float32).astype(np.float64)
    X0[m.fixed == 1] = m.rest[m.fixed == 1]
    its = []
    for precond in (0, 1):
        sim = casim.Sim(m, pcg_precond=precond)
        assert sim.stats().pcg_kernel == 5 and sim.sizes["n_free"] == rows
        sim.set_positions(X0)
        sim.step(1)
        assert sim.sync() == 0
        its.append(sim.history()[-1]["pcg_iters"])
        if precond == 0:
            X = sim.positions()
        sim.close()
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    want = loop.iterate(prep, X0, osprings.SpringState.empty(prep.query.shape[0]), m.alpha, m.spheres, m.w_knots,
                        m.k_spring, m.eps, m.collision)[0]
    assert np.abs(X - want).max() <= 1e-5 * m.bbox_diag()
    assert its[0] < 0.85 * its[1], its

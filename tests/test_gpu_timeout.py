"""Solves that give up: several contact-bearing iterations in one call, each of
whose bounded waits runs out (a round that waits for one block more than it has).
Every iteration starts its contact lists from empty and closes its record, so all
of them find the same contacts and cast the same rays: the positions stay put."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth

pytestmark = pytest.mark.gpu

FP64, MIXED = synth.PRECISION_FP64, synth.PRECISION_MIXED


@pytest.mark.parametrize("precision", [FP64, MIXED])
@pytest.mark.parametrize("broad", [0, 1])
@pytest.mark.parametrize("n_robots", [1, 2])
def test_iterations_after_a_timeout_start_from_empty_lists(precision, broad, n_robots):
    ms = [synth.small_finger(24, 5, 5, 4, seed=3 + r, n_iters=1, precision=precision) for r in range(n_robots)]
    dtype = np.float64 if precision == FP64 else np.float32
    X0 = np.concatenate([synth.perturbed_positions(m, 0.25, seed=7, dtype=dtype) for m in ms])
    sim = casim.Sim(ms if n_robots > 1 else ms[0], broad_phase=broad, wait_budget_cycles=2_000_000,
                    debug_flags=casim.CASIM_DEBUG_BARRIER_NEVER_COMPLETES)
    assert sim.stats().pcg_kernel == 5
    sim.set_positions(X0)
    sim.step(4)
    with pytest.raises(casim.CasimError) as ei:
        sim.sync()
    assert ei.value.code == casim.CASIM_E_TIMEOUT
    h = sim.history()
    assert sim.stats().iterations == 4 and len(h) == 4
    assert h[0]["n_self_pairs"] > 0 and h[0]["n_springs"] > 0
    for rec in h[1:]:
        assert rec["n_self_pairs"] == h[0]["n_self_pairs"]
        assert rec["n_springs"] == h[0]["n_springs"]
    assert np.array_equal(sim.positions(), X0)
    sim.close()

"""Calls around the team PCG: several handles in one process."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth

pytestmark = pytest.mark.gpu

FP64, MIXED = synth.PRECISION_FP64, synth.PRECISION_MIXED


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

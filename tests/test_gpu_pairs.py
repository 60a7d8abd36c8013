"""The hash broad phase and its narrow phase (one thread per tet over the listed
vertices of its cells) where their walk changes: tets whose boxes span many
bricks of cells, cells on both sides of the origin, lists of many vertices in one
cell, warps and blocks that are partly idle.  The pairs are the oracle's exactly,
so no tolerance enters."""
import numpy as np
import pytest

from paper_2203_02054_gb300 import casim, synth
from oracle import loop, springs as osprings

pytestmark = pytest.mark.gpu


def _state(m, seed, stretch, dtype):
    """Perturbed positions around the origin with a few vertices pulled away."""
    X = synth.perturbed_positions(m, 0.35, seed=seed, dtype=np.float64)
    X = X - X.mean(axis=0)
    rng = np.random.default_rng(seed)
    far = rng.choice(len(X), 6, replace=False)
    X[far] += stretch * m.h * rng.uniform(-1.0, 1.0, size=(6, 3))
    return X.astype(dtype).astype(np.float64)


def _oracle_pairs(m, X):
    prep = loop.prepare(m.rest, m.tets, m.group, m.fixed)
    return prep, loop.iterate(prep, X, osprings.SpringState.empty(prep.query.shape[0]), m.alpha, m.spheres, m.w_knots,
                              m.k_spring, m.eps, m.collision)[3]


@pytest.mark.parametrize("precision", [synth.PRECISION_FP64, synth.PRECISION_MIXED])
@pytest.mark.parametrize("shape,stretch,scale", [
    ((3, 3, 2, 1), 0.0, 1.0),
    ((20, 4, 4, 4), 12.0, 2.0),
    ((20, 4, 4, 4), 2.0, 6.0),
    ((31, 5, 7, 3), 6.0, 1.3),
])
def test_pairs_equal_oracle(precision, shape, stretch, scale):
    m = synth.small_finger(*shape, seed=3, n_iters=1, precision=precision)
    X = _state(m, 11, stretch, np.float64 if precision == synth.PRECISION_FP64 else np.float32)
    want = _oracle_pairs(m, X)[1]
    sim = casim.Sim(m, cell_scale=scale)
    sim.set_positions(X)
    sim.step(1)
    sim.sync()
    got = sim.contacts()[0]
    sim.close()
    assert np.array_equal(got, want)


def test_too_many_entries_are_refused():
    # 30 cells a tet on average; the declared capacity is 16 an item
    m = synth.small_finger(20, 4, 4, 4, seed=3, n_iters=1)
    sim = casim.Sim(m)
    sim.set_positions(_state(m, 11, 12.0, np.float32))
    sim.step(1)
    with pytest.raises(casim.CasimError) as e:
        sim.sync()
    assert e.value.code == casim.CASIM_E_OVERFLOW
    sim.close()


@pytest.mark.parametrize("cell", [0.3, 1.0, 5.0])
def test_noalloc_pairs_equal_oracle(cell):
    import torch

    m = synth.small_finger(nx=20, ny=4, nz=4, n_ch=4)
    X = _state(m, 7, 3.0, np.float32)
    prep, want = _oracle_pairs(m, X)
    xyz = torch.tensor(X.astype(np.float32), device="cuda").contiguous()
    tets = torch.tensor(m.tets.astype(np.int32), device="cuda").contiguous()
    q = torch.tensor(prep.query.astype(np.int32), device="cuda").contiguous()

    def call(query, t):
        count = torch.full((len(query),), -1, dtype=torch.int32, device="cuda")
        out = torch.full((len(query), 16), -1, dtype=torch.int32, device="cuda")
        rc = casim.casim_contacts_noalloc(m.n_verts, xyz.data_ptr(), m.n_tets, t.data_ptr(), len(query),
                                          query.data_ptr(), cell * m.h, 16, count.data_ptr(), out.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream)
        return rc, count.cpu().numpy(), out.cpu().numpy()

    rc, count, out = call(q, tets)
    assert rc == casim.CASIM_OK
    got = [(int(v), int(out[i, j])) for i, v in enumerate(prep.query) for j in range(count[i])]
    assert np.array_equal(np.array(got, dtype=np.int64).reshape(-1, 2), want)
    assert all((out[i, count[i]:] == -1).all() for i in range(len(count)))

    # ids out of range: refused, and the outputs stay as they were
    for bad_q, bad_t in ((m.n_verts, 0), (-1, 0), (None, m.n_verts), (None, -1)):
        q2, t2 = q.clone(), tets.clone()
        if bad_q is not None:
            q2[5] = bad_q
        else:
            t2[17, 2] = bad_t
        rc, count, out = call(q2, t2)
        assert rc == casim.CASIM_E_INVALID
        assert (count == -1).all() and (out == -1).all()

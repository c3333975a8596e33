"""The cell-sorted pair-distance histogram against all pairs, at the shapes where its cell grid
changes: one, two, three and more cells a side, cells that hold many molecules, ranges far below
the molecules' spacing, bins narrower than the FP32 error of a distance, replicas."""
import numpy as np
import pytest

from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


def all_pairs(s, x, nbins, dr):
    """floor(r / dr) of every pair of centres, formed as the definition forms them."""
    L = np.array(s.box)
    xm = x.reshape(s.M, s.na, 3)
    R = np.zeros((s.M, 3))
    for k in range(s.na):
        d = xm[:, k] - xm[:, 0]
        d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
        R += s.mass[k] * (xm[:, 0] + d)
    R /= s.mass.sum()
    R -= L * np.floor(R / L)
    R[R >= np.broadcast_to(L, R.shape)] -= np.broadcast_to(L, R.shape)[R >= np.broadcast_to(L, R.shape)]
    out = np.zeros(nbins, dtype=np.int64)
    for a in range(s.M - 1):
        d = R[a] - R[a + 1:]
        d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
        k = np.floor(np.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2]) / dr).astype(np.int64)
        out += np.bincount(k[k < nbins], minlength=nbins)
    return out


@pytest.mark.parametrize("M,box,nbins,dr", [
    (400, (14.0, 14.0, 20.4), 350, 0.02),      # the range is half the shortest edges: one cell there
    (700, (19.0, 19.5, 20.0), 100, 0.06),      # three cells
    (700, (13.0, 19.5, 28.0), 100, 0.06),      # two, three and four cells
    (1500, (28.0, 24.0, 22.0), 250, 0.02),     # four and five cells
    (1500, (28.0, 24.0, 22.0), 4096, 0.002),   # narrow bins
    (1500, (28.0, 24.0, 22.0), 2000, 1e-6),    # bins below the FP32 error: every pair in double
    (1501, (28.0, 24.0, 22.0), 3, 4e-1),       # range below the spacing
])
def test_counts_equal_all_pairs(M, box, nbins, dr):
    from paper_1806_10841_gb300 import adress

    s = inputs.tetra_system(M, box, 5.0, 2.5, seed=9)
    x, _ = inputs.tetra_state(s, min_contact=0.3, jitter=0.9)
    x[4 * 7:4 * 8] = x[4 * 3:4 * 4]  # two molecules on top of one another: distance zero
    for precision in ("fp32", "fp64"):
        sim = adress.AdResS(s, precision=precision)
        sim.set_state(x)
        got = sim.rdf_counts(nbins, dr)[0]
        again = sim.rdf_counts(nbins, dr)[0]
        sim.close()
        ref = all_pairs(s, x, nbins, dr)
        assert np.array_equal(got, ref) and np.array_equal(again, ref)


def test_replicas_of_unequal_boxes():
    from paper_1806_10841_gb300 import adress

    systems = inputs.replica_batch(5, m_lo=400, m_hi=1800, seed=11)
    x, _ = inputs.replica_states(systems, seed=12)
    sim = adress.AdResS(systems, precision="fp32")
    sim.set_state(x)
    got = sim.rdf_counts(200, 0.02)
    sim.close()
    a0 = np.concatenate([[0], np.cumsum([q.N for q in systems])])
    for r, s in enumerate(systems):
        assert np.array_equal(got[r], all_pairs(s, x[a0[r]:a0[r + 1]], 200, 0.02)), r

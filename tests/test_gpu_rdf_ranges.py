"""The pair-distance histogram out to half the box, where its cells are few and their molecules are
dealt out to many warps, against all pairs in double."""
import numpy as np
import pytest

from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


def beads(M, box, seed=5):
    """M single-atom molecules: their centres are their positions."""
    s = inputs.tetra_system(M, box, 5.0, 2.5, seed=seed)
    s.na, s.mass, s.bonds = 1, np.array([1.0]), np.zeros((0, 2), dtype=np.int32)
    return s


def all_pairs(x, box, nbins, dr):
    """Counts of floor(r / dr) over the pairs a < b, formed as the definition forms them."""
    import torch

    X = torch.from_numpy(x).cuda().T.contiguous()
    M = X.shape[1]
    out = torch.zeros(nbins, dtype=torch.int64, device="cuda")
    idx = torch.arange(M, device="cuda")
    rows = max(1, (1 << 27) // M)
    for a0 in range(0, M, rows):
        r2 = None
        for d in range(3):
            e = X[d, a0:a0 + rows, None] - X[d, None, a0:]
            L = float(box[d])
            e = torch.where(e > 0.5 * L, e - L, torch.where(e < -0.5 * L, e + L, e))
            r2 = e * e if r2 is None else r2 + e * e
        k = torch.floor(torch.sqrt(r2) / dr).to(torch.int64)
        keep = (idx[a0:] > idx[a0:a0 + rows, None]) & (k < nbins)
        out += torch.bincount(k[keep], minlength=nbins)
    return out.cpu().numpy()


def positions(M, box, spread, seed=3):
    """Uniform, or half of the molecules in an eighth of the box each way."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.0, 1.0, (M, 3))
    if spread == "clustered":
        x[::2] *= 0.125
    return np.minimum(x * np.array(box), np.nextafter(np.array(box), 0.0))


BOX = (64.0, 32.0, 32.0)


@pytest.mark.parametrize("spread", ["uniform", "clustered"])
@pytest.mark.parametrize("M", [37, 1003, 20011])
@pytest.mark.parametrize("nbins,dr", [
    (256, 0.0625),       # half the short edges: two cells by one by one
    (255, 0.0625),       # just below: four by two by two
    (700, 0.0146),       # a third: six by three by three
    (200, 0.04),         # a quarter: seven or eight by four by four
    (1, 16.0),
    (4096, 0.00390625),
])
def test_counts_equal_all_pairs(M, nbins, dr, spread):
    from paper_1806_10841_gb300 import adress

    s = beads(M, BOX)
    x = positions(M, BOX, spread)
    sim = adress.AdResS(s, precision="fp32", max_neighbors=8)
    sim.set_state(x)
    got = sim.rdf_counts(nbins, dr)[0]
    sim.close()
    assert np.array_equal(got, all_pairs(x, BOX, nbins, dr))


def test_boxes_of_unequal_fill():
    from paper_1806_10841_gb300 import adress

    boxes = [(16.0, 16.0, 16.0), BOX, (24.0, 48.0, 20.0)]
    sizes = [2003, 90, 5001]
    systems = [beads(M, box) for M, box in zip(sizes, boxes)]
    xs = [positions(M, box, "clustered", seed=r) for r, (M, box) in enumerate(zip(sizes, boxes))]
    sim = adress.AdResS(systems, precision="fp32", max_neighbors=8)
    sim.set_state(np.concatenate(xs))
    got = sim.rdf_counts(128, 0.0625)
    sim.close()
    for r in range(3):
        assert np.array_equal(got[r], all_pairs(xs[r], boxes[r], 128, 0.0625)), r


def test_more_pairs_in_a_cell_than_32_bits_count():
    """All molecules in one cell of many, so one warp counts every pair, all in one bin."""
    from paper_1806_10841_gb300 import adress

    M, box = 92_700, (200.0, 100.0, 100.0)
    assert M * (M - 1) // 2 > 2 ** 32
    s = beads(M, box)
    rng = np.random.default_rng(2)
    sim = adress.AdResS(s, precision="fp32", max_neighbors=8)
    sim.set_state(rng.uniform(1.0, 3.0, (M, 3)))  # farthest apart 3.5
    got = sim.rdf_counts(2, 2.5 * 1.5)[0]
    sim.close()
    assert got.tolist() == [M * (M - 1) // 2, 0]

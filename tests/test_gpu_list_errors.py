"""What a list build reports and leaves behind when a list does not fit or a wait gives up."""
import numpy as np
import pytest

from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


def lists_of(sim):
    items, nn, nbr = sim.neighbour_lists()
    return items, nn, [nbr[t, :nn[t]].copy() for t in range(len(nn))]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_one_overflowing_molecule_in_a_dense_cell_grows_the_capacity(seed, precision):
    """Dense cells are the build's last phase; the longest list alone does not fit.  The verdict on
    the build must wait for it: lists and forces are those of a capacity that fits at once."""
    from paper_1806_10841_gb300 import adress

    s = inputs.scaled_c3(8000, skin=0.8, seed=seed)
    x, _ = inputs.water_state(s)
    ref = adress.AdResS(s, precision=precision)
    ref.set_state(x)
    f_ref, _ = ref.forces()
    items, nn, rows = lists_of(ref)
    st = ref.list_stats()
    ref.close()
    assert 27 * s.M / st["n_cells"] > 160  # candidates of a cell: more than the sparse phase stages
    longest = int(nn.max())
    assert longest == st["max_nn"] and (nn == longest).sum() < s.M // 100
    for build in (lambda sim: sim.build_lists(), lambda sim: sim.compute_forces(energies=False)):
        sim = adress.AdResS(s, precision=precision, max_neighbors=longest - 1)
        sim.set_state(x)
        build(sim)
        assert sim.list_stats()["capacity"] >= longest
        items2, nn2, rows2 = lists_of(sim)
        assert np.array_equal(items, items2) and np.array_equal(nn, nn2)
        assert all(np.array_equal(a, b) for a, b in zip(rows, rows2))
        f, _ = sim.forces()
        assert np.array_equal(f, f_ref)
        sim.check()
        sim.close()

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


TIMEOUT = 6


def reported(call):
    from paper_1806_10841_gb300 import adress

    with pytest.raises(adress.AdressError) as ei:
        call()
    assert ei.value.status == TIMEOUT


def per_sm(n):
    import torch

    return n * torch.cuda.get_device_properties(0).multi_processor_count


# one block, the run kernel, a step and a list kernel per step; dense cells
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("make,M", [(inputs.scaled_c2, 216), (inputs.scaled_c2, 4001), (inputs.scaled_c2, (161, 3)),
                                    (inputs.scaled_c3, 4001)])
def test_a_grid_barrier_that_gives_up_is_reported_and_the_next_call_is_clean(make, M, precision):
    """Barriers limited to zero polls give up at once: a build returns the timeout, a run reports it
    at the check.  With the default limit again forces and trajectory are those of a fresh handle."""
    from paper_1806_10841_gb300 import adress

    M = per_sm(M[0]) + M[1] if isinstance(M, tuple) else M
    s = make(M, seed=5)
    x, v = inputs.tetra_state(s) if s.na == 4 else inputs.water_state(s)

    def run(sim):
        sim.set_state(x, v)
        sim.set_step(0)
        f, e = sim.forces()
        sim.run(60, sample_every=9)
        sim.check()
        return (f, *sim.get_state()), e

    ref = adress.AdResS(s, precision=precision)
    want, e_ref = run(ref)
    ref.close()
    sim = adress.AdResS(s, precision=precision)
    run(sim)
    calls = (sim.build_lists, lambda: sim.compute_forces(True), lambda: sim.compute_forces(False))
    for call in calls:
        sim.set_state(x, v)
        sim.set_limit(sim.LIMIT_BARRIER_POLLS, 0)
        reported(call)
        reported(sim.check)
        sim.check()  # reported once
        with pytest.raises(adress.AdressError):
            sim.step(1)  # no lists
        sim.set_limit(sim.LIMIT_BARRIER_POLLS, -1)
        got, e = run(sim)
        assert e == e_ref and all(np.array_equal(a, b) for a, b in zip(got, want))
    # lists due in the middle of a run, the run kernel's own barriers
    sim.set_limit(sim.LIMIT_BARRIER_POLLS, 0)
    sim.run(100, sample_every=9)
    reported(sim.check)
    sim.set_limit(sim.LIMIT_BARRIER_POLLS, -1)
    got, e = run(sim)
    assert e == e_ref and all(np.array_equal(a, b) for a, b in zip(got, want))
    sim.close()


def spheres(scheme):
    s = inputs.scaled_c2(3000, seed=7, scheme=scheme)
    L = np.array(s.box)
    s.d_at, s.d_hy = 4.0, 3.0
    s.centers = np.array([[0.2, 0.5, 0.5], [0.7, 0.3, 0.8]]) * L
    s.tf = 0.3 * np.cos(np.arange(int((s.d_at + s.d_hy) / s.tf_dx) + 2))
    return s


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("make", [lambda: spheres(0), lambda: spheres(1), lambda: inputs.scaled_c2(3000, scheme=1),
                                  lambda: inputs.scaled_c3(3000)])
def test_forces_behind_a_first_build_that_gave_up(make, precision):
    """Nothing was ever mapped when the first build of a handle gives up and the forces run behind
    it: they read the arrays as the handle was created, and the next call is that of a fresh handle."""
    from paper_1806_10841_gb300 import adress

    s = make()
    x, _ = inputs.tetra_state(s) if s.na == 4 else inputs.water_state(s)
    ref = adress.AdResS(s, precision=precision)
    ref.set_state(x)
    f_ref, e_ref = ref.forces()
    ref.check()
    ref.close()
    sim = adress.AdResS(s, precision=precision)
    sim.set_state(x)
    sim.set_limit(sim.LIMIT_BARRIER_POLLS, 0)
    reported(lambda: sim.compute_forces(True))
    reported(sim.check)
    reported(lambda: sim.compute_forces(False))
    reported(sim.check)
    sim.set_limit(sim.LIMIT_BARRIER_POLLS, -1)
    f, e = sim.forces()
    sim.check()
    assert e == e_ref and np.array_equal(f, f_ref)
    sim.close()


@pytest.mark.parametrize("max_neighbors", [0, 4])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_learned_force_behind_a_build_that_gave_up(precision, max_neighbors):
    """The network's candidate pairs belong to the last complete build: none are evaluated behind
    one that gave up, the first of a handle or a later one, with buffers that grew (four neighbours)
    or not, nor in the steps that follow."""
    from paper_1806_10841_gb300 import adress

    s = inputs.scaled_c2(3000, seed=8)
    x, v = inputs.tetra_state(s)
    rng = np.random.default_rng(5)
    params = dict(W1=rng.normal(0, 0.2, (64, 9)), b1=rng.normal(0, 0.1, 64), W2=rng.normal(0, 0.1, (64, 64)),
                  b2=rng.normal(0, 0.1, 64), w3=rng.normal(0, 0.1, 64), b3=0.1)

    def fresh(cap):
        sim = adress.AdResS(s, precision=precision, max_neighbors=cap)
        sim.mlp_set(params, np.full(9, 0.1), np.full(9, 0.8), 3.0)
        sim.set_cg_mode(1)
        return sim

    def run(sim):
        sim.set_state(x, v)
        sim.set_step(0)
        sim.compute_forces(energies=False)
        f = sim.get_state()[2]
        sim.run(20)
        sim.check()
        return (f, *sim.get_state())

    ref = fresh(0)
    want = run(ref)
    ref.close()
    sim = fresh(max_neighbors)
    for _ in range(2):
        sim.set_state(x, v)
        sim.set_limit(sim.LIMIT_BARRIER_POLLS, 0)
        reported(lambda: sim.compute_forces(False))
        reported(sim.check)
        sim.set_limit(sim.LIMIT_BARRIER_POLLS, -1)
        assert all(np.array_equal(a, b) for a, b in zip(run(sim), want))
    sim.set_limit(sim.LIMIT_BARRIER_POLLS, 0)
    sim.run(100)
    reported(sim.check)
    sim.set_limit(sim.LIMIT_BARRIER_POLLS, -1)
    assert all(np.array_equal(a, b) for a, b in zip(run(sim), want))
    sim.close()

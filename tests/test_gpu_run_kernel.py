"""The MD step at the sizes where its launch form changes: the run kernel (all steps in one
cooperative launch) against the step and list kernels, the lanes per molecule, ragged tiles."""
import numpy as np
import pytest

import oracle
from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


def per_sm(n):
    """n molecules per multiprocessor."""
    import torch

    return n * torch.cuda.get_device_properties(0).multi_processor_count


# envelopes of the 100-step divergence curve (tests/test_gpu_parity.py); 30 steps stay inside
ENV = {"fp64": (1e-11, 1e-9), "fp32": (1e-5, 1e-3)}


# fixed sizes, or (molecules per SM at an edge of a rule, molecules past it)
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("precision,size", [("fp64", 47), ("fp64", 1001), ("fp64", (32, 0)), ("fp64", (32, 1)),
                                            ("fp32", 47), ("fp32", 1001), ("fp32", (40, 0)), ("fp32", (40, 1)),
                                            ("fp32", (160, 0)), ("fp32", (160, 1))])
def test_trajectory_at_the_edges_of_the_launch_rule(size, precision, scheme):
    from paper_1806_10841_gb300 import adress

    M = per_sm(size[0]) + size[1] if isinstance(size, tuple) else size
    s = inputs.scaled_c2(M, seed=3, scheme=scheme)
    x, v = inputs.tetra_state(s)
    o = oracle.Oracle(s)
    f, _ = o.forces(x)
    sim = adress.AdResS(s, precision=precision)
    sim.set_state(x, v)
    sim.compute_forces(energies=False)
    sim.run(25, sample_every=7)  # stretches of 7, a ragged last one
    sim.step(5)
    sim.check()
    assert sim.get_step() == 30
    counts, n = sim.density_get()
    xg, vg, _ = sim.get_state()
    stats = sim.list_stats()
    sim.close()
    xo, vo, fo, ref = x, v, f, 0
    for k in range(1, 26):
        xo, vo, fo = o.run(xo, vo, fo, k - 1, 1)
        if k % 7 == 0:
            ref = ref + o.density(xo, len(s.tf), 10)[0]
    xo, vo, fo = o.run(xo, vo, fo, 25, 5)
    L = np.array(s.box)
    dx = xg - xo
    dx -= L * np.rint(dx / L)
    assert np.abs(dx).max() < ENV[precision][0] and np.abs(vg - vo).max() < ENV[precision][1]
    assert n == 3 and np.array_equal(counts, ref)
    assert stats["rebuilds"] >= 1 and stats["n_hr"] + stats["n_cg"] == s.M


@pytest.mark.parametrize("na", [1, 2, 3])
@pytest.mark.parametrize("M", [300, 7001])
def test_smaller_molecules_through_the_run_kernel(na, M):
    """One to three atoms per molecule: pairs of atoms with an odd or missing second one."""
    from paper_1806_10841_gb300 import adress

    s = inputs.scaled_c2(M, seed=4)
    s.na, s.mass = na, np.array([1.0, 2.0, 1.5])[:na]
    s.bonds = inputs.tetra_bonds()[[i for i, b in enumerate(inputs.tetra_bonds()) if b.max() < na]].reshape(-1, 2)
    x, v = inputs.tetra_state(s, body=inputs.tetra_sites()[:na])
    o = oracle.Oracle(s)
    f, e = o.forces(x)
    sim = adress.AdResS(s, precision="fp32")
    sim.set_state(x, v)
    fg, eg = sim.forces()
    assert np.sqrt(((fg - f) ** 2).sum() / (f ** 2).sum()) <= 2e-5
    assert eg["E_at"] == pytest.approx(e["E_at"], rel=2e-5, abs=1e-6) and eg["virial"] == pytest.approx(e["virial"], rel=2e-5, abs=1e-3)
    sim.close()


@pytest.mark.parametrize("na", [1, 2, 3])
@pytest.mark.parametrize("M", [300, 7001])
def test_trajectory_of_smaller_molecules(na, M):
    """The same molecules with their centres apart by 1.6 (the coarse-grained force of a closer
    pair is thousands of times the thermal one), 20 steps."""
    from paper_1806_10841_gb300 import adress

    s = inputs.scaled_c2(M, seed=4)
    s.na, s.mass = na, np.array([1.0, 2.0, 1.5])[:na]
    s.bonds = inputs.tetra_bonds()[[i for i, b in enumerate(inputs.tetra_bonds()) if b.max() < na]].reshape(-1, 2)
    x, v = inputs.tetra_state(s, body=inputs.tetra_sites()[:na], min_contact=1.6, jitter=0.05)
    o = oracle.Oracle(s)
    f, _ = o.forces(x)
    sim = adress.AdResS(s, precision="fp32")
    sim.set_state(x, v)
    sim.compute_forces(energies=False)
    sim.step(20)
    sim.check()
    xg, vg, _ = sim.get_state()
    sim.close()
    xo, vo, _ = o.run(x, v, f, 0, 20)
    L = np.array(s.box)
    dx = xg - xo
    dx -= L * np.rint(dx / L)
    assert np.abs(dx).max() < ENV["fp32"][0] and np.abs(vg - vo).max() < ENV["fp32"][1]


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("size", [1500, (64, 1), (160, 1), (320, 1)])
def test_water_forces_at_every_lane_count(size, scheme):
    """The water-like fluid at each choice of lanes per molecule: forces, energies (FP32, the
    bound of tests/test_gpu_water.py) and a few steps."""
    from paper_1806_10841_gb300 import adress

    M = per_sm(size[0]) + size[1] if isinstance(size, tuple) else size
    s = inputs.scaled_c3(M, seed=6, scheme=scheme)
    x, v = inputs.water_state(s)
    x = x + np.random.default_rng(1).normal(0, 0.002, x.shape)  # bonded terms off their minimum
    x = np.mod(x, np.array(s.box))
    o = oracle.Oracle(s)
    f, e = o.forces(x)
    sim = adress.AdResS(s, precision="fp32")
    sim.set_state(x, v)
    fg, eg = sim.forces()
    assert np.sqrt(((fg - f) ** 2).sum() / (f ** 2).sum()) <= 2e-5
    scale = sum(abs(e[k]) for k in ("E_at", "E_cg", "E_bond"))
    for k in ("E_at", "E_cg", "E_bond"):
        assert abs(eg[k] - e[k]) <= 2e-5 * scale, k
    sim.step(3)
    sim.check()
    xg, _, _ = sim.get_state()
    sim.close()
    xo, _, _ = o.run(x, v, f, 0, 3)
    L = np.array(s.box)
    dx = xg - xo
    dx -= L * np.rint(dx / L)
    assert np.abs(dx).max() < ENV["fp32"][0]

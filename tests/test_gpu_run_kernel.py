"""The MD step at the sizes where its launch form changes: the run kernel (all steps in one
cooperative launch) against the step and list kernels, ragged tiles, a single tile."""
import numpy as np
import pytest

import oracle
from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


def resident_edge():
    """Molecules of one 32-molecule tile per multiprocessor."""
    import torch

    return 32 * torch.cuda.get_device_properties(0).multi_processor_count


# envelopes of the 100-step divergence curve (tests/test_gpu_parity.py); 30 steps stay inside
ENV = {"fp64": (1e-11, 1e-9), "fp32": (1e-5, 1e-3)}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("size", [47, 1001, "edge", "edge+1"])
def test_trajectory_at_the_edges_of_the_launch_rule(size, precision):
    from paper_1806_10841_gb300 import adress

    M = resident_edge() + (size == "edge+1") if isinstance(size, str) else size
    s = inputs.scaled_c2(M, seed=3)
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

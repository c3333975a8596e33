"""The force kernels' block size changes no result: systems of the run kernel (whose blocks keep their
size) and of the step kernel."""
import numpy as np
import pytest

from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("M", [301, 4001, 30011])
def test_trajectories_agree_bit_for_bit(M, precision):
    from paper_1806_10841_gb300 import adress

    s = inputs.scaled_c2(M, seed=13)
    x, v = inputs.tetra_state(s)
    out = []
    for block in (128, 64, 32):
        sim = adress.AdResS(s, precision=precision)
        sim.set_tuning(block, s.skin)
        sim.set_state(x, v)
        sim.compute_forces(energies=False)
        sim.run(40, sample_every=7)
        sim.check()
        out.append((*sim.get_state(), *sim.density_get()))
        sim.close()
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(o, out[0]))

"""The step kernel of the learned-force mode (ordered force sums) at ragged sizes and every number
of atoms per molecule: in an all-atomistic system the network has no weight, so forces, energies
and a short trajectory are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("na", [1, 2, 3, 4])
@pytest.mark.parametrize("M", [47, 129, 3001])
def test_ordered_sums_match_oracle(na, M):
    from paper_1806_10841_gb300 import adress

    s = inputs.scaled_c2(M, seed=4)
    s.d_at = 1e3
    s.na, s.mass = na, np.array([1.0, 2.0, 1.5, 1.0])[:na]
    s.bonds = inputs.tetra_bonds()[[i for i, b in enumerate(inputs.tetra_bonds()) if b.max() < na]].reshape(-1, 2)
    x, v = inputs.tetra_state(s, body=inputs.tetra_sites()[:na], min_contact=1.6, jitter=0.05)
    o = oracle.Oracle(s)
    f, e = o.forces(x)
    sim = adress.AdResS(s, precision="fp32")
    rng = np.random.default_rng(1)
    params = dict(W1=rng.normal(0, 0.2, (64, 9)), b1=np.zeros(64), W2=rng.normal(0, 0.2, (64, 64)), b2=np.zeros(64),
                  w3=rng.normal(0, 0.2, 64), b3=0.0)
    sim.mlp_set(params, np.zeros(9), np.ones(9), 1.0)
    sim.set_cg_mode(1)
    sim.set_state(x, v)
    fg, eg = sim.forces()
    sim.step(20)
    sim.check()
    xg, vg, _ = sim.get_state()
    sim.close()
    # the FP32 path's bound (2e-5 relative) and the envelope of the 100-step divergence curve
    # (tests/test_gpu_parity.py); a single loose atom may feel no force at all
    assert np.sqrt(((fg - f) ** 2).sum()) <= 2e-5 * np.sqrt((f ** 2).sum()) + 1e-12
    scale = abs(e["E_at"]) + abs(e["E_bond"])
    for k in ("E_at", "E_bond", "virial"):
        assert abs(eg[k] - e[k]) <= 2e-5 * max(scale, abs(e["virial"])) + 1e-12, k
    xo, vo, _ = o.run(x, v, f, 0, 20)
    L = np.array(s.box)
    dx = xg - xo
    dx -= L * np.rint(dx / L)
    assert np.abs(dx).max() < 1e-5 and np.abs(vg - vo).max() < 1e-3

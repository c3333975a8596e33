"""The FP64 path's FP32 pre-test of pairs: centres placed within 1e-11 .. 1e-5 of the cutoffs, on
either side, in boxes of very different size, must be decided as FP64 decides them."""
import numpy as np
import pytest

import oracle
from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


# (in the longest box the fixed-point centres are good to 2e-5, the coordinates to 1e-11)
@pytest.mark.parametrize("na,L,nearest", [(1, 24.0, -11), (4, 24.0, -11), (1, 800.0, -11), (4, 800.0, -11), (1, 1.0e5, -9)])
@pytest.mark.parametrize("scheme", [0, 1])
def test_pairs_at_the_cutoffs(na, L, nearest, scheme):
    from paper_1806_10841_gb300 import adress

    n = 40  # molecule pairs, centres a cutoff apart to within 10^nearest .. 1e-5 of it
    box = (L, 24.0, 24.0)
    s = inputs.tetra_system(2 * n, box, 8.0, 4.0, seed=2, scheme=scheme)
    s.na, s.mass = na, np.ones(na)
    if na == 1:
        s.bonds = np.zeros((0, 2), np.int32)
    s.cg_F = s.cg_F + 1.0  # a force step at rc_cg, so that a wrong decision shows
    rng = np.random.default_rng(5)
    body = inputs.tetra_sites()[:na]
    x = np.zeros((2 * n, na, 3))
    for k in range(n):
        # along x across the whole resolution range, pairs far from one another in y and z
        c = np.array([s.xc - 0.4 * L + 0.8 * L * k / n if L < 100 else s.xc - 11 + 22.0 * k / n,
                      4.0 + 16.0 * (k % 3) / 2 * 0.75, 4.0 + 16.0 * (k // 3 % 3) / 2 * 0.75])
        u = rng.normal(size=3)
        u /= np.linalg.norm(u)
        rc = s.rc_cg if k % 2 else s.rc_at
        d = rc * (1 + rng.choice([-1, 1]) * 10.0 ** rng.uniform(nearest, -5))
        x[2 * k] = c + body
        x[2 * k + 1] = c + d * u + (body if na == 1 or k % 2 else -body)
    x = np.mod(x.reshape(-1, 3), np.array(box))
    f, e = oracle.Oracle(s).forces(x)
    sim = adress.AdResS(s, precision="fp64")
    sim.set_state(x)
    fg, eg = sim.forces()
    sim.check()
    sim.close()
    assert np.abs(fg - f).max() <= 1e-9 * max(1.0, np.abs(f).max())
    for key in e:
        assert eg[key] == pytest.approx(float(e[key]), rel=1e-10, abs=1e-10), key

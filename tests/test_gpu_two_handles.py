"""Two handles that step at the same time, each from its own thread on its own stream: their
cooperative kernels share the device, and each gives what it gives alone."""
import threading

import numpy as np
import pytest

from paper_1806_10841_gb300 import inputs

pytestmark = pytest.mark.gpu


def block(sim, x, v):
    sim.set_state(x, v)
    sim.set_step(0)
    f, _ = sim.forces()
    for _ in range(4):
        sim.run(50, sample_every=7)
    sim.check()
    return (f, *sim.get_state())


# the run kernel with itself, with the list kernel of a larger system, the list kernels of two
@pytest.mark.parametrize("sizes", [(1500, 20001), (6007, 30011), (30011, 40009)])
def test_two_handles_at_once(sizes):
    import torch
    from paper_1806_10841_gb300 import adress

    systems = [inputs.scaled_c2(M, seed=31 + M % 7) for M in sizes]
    states = [inputs.tetra_state(s) for s in systems]
    sims = [adress.AdResS(s, precision="fp32", stream=torch.cuda.Stream()) for s in systems]
    for sim in sims:
        sim.set_limit(sim.LIMIT_BARRIER_POLLS, 1 << 20)  # a fraction of a second
    alone = [block(sim, *st) for sim, st in zip(sims, states)]
    out, errors = [None, None], []

    def work(k):
        try:
            for _ in range(5):
                out[k] = block(sims[k], *states[k])
                assert all(np.array_equal(a, b) for a, b in zip(out[k], alone[k]))
        except Exception as e:  # reported by the main thread
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for sim in sims:
        sim.close()
    assert not errors, errors

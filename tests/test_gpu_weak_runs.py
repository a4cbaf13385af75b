"""Runs whose sub-steps lie on both sides of the step sizes that the short
solve of weak pairs takes, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1402_3325_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,dt", [(4, 6.5e-19), (8, 5e-19)])
def test_composed_step_across_the_smallest_step_size(order, dt):
    # cold, so that the velocities after the step are its increments: 3 and 27
    # sub-steps, each with 1e-13 of its own increments, which are up to 8 times
    # the whole step's; in a fresh context, whose scratch holds nothing else
    import torch
    from paper_1402_3325_gb300 import sakura as sk
    s = ics.random_cluster(1000, seed=4)
    s.v[:] = 0.0
    sk.finalize()
    sk.init(0, stream=torch.cuda.current_stream().cuda_stream, guess=sk.GUESS_FP32)
    state, mass = torch.tensor(s.soa(), device="cuda"), torch.tensor(s.m, device="cuda")
    sk.step(state, mass, dt, order)
    sk.check()
    r, v = ics.from_soa(state.cpu().numpy())
    rc, r1, v1 = oracle.evolve(s.m, s.r, s.v, dt, 1, order)
    assert rc == oracle.OK
    assert np.array_equal(r, r1)
    scale = np.sqrt((v1 ** 2).sum(1).mean())
    assert np.abs(v - v1).max() <= 27 * 8 * 1e-13 * scale

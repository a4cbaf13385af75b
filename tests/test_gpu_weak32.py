"""FP32-class pairs of the mixed form that move little (csrc/kepler_weak32.cuh)
in the row-group kernel, at the edges of tiles and of the limits."""
import os

import numpy as np
import pytest

import oracle
from paper_1402_3325_gb300 import ics

pytestmark = pytest.mark.gpu
NCPU = os.cpu_count() or 1


# an FP32 pair's increments are within 16 units of 2^-24 of their size (the
# iteration's are within 10, the direct solve's within 7); 1.5 covers the
# change of 1 / r^2 along the step
def _bounds(s, dt):
    d = s.r[:, None] - s.r[None]
    r2 = (d ** 2).sum(2) + np.where(np.eye(s.n, dtype=bool), np.inf, 0.0)
    ev = 16 * 2.0 ** -24 * 1.5 * abs(dt) * (s.m / r2).sum(1)
    return abs(dt) * ev + 1e-13, ev + 1e-13


@pytest.mark.parametrize("order", [2, 1, -1])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 65, 256, 257, 1025])
def test_mixed_step_of_weak_and_general_pairs(n, order):
    import torch
    from paper_1402_3325_gb300 import sakura as sk
    s = ics.random_cluster(n, seed=n, mass_spread=2.0)
    for dt in (s.dt, -s.dt, 16 * s.dt):  # the last: some pairs beyond the limits
        sk.init(0, stream=torch.cuda.current_stream().cuda_stream, precision=sk.PREC_MIXED,
                mixed_rule=sk.MIXED_RULE_HYP, guess=sk.GUESS_FP32, flags=sk.FLAG_STATS)
        state, mass = torch.tensor(s.soa(), device="cuda"), torch.tensor(s.m, device="cuda")
        classes = int(sk.pair_classes(state, mass, dt, order).sum())
        sk.get_stats(reset=True)
        sk.step(state, mass, dt, order)
        sk.check()
        assert sk.get_stats(reset=True)["fp32_pairs"] == classes
        rc, r, v = oracle.step(s.m, s.r, s.v, dt, order, nthreads=NCPU)
        assert rc == oracle.OK
        got = ics.from_soa(state.cpu().numpy())
        for a, b, tol in zip(got, (r, v), _bounds(s, dt)):
            assert (np.linalg.norm(a - b, axis=1) <= tol + 1e-12 * np.linalg.norm(b, axis=1)).all()


@pytest.mark.parametrize("n", [160, 161, 352, 353, 640, 641])
def test_mixed_step_on_either_side_of_its_kernels_ranges(n):
    import torch
    from paper_1402_3325_gb300 import sakura as sk
    s = ics.random_cluster(n, seed=n, mass_spread=2.0)
    sk.init(0, stream=torch.cuda.current_stream().cuda_stream, precision=sk.PREC_MIXED,
            mixed_rule=sk.MIXED_RULE_HYP, guess=sk.GUESS_FP32, flags=sk.FLAG_STATS)
    state, mass = torch.tensor(s.soa(), device="cuda"), torch.tensor(s.m, device="cuda")
    classes = int(sk.pair_classes(state, mass, s.dt, 2).sum())
    run, one = state.clone(), state.clone()
    sk.get_stats(reset=True)
    sk.step(state, mass, s.dt, 2)
    st = sk.get_stats(reset=True)
    assert st["fp32_pairs"] == classes and st["group_launches"] == (1 if n > 640 else 0)
    rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    assert rc == oracle.OK
    for a, b, tol in zip(ics.from_soa(state.cpu().numpy()), (r, v), _bounds(s, s.dt)):
        assert (np.linalg.norm(a - b, axis=1) <= tol + 1e-12 * np.linalg.norm(b, axis=1)).all()
    # a run's steps (drifts fused into the sums on tiles) are the single ones
    sk.evolve(run, mass, s.dt, 2, 3)
    for _ in range(3):
        sk.step(one, mass, s.dt, 2)
    sk.check()
    assert torch.equal(run, one)

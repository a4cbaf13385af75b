"""The weak pairs of the seeded FP64 step and of the double-word form (csrc/kepler_weak.cuh, csrc/step_weak.cu)
on tiles and in row groups against the oracle, at ragged sizes and for mixes
of weak and strong pairs."""
import os

import numpy as np
import pytest

import oracle
from paper_1402_3325_gb300 import ics

pytestmark = pytest.mark.gpu
TOL = 1e-12  # as tests/test_gpu_step.py
NCPU = os.cpu_count() or 1


def _step(s, dt, order=2, nsteps=1, **options):
    import torch
    from paper_1402_3325_gb300 import sakura as sk
    options = {"guess": sk.GUESS_FP32, **options}
    sk.init(0, stream=torch.cuda.current_stream().cuda_stream, **options)
    if options["guess"] == sk.GUESS_LEARNED:
        from paper_1402_3325_gb300 import learned
        learned.load_default()
    state = torch.tensor(s.soa(), device="cuda")
    mass = torch.tensor(s.m, device="cuda")
    sk.get_stats(reset=True)
    if nsteps == 1:
        sk.step(state, mass, dt, order)
    else:
        sk.evolve(state, mass, dt, order, nsteps)
    sk.check()
    return ics.from_soa(state.cpu().numpy()), sk.get_stats(reset=True)


def _close(got, ref, tol=TOL):
    for a, b in zip(got, ref):
        scale = np.maximum(np.linalg.norm(b, axis=1), np.sqrt((b ** 2).sum(1).mean()))
        assert (np.linalg.norm(a - b, axis=1) <= tol * scale).all()


def _kinds(n):
    yield "cluster", ics.random_cluster(n, seed=n, mass_spread=3.0)
    s = ics.random_cluster(n, seed=n + 1)       # in a plane: exact zero differences
    s.r[:, 2] = s.v[:, 2] = 0.0
    yield "planar", s
    if n < 1000:                                # fast: every pair strong (at 1000 bodies the
        s = ics.random_cluster(n, seed=n + 2)   # map amplifies any rounding to 1e-9)
        yield "swarm", ics.System(s.m, s.r * 1e-3, s.v * 100.0, s.dt)
    s = ics.random_cluster(n, seed=n + 3)       # separations of exact powers of two
    s.r[:, :] = np.stack(np.unravel_index(np.arange(n), (16, 16, 32)), 1) * 2.0 ** -2
    yield "lattice", s


@pytest.mark.parametrize("flag", [32, 64], ids=["tiles", "groups"])
@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "df64"])
@pytest.mark.parametrize("n", [21, 32, 33, 64, 95, 129, 1000])
def test_weak_step_matches_oracle(n, precision, flag):
    for name, s in _kinds(n):
        got, st = _step(s, s.dt, flags=flag | 2, precision=precision)
        rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
        assert rc == oracle.OK
        _close(got, (r, v))
        assert st["iters"] >= st["solves"]
        again, _ = _step(s, s.dt, flags=flag | 2, precision=precision)
        assert np.array_equal(got[0], again[0]) and np.array_equal(got[1], again[1])
        if name == "planar":
            assert not got[0][:, 2].any() and not got[1][:, 2].any()


@pytest.mark.parametrize("flag", [32, 64], ids=["tiles", "groups"])
@pytest.mark.parametrize("blocks", [1, 5, 151, 4000])
def test_weak_step_on_any_grid(flag, blocks):
    s = ics.plummer_binaries(700, seed=4)
    s = ics.System(s.m, s.r, s.v, 2.0 ** -7)  # a few per cent of strong pairs
    got, _ = _step(s, s.dt, flags=flag, grid_blocks=blocks)
    rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    _close(got, (r, v))


@pytest.mark.parametrize("flag", [32, 64], ids=["tiles", "groups"])
@pytest.mark.parametrize("order,dt", [(4, 2.0 ** -8), (2, -(2.0 ** -8)), (2, 1e-17), (2, 1e-19),
                                      (2, 0.0), (2, 2.0)])
def test_weak_step_orders_and_step_sizes(flag, order, dt):
    s = ics.random_cluster(150, seed=8)
    got, _ = _step(s, dt, order, 3, flags=flag)
    rc, r, v = oracle.evolve(s.m, s.r, s.v, dt, 3, order, nthreads=NCPU)
    _close(got, (r, v), 1e-10 if dt == 2.0 else 12 * TOL)


@pytest.mark.parametrize("flag", [32, 64], ids=["tiles", "groups"])
@pytest.mark.parametrize("kind", ["bh", "radial", "bound"])
def test_weak_literal_mixed_step_keeps_the_classes(kind, flag):
    # e_max < 1: bound pairs only; a radially expanding cluster (h^2 = 0 up to
    # rounding in every pair) and one with every pair bound
    from paper_1402_3325_gb300 import sakura as sk
    s = ics.bh_cluster(417, seed=6)
    if kind == "radial":
        s.v = 3.0 * s.r
    if kind == "bound":
        s = ics.random_cluster(417, seed=6)
        s.v *= 0.02
    opts = dict(precision=sk.PREC_MIXED, mixed_rule=sk.MIXED_RULE_LITERAL, flags=flag | 2)
    got, st = _step(s, s.dt, **opts)
    import torch
    classes = sk.pair_classes(torch.tensor(s.soa(), device="cuda"),
                              torch.tensor(s.m, device="cuda"), s.dt, 2)
    assert st["fp32_pairs"] == int(classes.sum())
    rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    # a pair in single precision: 2^-21 of its increment, the largest of
    # which is below 0.02 of the scale here
    _close(got, (r, v), 1e-8)


@pytest.mark.parametrize("flag", [32, 64], ids=["tiles", "groups"])
@pytest.mark.parametrize("guess", [0, 1, 2], ids=["standard", "learned", "taylor"])
@pytest.mark.parametrize("n", [33, 129, 1000])
def test_weak_step_with_the_other_guesses(n, guess, flag):
    # (without statistics: with them every pair iterates from its guess)
    for name, s in _kinds(n):
        got, _ = _step(s, s.dt, flags=flag, guess=guess)
        rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
        _close(got, (r, v))


@pytest.mark.parametrize("guess", [0, 3])
def test_one_iteration_without_bisection_still_fails_or_carries(guess):
    # from t / r0 one evaluation converges no pair; the seed's carries
    from paper_1402_3325_gb300 import sakura as sk
    s = ics.random_cluster(64, seed=2)
    if guess == 3:
        got, _ = _step(s, s.dt, guess=guess, kepler_max_iter=1, kepler_bisection=0)
        rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
        _close(got, (r, v))
    else:
        with pytest.raises(sk.SakuraError):
            _step(s, s.dt, guess=guess, kepler_max_iter=1, kepler_bisection=0)


@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "df64"])
@pytest.mark.parametrize("n", [21, 256, 257, 512, 513, 736, 768, 769, 928, 929])
def test_small_weak_step_at_the_ends_of_its_ranges(n, precision):
    # 2, 4 and 8 tile-steps per warp (152 SMs), then the general tile kernel,
    # which grid_blocks forces too
    s = ics.random_cluster(n, seed=n, mass_spread=3.0)
    got, _ = _step(s, s.dt, 4, 2, precision=precision)
    general, _ = _step(s, s.dt, 4, 2, precision=precision, grid_blocks=7)
    rc, r, v = oracle.evolve(s.m, s.r, s.v, s.dt, 2, 4, nthreads=NCPU)
    assert rc == oracle.OK
    _close(got, (r, v), 12 * TOL)
    _close(got, general, 12 * TOL)


@pytest.mark.parametrize("order,nsteps", [(2, 1), (2, 2), (4, 1)])
def test_small_weak_step_on_pinned_host_arrays(order, nsteps):
    import torch
    from paper_1402_3325_gb300 import sakura as sk
    s = ics.plummer(100, seed=3)
    ref, _ = _step(s, s.dt, order, nsteps)
    state = torch.tensor(s.soa()).pin_memory().numpy()
    mass = torch.tensor(s.m).pin_memory().numpy()
    sk.evolve_host(state, mass, s.dt, order, nsteps)
    got = ics.from_soa(state)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])

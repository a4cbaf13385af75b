"""Steps whose pairs are partly or mostly strong (csrc/step_weak.cu): tiles of
both kinds of pairs, and the choice of the kernels that solve every pair,
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1402_3325_gb300 import ics
from test_gpu_weak import (NCPU, TOL, _close, _step,
                           test_weak_literal_mixed_step_keeps_the_classes as _keeps_the_classes)

pytestmark = pytest.mark.gpu

FORMS = {"fp64": {}, "standard": {"guess": 0}, "learned": {"guess": 1}, "taylor": {"guess": 2},
         "df64": {"precision": 2},
         # no pair is far enough for single precision
         "literal": {"precision": 1, "mixed_rule": 0, "mixed_r_min": 1e9}}


def _clumps(n, clump):
    """A wide, slow cluster with a fast clump, whose own pairs are strong:
    clump gives its members within each of the first five blocks of 32."""
    s = ics.random_cluster(n, seed=n, mass_spread=3.0)
    r, v = s.r * 30.0, s.v.copy()
    inside = np.concatenate([32 * b + np.asarray(clump(b)) for b in range(min(5, (n + 31) // 32))])
    inside = inside[inside < n].astype(int)
    r[inside], v[inside] = s.r[inside] * 0.03, s.v[inside] * 10.0
    return ics.System(s.m, r, v, s.dt)


# 16 members, shifted by 4 from block to block: a tile's steps have 0 to 16
# strong pairs, those with more than 8 solved in place; 13 members; all; 3:
# batches that straddle tiles
CLUMPS = {"shifted": lambda b: np.arange(16) + 4 * (b % 4), "queued": lambda b: np.arange(13),
          "all": lambda b: np.arange(32), "few": lambda b: np.arange(3)}


def _tolerance(s, form):
    """TOL, and 16 times what the oracle's result moves by when every input
    moves by one unit in the last place (close encounters amplify it): the
    roundings of the differences, roots and products ahead of the map.  A
    double-word's are 2^-47, 64 times as large."""
    rng = np.random.default_rng(1)
    _, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    r1, v1 = (np.nextafter(x, x + rng.choice([-1.0, 1.0], x.shape)) for x in (s.r, s.v))
    _, r1, v1 = oracle.step(s.m, r1, v1, s.dt, 2, nthreads=NCPU)
    moved = max(np.max(np.linalg.norm(a - b, axis=1) /
                       np.maximum(np.linalg.norm(b, axis=1), np.sqrt((b ** 2).sum(1).mean())))
                for a, b in ((r1, r), (v1, v)))
    return TOL + 16 * moved * (64 if form == "df64" else 1)


def _tolerance(s, form):
    """TOL, and 16 times what the oracle's result moves by when every input
    moves by one unit in the last place (close encounters amplify it): the
    roundings of the differences, roots and products ahead of the map.  A
    double-word's are 2^-47, 64 times as large."""
    rng = np.random.default_rng(1)
    _, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    r1, v1 = (np.nextafter(x, x + rng.choice([-1.0, 1.0], x.shape)) for x in (s.r, s.v))
    _, r1, v1 = oracle.step(s.m, r1, v1, s.dt, 2, nthreads=NCPU)
    moved = max(np.max(np.linalg.norm(a - b, axis=1) /
                       np.maximum(np.linalg.norm(b, axis=1), np.sqrt((b ** 2).sum(1).mean())))
                for a, b in ((r1, r), (v1, v)))
    return TOL + 16 * moved * (64 if form == "df64" else 1)


@pytest.mark.parametrize("flag", [0, 32, 64], ids=["default", "tiles", "groups"])
@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("n", [49, 160, 331])
def test_partly_strong_tiles_match_the_oracle(n, form, flag):
    for name, clump in CLUMPS.items():
        s = _clumps(n, clump)
        got, _ = _step(s, s.dt, flags=flag, **FORMS[form])
        rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
        assert rc == oracle.OK
        _close(got, (r, v), _tolerance(s, form))


@pytest.mark.parametrize("blocks", [1, 7, 300])
@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_partly_strong_tiles_cut_anywhere(form, blocks):
    s = _clumps(331, CLUMPS["shifted"])
    got, _ = _step(s, s.dt, flags=32, grid_blocks=blocks, **FORMS[form])
    rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    _close(got, (r, v), _tolerance(s, form))


@pytest.mark.parametrize("form", ["fp64", "df64", "literal"])
def test_statistics_count_every_pair_once(form):
    # a solve each of the pairs: at least one evaluation, and all of the run's
    # ordered pairs counted, whichever of the two loops takes them
    s = _clumps(331, CLUMPS["shifted"])
    _, st = _step(s, s.dt, flags=2 | 32, **FORMS[form])
    assert st["pairs"] == 331 * 330 and st["iters"] >= st["solves"]


def _far(n):
    """A cluster at separations out of the short solve's range: its units of
    length and time scaled by 2^32 and 2^48, which changes no bit of a general
    solve's mantissas."""
    s = ics.random_cluster(n, seed=n, mass_spread=3.0)
    return ics.System(s.m, s.r * 2.0 ** 32, s.v * 2.0 ** -16, s.dt * 2.0 ** 48)


@pytest.mark.parametrize("flag", [0, 32, 64], ids=["default", "tiles", "groups"])
@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("n,order,nsteps", [(33, 2, 1), (1301, 2, 1), (1301, 4, 2)])
def test_steps_of_strong_pairs_match_the_oracle(n, order, nsteps, form, flag):
    s, o = _far(n), dict(FORMS[form])
    if form == "literal":
        o["mixed_r_min"] = 1e18
    got, _ = _step(s, s.dt, order, nsteps, flags=flag, **o)
    rc, r, v = oracle.evolve(s.m, s.r, s.v, s.dt, nsteps, order, nthreads=NCPU)
    assert rc == oracle.OK
    _close(got, (r, v), TOL if nsteps == 1 else 12 * TOL)


@pytest.mark.parametrize("flag", [32, 64], ids=["tiles", "groups"])
def test_strong_pairs_take_the_kernels_that_solve_every_pair(flag):
    # statistics keep a run with this guess to those kernels, in the same
    # grid: the same bits; ordinary pairs take the short solve, whose differ
    for s, same in ((_far(1000), True), (ics.random_cluster(1000, seed=1000), False)):
        a, _ = _step(s, s.dt, guess=0, flags=flag, grid_blocks=152)
        b, _ = _step(s, s.dt, guess=0, flags=flag | 2, grid_blocks=152)
        assert all(np.array_equal(x, y) for x, y in zip(a, b)) == same


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("n", [33, 257, 600, 928])
def test_small_kernel_of_every_form(n, form):
    s = ics.random_cluster(n, seed=n, mass_spread=3.0)
    got, _ = _step(s, s.dt, **FORMS[form])
    rc, r, v = oracle.step(s.m, s.r, s.v, s.dt, 2, nthreads=NCPU)
    _close(got, (r, v))


@pytest.mark.parametrize("kind", ["bh", "radial", "bound"])
def test_small_kernel_keeps_the_literal_rules_classes(kind):
    _keeps_the_classes(kind, 0)

"""Compiled plans of common line lengths and the wide radices (6, 9, 10, 12,
15) against the oracle: one ARK4 step with its error norm, each length along
each axis in turn, and explicit orders of the wide radices in the generic
stages of both precisions."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

LENGTHS = [24, 30, 32, 36, 40, 48, 50, 54, 60, 72, 80, 90, 96, 100, 108, 120, 144, 150, 160, 162, 180, 192, 200, 216, 240,
           250, 270, 288, 300, 320, 324, 360, 384, 400, 432, 450, 480, 486, 500, 512, 640]


@pytest.fixture(scope="module")
def pfg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_36100_gb300 as m
    m.build()
    return m


def relerr(a, b):
    return np.array([np.linalg.norm((a[f] - b[f]).ravel()) / np.linalg.norm(b[f].ravel()) for f in range(4)])


def step_case(pfg, p, shape, prec, seed, cfg=None, widths=0):
    y = synth.random_state(shape, seed, phi_scale=0.9)
    m = oracle.Model(shape, p)
    ref, e_ref, _ = oracle.ark_step(m, m.to_k(y), 0.5, oracle.ark436l2sa(), p["rtol"], p["atol"])
    with pfg.Simulation(shape, p, "ark4", prec) as s:
        if cfg:
            c = s.tuning()
            for axis, order in cfg.items():
                c[4 + 11 * axis:4 + 11 * (axis + 1)] = [len(order)] + order + [0] * (10 - len(order))
            s.set_tuning(c)
            assert s.tuning() == c
        else:
            c = s.tuning()
            c[1] = c[37] = widths  # y pass, z passes (0: untuned)
            s.set_tuning(c)  # what a context reports it takes back
        s.set_state(y)
        e = s.step(0.5)
        return relerr(s.state_hat().cpu().numpy(), ref), abs(e - e_ref) / e_ref


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_default_plans_match_oracle(pfg, params, n, axis):
    shape = [12, 10, 6]  # half rows of four columns: every tile ends in the middle of a plane
    shape[2 - axis] = n
    err, e = step_case(pfg, params, tuple(shape), "fp32bulk", 10 + n)
    assert np.all(err <= 1e-5), err
    assert e <= 1e-3


@pytest.mark.parametrize("n", [n for n in LENGTHS if 48 < n <= 384])
@pytest.mark.parametrize("axis", [1, 2])
def test_wide_tiles_match_oracle(pfg, params, n, axis):
    """The column passes at 16 columns a tile, the width the plans of these lengths are compiled for and grids of real
    size run: the small grids of test_default_plans_match_oracle have too few columns for it and run the generic stages.
    24 or 40 columns a field, so the last tile is half empty."""
    assert 2 * 16 * n * 8 <= 128 * 1024  # what the library caps a tuned width by
    shape = (n, 10, 6) if axis == 2 else (6, n, 6)
    err, e = step_case(pfg, params, shape, "fp32bulk", 30 + n, widths=16)
    assert np.all(err <= 1e-5), err
    assert e <= 1e-3


@pytest.mark.parametrize("shape", [(108, 48, 80), (48, 150, 80), (36, 40, 180)])
def test_untuned_wide_tiles_match_oracle(pfg, params, shape):
    """Enough columns (4 fields of 1620 and more) for an untuned tile of 16."""
    err, e = step_case(pfg, params, shape, "fp32bulk", 7)
    assert np.all(err <= 1e-5), err
    assert e <= 1e-3


LONG = [540, 576, 600, 640, 648, 720, 750, 768, 800, 810, 864, 900, 960, 972, 1000, 1024]


@pytest.mark.parametrize("n", LONG)
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("prec,tol,etol", [("fp64", 1e-11, 1e-8), ("fp32bulk", 1e-5, 1e-3)])
def test_long_default_plans_match_oracle(pfg, params, n, axis, prec, tol, etol):
    shape = [6, 10, 6]
    shape[2 - axis] = n
    err, e = step_case(pfg, params, tuple(shape), prec, 50 + n)
    assert np.all(err <= tol), err
    assert e <= etol


@pytest.mark.parametrize("prec,tol,etol", [("fp64", 1e-11, 1e-8), ("fp32bulk", 1e-5, 1e-3)])
@pytest.mark.parametrize("orders", [
    {0: [6, 15], 1: [12], 2: [10, 9]},
    {0: [9, 10], 1: [2, 6], 2: [15, 6]},
    {0: [10, 3, 3], 1: [3, 4], 2: [6, 15]},
])
def test_wide_radices_match_oracle(pfg, params, prec, tol, etol, orders):
    err, e = step_case(pfg, params, (90, 12, 90), prec, 5, orders)
    assert np.all(err <= tol), err
    assert e <= etol


def test_radix_that_is_none_refused(pfg, params):
    with pfg.Simulation((14 * 5 + 10, 12, 10), params, "ark4", "fp64") as s:
        c = s.tuning()
        for bad in ([20, 4], [7, 10], [80], [0, 80], [-8, -10]):
            c[4 + 22:4 + 33] = [len(bad)] + bad + [0] * (10 - len(bad))
            with pytest.raises(pfg.PFError):
                s.set_tuning(c)


@pytest.mark.parametrize("n", [24, 30, 32, 36, 40, 48])
@pytest.mark.parametrize("prec", ["fp64", "fp32bulk"])
def test_short_lines_have_no_wide_radices(pfg, params, n, prec):
    with pfg.Simulation((n, n, n), params, "euler", prec) as s:
        c = s.tuning()
    for axis in range(3):
        count, order = c[4 + 11 * axis], c[5 + 11 * axis:5 + 11 * axis + c[4 + 11 * axis]]
        assert count > 0 and np.prod(order) == n and max(order) <= 8, order


@pytest.mark.parametrize("n", [24, 30, 32, 36, 40, 48, 50, 96, 100, 108, 120, 150, 180, 240])
def test_fp64_default_plans_match_oracle(pfg, params, n):
    """FP64 plans of the fewest instructions, along every axis."""
    for axis in range(3):
        shape = [12, 10, 6]
        shape[2 - axis] = n
        err, e = step_case(pfg, params, tuple(shape), "fp64", 20 + n)
        assert np.all(err <= 1e-11), (axis, err)
        assert e <= 1e-8


@pytest.mark.parametrize("n,limit", [(96, 5.0e-4), (128, 3.27e-4)])
def test_noise_of_the_fp32_error_estimate(pfg, params, n, limit):
    """What FP32 rounding of the right-hand sides adds to the error estimate, per unit of the step: sqrt(e32^2 - e64^2)
    / dt for steps so short that the true estimate is smaller.  The limits are 4 to 5 % above what transforms that
    multiply by the twiddles first (one rounded table entry an input, plain butterflies) give: 4.75e-4 and 3.15e-4."""
    v = []
    for seed in (1, 2, 3):
        y = synth.ic_spheres(n, 4, 3.0, 5.0, seed, params)
        e = []
        for prec in ("fp64", "fp32bulk"):
            with pfg.Simulation((n, n, n), params, "ark4", prec) as s:
                s.set_state(y)
                e.append([s.step(dt) for dt in (0.02, 0.05)])
        v += [np.sqrt(b * b - a * a) / dt for a, b, dt in zip(e[0], e[1], (0.02, 0.05))]
    assert np.mean(v) <= limit, v

"""The FP64 step's fused path (fixed-point right-hand side and circulant solves) at the sizes and
values where it can go wrong: ragged tiles, segments and strips, decays shorter and longer than a
system, |C| from tiny to far above 1, forcing, and what it hands over to the LU path (no implicit
part, stiff operators)."""
import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_ch import _run_gpu, step_tolerance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _both(ny, nx, lx, ly, gamma, dt, steps, scale=1.0, seed=1):
    c0 = scale * synth.field(seed, ny, nx, -0.9, 0.9)
    cm = c0 + dt * scale * synth.field(seed + 1, ny, nx, -1, 1)
    got, gprev = _run_gpu(c0, cm, lx, ly, gamma, dt, steps)
    ref, rprev = oracle.ch_run(c0, cm, lx, ly, gamma, dt, steps)
    return c0, cm, got, gprev, ref, rprev


# (8, 8): the smallest; odd and prime sizes; 33, 65: one past the tiles; 511 / 513: around the strip
# width's rule; 4099: more than one tile of every kind and a row per block
@pytest.mark.parametrize("ny,nx", [(8, 8), (9, 11), (17, 33), (65, 31), (130, 128), (127, 509), (64, 511), (61, 512),
                                   (450, 600), (16, 4099), (2053, 24), (4096, 12)])
@pytest.mark.parametrize("stiff", [1e-3, 3.0, 2e4])
def test_step_matches_the_oracle(ny, nx, stiff):
    dx, gamma, dt = 0.02, 0.01, 1e-4
    lx, ly = nx * dx, ny * dx * (1.0 if nx % 2 else 1.1)  # square and unequal cells
    gamma = stiff * dx**4 / (2 / 3 * dt)
    for steps in (1, 2):
        c0, cm, got, gprev, ref, rprev = _both(ny, nx, lx, ly, gamma, dt, steps)
        tol = step_tolerance(ref, c0, cm, lx, ly, gamma, dt)
        assert np.max(np.abs(got - ref)) <= steps * tol
        assert np.max(np.abs(gprev - rprev)) <= steps * tol


# the cubic's scaling: below, around and above |C| = 1 (a step of the cubic grows with the cube)
@pytest.mark.parametrize("scale", [1e-200, 1e-30, 1e-3, 0.6, 2.3, 40.0, 1e6])
def test_step_over_the_range_of_values(scale):
    n, l, gamma, dt = 96, 2 * np.pi, 0.01, 1e-3
    c0, cm, got, _, ref, _ = _both(n, n, l, l, gamma, dt, 1, scale)
    assert np.max(np.abs(got - ref)) <= step_tolerance(ref, c0, cm, l, l, gamma, dt)


def test_values_of_very_different_size_keep_the_rows_apart():
    """A block of large values in a corner of a small background: errors stay at the rounding of the
    largest value, and a background of exact zeros far from it stays below that."""
    n, l, gamma, dt = 256, 2 * np.pi, 1e-4, 1e-5
    c0 = np.zeros((n, n))
    c0[:20, :20] = synth.field(3, 20, 20, -0.9, 0.9)
    got, _ = _run_gpu(c0, c0, l, l, gamma, dt, 1)
    ref, _ = oracle.ch_run(c0, c0, l, l, gamma, dt, 1)
    assert np.max(np.abs(got - ref)) <= step_tolerance(ref, c0, c0, l, l, gamma, dt)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_stay_non_finite(bad):
    n, l = 70, 2 * np.pi
    c0 = synth.field(3, n, n, -0.9, 0.9)
    c0[31, 32] = bad
    got, gprev = _run_gpu(c0, c0, l, l, 0.01, 1e-3, 1)
    assert np.isnan(got[31, 32]) and np.array_equal(gprev, c0, equal_nan=True)
    assert not np.isfinite(got[31]).any() and not np.isfinite(got[:, 32]).any()


# a = 0 and a above the fused path's limit in one direction or both: the LU solves
@pytest.mark.parametrize("ax,ay", [(0.0, 0.0), (6e4, 6e4), (6e4, 10.0), (10.0, 6e4)])
def test_operators_left_to_the_lu_solves(ax, ay):
    n, dt = 96, 1e-4
    dx = 0.02
    gamma = max(ax, 1e-300) * dx**4 / (2 / 3 * dt) if ax else 0.0
    dy = dx * (ax / ay) ** 0.25 if ax else dx
    c0, cm, got, _, ref, _ = _both(n, n, n * dx, n * dy, gamma, dt, 1)
    assert np.max(np.abs(got - ref)) <= step_tolerance(ref, c0, cm, n * dx, n * dy, gamma, dt)


def test_every_second_row_of_blocks_and_roles():
    """Odd step counts swap the buffers in the end; the kept roles are the caller's."""
    ny, nx, l = 75, 130, 2 * np.pi
    for steps in (3, 5):
        c0, cm, got, gprev, ref, rprev = _both(ny, nx, l, l, 0.01, 1e-3, steps)
        tol = steps * step_tolerance(ref, c0, cm, l, l, 0.01, 1e-3)
        assert np.max(np.abs(got - ref)) <= tol and np.max(np.abs(gprev - rprev)) <= tol

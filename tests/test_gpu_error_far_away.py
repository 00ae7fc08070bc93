"""The Cahn-Hilliard steps in fixed point bound errors by the largest value: far from a block of values
of order one a background of 1e-9 keeps the absolute accuracy that the header states, in every entry."""
import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_ch import _rhs_norm, _run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


# FP32+refine plans of these sizes take the same kernels, so the same bound
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ny,nx", [(256, 256), (203, 330)])
@pytest.mark.parametrize("stiff", [1e-2, 3.0, 300.0])
def test_2d_step(ny, nx, stiff, precision):
    dx, dt = 0.02, 1e-4
    gamma = stiff * dx**4 / (2 / 3 * dt)
    c0 = 1e-9 * synth.field(nx, ny, nx, -1, 1)
    c0[:24, :24] = synth.field(3, 24, 24, -0.9, 0.9)
    got, _ = _run_gpu(c0, c0, nx * dx, ny * dx, gamma, dt, 1, precision)
    ref, _ = oracle.ch_run(c0, c0, nx * dx, ny * dx, gamma, dt, 1)
    err = np.abs(got - ref)
    bound = 4 * EPS * _rhs_norm(c0, c0, nx * dx, ny * dx, gamma, dt)
    assert np.max(err[84:ny - 60, 84:nx - 60]) <= bound
    assert np.max(err) <= bound + 1e-11 * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [256, 411])
@pytest.mark.parametrize("dt", [1e-6, 1e-4, 2e-3])
def test_1d_step(n, dt):
    import paper_2101_06550_gb300 as chx

    batch, l, gamma = 37, 2 * np.pi * n / 256, 0.01
    c0 = 1e-9 * synth.uniform(n, n * batch, -1, 1).reshape(n, batch)
    c0[100:110] = synth.uniform(7, 10 * batch, -0.9, 0.9).reshape(10, batch)
    c = torch.from_numpy(c0.ravel().copy()).cuda()
    chx.Ch1DPlan(n, batch, l, gamma, dt).step(c, 1)
    ref = oracle.ch1d_run(c0.ravel(), l, gamma, dt, 1, batch).reshape(n, batch)
    err = np.abs(c.cpu().numpy().reshape(n, batch) - ref)
    cubic = c0**3 - c0
    lap = np.roll(cubic, 1, 0) + np.roll(cubic, -1, 0) - 2 * cubic
    f = np.max(np.abs(c0 + dt / (l / n) ** 2 * lap), axis=0)
    far = np.r_[0:40, 170:n]
    assert np.all(err[far] <= 64 * EPS * f)
    assert np.all(err <= 64 * EPS * (1 + 16 * gamma * dt / (l / n) ** 4) * f)

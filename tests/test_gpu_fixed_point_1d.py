"""The 1D time steps in fixed point: the unit follows a system's largest value, so values from tiny
to far above 1, systems of very different size side by side, and non-finite ones."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


def _step(c0, n, batch, l, gamma, dt):
    import paper_2101_06550_gb300 as chx

    c = torch.from_numpy(c0.copy()).cuda()
    chx.Ch1DPlan(n, batch, l, gamma, dt).step(c, 1)
    return c.cpu().numpy()


def _tol(c0, n, l, gamma, dt):
    """Rounding of the right-hand side at its largest value, through the solve (64 eps cond as for
    the other solver paths; the smallest eigenvalue is 1)."""
    m, dx = np.max(np.abs(c0)), l / n
    f = m + 4 * dt / dx**2 * m * (1 + m * m)
    return 64 * EPS * (1 + 16 * gamma * dt / dx**4) * f


@pytest.mark.parametrize("n", [8, 9, 15, 33, 64, 257])
@pytest.mark.parametrize("scale", [1e-200, 1e-12, 0.1, 0.9, 2.3, 1e4])
def test_ch1d_over_the_range_of_values(n, scale):
    batch, l, gamma = 35, 2 * np.pi, 0.01
    for dt in (1e-7, 0.1 * l / n):
        c0 = scale * synth.uniform(n, n * batch, -1, 1)
        got = _step(c0, n, batch, l, gamma, dt)
        ref = oracle.ch1d_run(c0, l, gamma, dt, 1, batch)
        assert np.max(np.abs(got - ref)) <= _tol(c0, n, l, gamma, dt)


def test_systems_keep_their_own_units():
    n, batch, l, gamma, dt = 64, 40, 2 * np.pi, 0.01, 1e-3
    sizes = 10.0 ** np.linspace(-30, 2, batch)
    c0 = (synth.uniform(3, n * batch, -1, 1).reshape(n, batch) * sizes).ravel()
    got = _step(c0, n, batch, l, gamma, dt).reshape(n, batch)
    ref = oracle.ch1d_run(c0, l, gamma, dt, 1, batch).reshape(n, batch)
    for s in range(batch):
        assert np.max(np.abs(got[:, s] - ref[:, s])) <= _tol(c0.reshape(n, batch)[:, s], n, l, gamma, dt)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_systems_stay_alone(bad):
    import paper_2101_06550_gb300 as chx

    n, batch = 40, 37
    c0 = synth.uniform(5, n * batch, -0.5, 0.5).reshape(n, batch)
    c0[7, 11] = bad
    got = _step(c0.ravel(), n, batch, 2 * np.pi, 0.01, 1e-3).reshape(n, batch)
    c = torch.from_numpy(c0.ravel().copy()).cuda()
    chx.CN1DPlan(4, n, batch, 1.0, 1.0, 1e-6, False).step(c, 1)
    for out in (got, c.cpu().numpy().reshape(n, batch)):
        assert not np.isfinite(out[:, 11]).any()
        assert np.isfinite(np.delete(out, 11, axis=1)).all()

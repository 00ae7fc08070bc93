"""Linear solves keep the digits of entries that are small next to others of their system: a peak over
a background 1e14 times smaller, and halves of different size.  Every entry is held to its own bound,
K eps |A^-1| |A| |x|, the componentwise backward error of a substitution with two constants (|L| |L^T| =
|A|, the signs of the factors alternate): five roundings per row and sweep with the closure's, as many
again for the coefficients, the scale and the next row's share, K = 32."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps
K = 32


def solve_extended(row, f):
    """Cyclic band solve of the symmetric row in long double: LU with the last unknowns bordered."""
    ld = np.longdouble
    h, n = len(row) // 2, f.shape[0]
    m = n - h
    a = np.zeros((n, n), dtype=ld)
    for o, c in enumerate(row):
        a[np.arange(n), (np.arange(n) + o - h) % n] += ld(c)
    u, x = a, f.astype(ld)
    for r in range(m):  # rows below within the band, and the bordered last rows
        for i in sorted(set(range(r + 1, min(r + h, m - 1) + 1)) | set(range(m, n))):
            q = u[i, r] / u[r, r]
            cols = np.r_[r:min(r + h, n - 1) + 1, max(m, r + h + 1):n]
            u[i, cols] -= q * u[r, cols]
            x[i] -= q * x[r]
    for r in range(m, n):
        for i in range(r + 1, n):
            q = u[i, r] / u[r, r]
            u[i, r:] -= q * u[r, r:]
            x[i] -= q * x[r]
    for r in range(n - 1, -1, -1):
        for j in sorted(set(range(r + 1, min(r + h, n - 1) + 1)) | set(range(max(m, r + 1), n))):
            x[r] -= u[r, j] * x[j]
        x[r] /= u[r, r]
    return x


def entry_bound(row, x):
    """eps (|A^-1| |A| |x|) entry by entry."""
    n, h = x.shape[0], len(row) // 2
    e0 = np.zeros(n)
    e0[0] = 1
    green = np.abs(solve_extended(row, e0)).astype(np.float64)
    inv = green[(np.arange(n)[:, None] - np.arange(n)[None, :]) % n]
    ax = sum(abs(c) * np.roll(np.abs(x).astype(np.float64), h - o, axis=0) for o, c in enumerate(row))
    return EPS * (inv @ ax)


def peak(n, at):
    """A value of order one in row `at`, a background of 1e-14."""
    u = synth.uniform(n + at, 2 * n, 0.5, 1.5).reshape(n, 2)
    f = 1e-14 * u
    f[at] = u[at]
    return f


def cn_row(order, sigma):
    return [sigma, -4 * sigma, 1 + 6 * sigma, -4 * sigma, sigma] if order == 4 else [-sigma, 1 + 2 * sigma, -sigma]


def check_cn(order, sigma, f):
    import paper_2101_06550_gb300 as chx

    n = f.shape[0]
    dt = 2 * sigma * (1.0 / n) ** order  # sigma = dt / (2 dx^order); its roundings are part of K
    x = solve_extended(cn_row(order, sigma), f)
    c = torch.from_numpy(f.ravel().copy()).cuda()
    chx.CN1DPlan(order, n, f.shape[1], 1.0, 1.0, dt).step(c, 1)
    err = np.abs(c.cpu().numpy().reshape(f.shape) - (2 * x - f))
    assert np.all(err <= 2 * K * entry_bound(cn_row(order, sigma), x) + EPS * (2 * np.abs(x) + np.abs(f)))


# the peak far from both ends: the closure of the periodic system stays below its background
@pytest.mark.parametrize("n", [511, 1024])
@pytest.mark.parametrize("sigma", [1e-3, 1.0])
def test_cn_hyperdiffusion(n, sigma):
    check_cn(4, sigma, peak(n, n // 2))


def halves(n, at):
    """Values of order one from row `at` on, 1e-16 of that before it."""
    f = synth.uniform(n + at, 2 * n, 0.5, 1.5).reshape(n, 2)
    f[:at] *= 1e-16
    return f


# large values where the periodic closure carries them to the first rows' background
CLOSED = [(peak, 1.0), (halves, 0.5)]


@pytest.mark.parametrize("n", [9, 65, 511, 1024])
@pytest.mark.parametrize("sigma", [1e-3, 1.0, 50.0, 7e3])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("make,where", CLOSED)
def test_closure_of_cn_steps(order, sigma, n, make, where):
    check_cn(order, sigma, make(n, int(where * n) - (where == 1.0)))


@pytest.mark.parametrize("n", [9, 65, 511, 1024])
@pytest.mark.parametrize("row", [cn_row(o, s) for o in (2, 4) for s in (1e-3, 1.0, 50.0, 7e3)] +
                         [[0.1, 0.3, 1.5, 0.3, 0.1], [0.4, 1.0, 0.4]])
@pytest.mark.parametrize("make,where", CLOSED)
def test_closure_of_uniform_solves(row, n, make, where):
    import paper_2101_06550_gb300 as chx

    f = make(n, int(where * n) - (where == 1.0))
    x = solve_extended(row, f)
    got = torch.from_numpy(f.ravel().copy()).cuda()
    (chx.PentaPlan if len(row) == 5 else chx.TriPlan)(n, row, 2, mode=chx.COEF_UNIFORM).solve(got)
    assert np.all(np.abs(got.cpu().numpy().reshape(f.shape) - x) <= K * entry_bound(row, x))

"""UNIFORM symmetric rows take the circulant factorisation; the same rows given as SHARED take LU
with bordering.  Both against the oracle over sizes around the sweep's blocks of eight rows,
decays from none (identity) to none within the system, definite rows of either sign, and rows the
circulant form declines (indefinite, unsymmetric, too stiff)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps

PENTA = [(0.0, 0.0, 1.0, 0.0, 0.0), (1e-9, -4e-9, 1 + 6e-9, -4e-9, 1e-9), (1.0, -4.0, 7.0, -4.0, 1.0),
         (7e3, -2.8e4, 42001.0, -2.8e4, 7e3), (-2.0, 8.0, -13.0, 8.0, -2.0), (0.1, 0.3, 1.5, 0.3, 0.1),
         (0.0, -5.0, 11.0, -5.0, 0.0), (0.2, 0.1, 2.0, -0.3, 0.1), (1.0, 0.3, -0.25, 0.3, 1.0),
         (1e10, -4e10, 1 + 6e10, -4e10, 1e10)]
TRI = [(0.0, 1.0, 0.0), (-1e-6, 1 + 2e-6, -1e-6), (-5.0, 11.0, -5.0), (-1e5, 200001.0, -1e5), (3.0, -7.0, 3.0),
       (0.4, 1.0, 0.4), (0.2, 1.0, -0.3)]


def _cond(row, n):
    h = len(row) // 2
    k = 2j * np.pi * np.arange(n) / n
    lam = np.abs(sum(c * np.exp(k * (o - h)) for o, c in enumerate(row)))
    return lam.max() / max(lam.min(), 1e-300)


@pytest.mark.parametrize("n", [5, 7, 8, 9, 15, 16, 17, 64, 71, 1000])
@pytest.mark.parametrize("row", PENTA + TRI)
def test_uniform_rows_match_the_general_path(row, n):
    import paper_2101_06550_gb300 as chx

    make, ora = (chx.PentaPlan, oracle.penta_cyclic_batch) if len(row) == 5 else (chx.TriPlan, oracle.tri_cyclic_batch)
    batch = 33
    f = synth.uniform(5 * n + len(row), n * batch, -1, 1)
    cond = _cond(row, n)
    got = {}
    for mode in (chx.COEF_UNIFORM, chx.COEF_SHARED):
        try:
            plan = make(n, row, batch, mode=mode)
        except chx.ChxError as e:
            got[mode] = e.status
            continue
        x = torch.from_numpy(f.copy()).cuda()
        plan.solve(x)
        plan.sync_status()
        got[mode] = x.cpu().numpy()
    a, b = got[chx.COEF_UNIFORM], got[chx.COEF_SHARED]
    if isinstance(b, int):
        assert a == b  # refused by both
        return
    if cond > 1e9:  # no digits to hold either path to; the circulant form declines such rows
        assert np.array_equal(a, b)
        return
    ref = ora(*[np.full(n, c) for c in row], f, batch)
    tol = 64 * EPS * cond * np.max(np.abs(ref))
    assert np.max(np.abs(b - ref)) <= tol
    assert np.max(np.abs(a - ref)) <= tol


@pytest.mark.parametrize("n", [8, 9, 16, 23, 256, 257])
@pytest.mark.parametrize("gamma", [0.0, 0.01])
def test_ch1d_and_cn_closure_lengths(n, gamma):
    """gamma = 0 (identity operator) and closures longer and shorter than the system."""
    import paper_2101_06550_gb300 as chx

    batch, l = 37, 2 * np.pi
    for dt in (1e-6, 0.1 * l / n):
        c0 = synth.uniform(n, n * batch, -0.1, 0.1)
        c = torch.from_numpy(c0.copy()).cuda()
        chx.Ch1DPlan(n, batch, l, gamma, dt).step(c, 2)
        ref = oracle.ch1d_run(c0, l, gamma, dt, 2, batch)
        cond = 1 + 16 * gamma * dt / (l / n) ** 4
        scale = np.max(np.abs(c0)) * (1 + 4 * dt / (l / n) ** 2) ** 2
        assert np.max(np.abs(c.cpu().numpy() - ref)) <= 2 * 64 * EPS * cond * scale


@pytest.mark.parametrize("row", [PENTA[3], PENTA[2], TRI[3], TRI[2]])
def test_large_batches_both_sides_of_the_rule(row):
    """More warps than the rule's limit: a closure of the whole system (LU is chosen) and a short one."""
    import paper_2101_06550_gb300 as chx

    make, ora = (chx.PentaPlan, oracle.penta_cyclic_batch) if len(row) == 5 else (chx.TriPlan, oracle.tri_cyclic_batch)
    n, batch = 203, 24011
    f = synth.uniform(77, n * batch, -1, 1)
    x = torch.from_numpy(f.copy()).cuda()
    make(n, row, batch, mode=chx.COEF_UNIFORM).solve(x)
    pick = np.r_[0:40, batch - 40:batch]
    ref = ora(*[np.full(n, c) for c in row], f.reshape(n, batch)[:, pick].ravel(), pick.size).reshape(n, pick.size)
    err = np.max(np.abs(x.cpu().numpy().reshape(n, batch)[:, pick] - ref))
    assert err <= 64 * EPS * _cond(row, n) * np.max(np.abs(ref))

"""Observables at the edges of the reduction kernels' work units (8 rows x 256 columns of the
field, 8 rows x 32 modes of the half spectrum): single points past a unit, odd and even counts
(Simpson's weights by parity, the unpaired spectral rows 0 and ny/2)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("ny,nx", [(8, 8), (9, 8), (8, 9), (15, 62), (16, 63), (17, 64), (14, 255), (9, 256), (8, 257),
                                   (31, 513), (300, 10)])
def test_observables_at_unit_edges(ny, nx):
    import paper_2101_06550_gb300 as chx

    lx, ly, gamma = 3.0, 2.0, 0.02
    c = synth.field(31 * nx + ny, ny, nx, -0.9, 0.9)
    plan = chx.ChPlan(nx, ny, lx, ly, gamma, 1e-3)
    out = torch.empty(4, dtype=torch.float64, device="cuda")
    diag = torch.empty(2, dtype=torch.float64, device="cuda")
    ct = torch.from_numpy(c).cuda()
    plan.observables(ct, out)
    plan.diagnostics(ct, diag)
    plan.sync_status()
    m, e, s, k1 = oracle.observables(c, lx, ly, gamma)
    n, cell = c.size, lx * ly / c.size
    # a sum of n terms is within n eps of the sum of magnitudes in any order
    for got in (out, diag):
        assert abs(got[0].item() - m) <= n * EPS * np.abs(c).sum() * cell
        assert abs(got[1].item() - e) <= n * EPS * e
    assert out[2].item() == pytest.approx(s, rel=n * EPS)
    assert out[3].item() == pytest.approx(k1, rel=1e-12)

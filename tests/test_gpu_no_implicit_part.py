"""FP32 + refinement without an implicit part (gamma = 0): the reduced systems couple no segment to
another, so only a segment's own block of the inverse is kept."""
import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_ch import _rel, _run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DX, DT = 0.02, 1e-4


# two and three segments, one, 17
@pytest.mark.parametrize("ny,nx", [(64, 48), (96, 96), (33, 47), (40, 1411), (1408, 64)])
def test_plan(ny, nx):
    c0 = synth.field(nx, ny, nx, -0.4, 0.4)
    cm = c0 + DT * synth.field(ny, ny, nx, -1, 1)
    for steps in (1, 2):
        got, _ = _run_gpu(c0, cm, nx * DX, ny * DX, 0.0, DT, steps, precision=1)
        ref, _ = oracle.ch_run(c0, cm, nx * DX, ny * DX, 0.0, DT, steps)
        assert _rel(got, ref) <= steps * 1e-6


@pytest.mark.parametrize("n", [64, 96])
def test_ensemble_group(n):
    import paper_2101_06550_gb300 as chx

    c0 = synth.field(n, n, n, -0.4, 0.4)
    ens = chx.Ensemble(DT, chx.PREC_F32_REFINE)
    gid = ens.group_create(n, n * DX, 0.0, 2)
    for s in range(2):
        ens.load(gid, s, torch.from_numpy(c0).cuda())
    ens.set_active(gid, 2)
    ens.step(3)
    ens.sync_status()
    ref, _ = oracle.ch_run(c0, c0, n * DX, n * DX, 0.0, DT, 3)
    for s in range(2):
        out = torch.empty((n, n), dtype=torch.float64, device="cuda")
        ens.read(gid, s, out)
        assert _rel(out.cpu().numpy(), ref) <= 3e-6

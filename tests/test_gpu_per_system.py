"""PER_SYSTEM solves at the edges of their pipeline: systems shorter than, equal to and one past the
eight rows in flight, rows left over by the factorisation's load blocks, batches of one, a full warp
and one past it; near-singular systems on both sides of the pivot test."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()


@pytest.mark.parametrize("batch", [1, 32, 33])
@pytest.mark.parametrize("n", [5, 6, 7, 8, 9, 10, 11, 12, 17, 18, 19, 26])
@pytest.mark.parametrize("kind", ["penta", "tri"])
def test_per_system_pipeline_edges(kind, n, batch):
    import paper_2101_06550_gb300 as chx

    gen, make, ora = {"penta": (synth.diag_dominant_penta, chx.PentaPlan, oracle.penta_cyclic_batch),
                      "tri": (synth.diag_dominant_tri, chx.TriPlan, oracle.tri_cyclic_batch)}[kind]
    co = gen(100 + n, n, batch)
    f = synth.uniform(200 + n + batch, n * batch, -1, 1)
    ref = ora(*co, f, batch)
    # strictly dominant by 1.5: cond <= 5, and a row's arithmetic is under 16 roundings
    plan = make(n, [_dev(c) for c in co], batch, mode=chx.COEF_PER_SYSTEM)
    x = _dev(f)
    plan.solve(x)
    plan.sync_status()
    assert np.max(np.abs(x.cpu().numpy() - ref)) <= 80 * EPS * np.max(np.abs(ref)) * 4
    p32 = make(n, [_dev(c) for c in co], batch, mode=chx.COEF_PER_SYSTEM, dtype=chx.F32)
    x32 = _dev(f.astype(np.float32))
    p32.solve(x32)
    assert np.max(np.abs(x32.cpu().numpy() - ref)) <= 80 * 2.0 ** -23 * np.max(np.abs(ref)) * 4


@pytest.mark.parametrize("scale", [1e-140, 1.0, 1e140])
@pytest.mark.parametrize("kind", ["penta", "tri"])
def test_per_system_pivot_test_both_sides(kind, scale):
    """A first pivot of 2^-k of the row's largest entry: refused from 1e3 eps of the row sum down, taken above."""
    import paper_2101_06550_gb300 as chx

    n, batch = 12, 3
    for k, refused in ((30, False), (37, False), (41, False), (44, True), (60, True)):
        a = np.zeros((n, batch))
        d, off = np.full((n, batch), 8.0), np.zeros((n, batch))
        # row 0: pivot 2^-k (tri: b_1 enters doubled), neighbour 1; every other row diagonal
        d[0, 1] = 2.0 ** -k / (2.0 if kind == "tri" else 1.0)
        off[0, 1] = 1.0
        co = [a, a, d, off, a] if kind == "penta" else [a, d, off]
        make = chx.PentaPlan if kind == "penta" else chx.TriPlan
        plan = make(n, [_dev(c * scale) for c in co], batch, mode=chx.COEF_PER_SYSTEM)
        if refused:
            with pytest.raises(chx.ChxError) as e:
                plan.sync_status()
            assert e.value.status == -2
        else:
            plan.sync_status()

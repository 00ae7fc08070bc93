"""The double-float right-hand side and the FP32 + refinement solves on rectangles, unequal spacing, odd
sizes, fields off 16-byte boundaries, captured steps and forcing.  Plans of up to 2^20 points and 1400 a
side step in fixed point, so these have a longer side, or an operator that fixed point declines (a' >
5e4 in one direction); the tests see by the bits that the FP64 kernels did not run.
The tolerance is the mode's own, 1e-6 of max|c| per step."""
import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_ch import _rel, _run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DX, DT = 0.02, 1e-4
TOL = 1e-6


def _gamma(stiff):
    return stiff * DX**4 / (2 / 3 * DT)  # a' = stiff along x


def _fields(ny, nx):
    c0 = synth.field(nx, ny, nx, -0.4, 0.4)
    return c0, c0 + DT * synth.field(ny, ny, nx, -1, 1)


def _check(ny, nx, lx, ly, gamma, steps, tol=TOL):
    c0, cm = _fields(ny, nx)
    got, gprev = _run_gpu(c0, cm, lx, ly, gamma, DT, steps, precision=1)
    assert not np.array_equal(got, _run_gpu(c0, cm, lx, ly, gamma, DT, steps)[0])
    ref, rprev = oracle.ch_run(c0, cm, lx, ly, gamma, DT, steps)
    assert _rel(got, ref) <= steps * tol
    assert _rel(gprev, rprev) <= steps * tol
    # the mean follows the scheme's k = 0 mode
    if steps == 1:
        assert abs(got.sum() - (4 * c0.sum() - cm.sum()) / 3) <= tol * np.abs(c0).sum()


# 1411 = 17 x 83, 1503 = 9 x 167, 1409 prime (one segment), 1408: even segments; both directions
@pytest.mark.parametrize("ny,nx", [(40, 1411), (1411, 40), (33, 1503), (1503, 33), (8, 1409), (1409, 9), (96, 1408),
                                   (1408, 130)])
@pytest.mark.parametrize("aspect", [1.0, 1.3])
@pytest.mark.parametrize("stiff", [1.0, 500.0])
def test_rectangles(ny, nx, aspect, stiff):
    for steps in (1, 2):
        _check(ny, nx, nx * DX, ny * DX * aspect, _gamma(stiff), steps)


# smooth fields: a step from a rough one is off by more where the operator is this stiff
@pytest.mark.parametrize("ax,ay", [(6e4, 10.0), (10.0, 6e4), (6e4, 6e4)])
@pytest.mark.parametrize("ny,nx", [(96, 96), (64, 80), (47, 33)])
def test_second_refinement_pass_in_one_direction(ny, nx, ax, ay):
    lx, ly = nx * DX, ny * DX * (ax / ay) ** 0.25
    x, y = 2 * np.pi * np.arange(nx) / nx, 2 * np.pi * np.arange(ny) / ny
    c0 = 0.3 * np.cos(x)[None, :] * np.sin(2 * y)[:, None] + 0.1
    got, _ = _run_gpu(c0, c0, lx, ly, _gamma(ax), DT, 1, precision=1)
    assert not np.array_equal(got, _run_gpu(c0, c0, lx, ly, _gamma(ax), DT, 1)[0])
    ref, _ = oracle.ch_run(c0, c0, lx, ly, _gamma(ax), DT, 1)
    assert _rel(got, ref) <= TOL


@pytest.mark.parametrize("ny,nx", [(64, 1408), (40, 1411)])
def test_same_on_fields_off_16_byte_boundaries(ny, nx):
    """The y solve's two columns per thread give way to one; the arithmetic is the same."""
    import paper_2101_06550_gb300 as chx

    c0, cm = _fields(ny, nx)
    plan = chx.ChPlan(nx, ny, nx * DX, ny * DX * 1.2, _gamma(50.0), DT, chx.PREC_F32_REFINE)
    work, n = plan.alloc_work(), ny * nx
    a, b = torch.from_numpy(c0).cuda(), torch.from_numpy(cm).cuda()
    buf = torch.zeros(2 * n + 2, dtype=torch.float64, device="cuda")  # n is even
    ua, ub = buf[1:1 + n].view(ny, nx), buf[1 + n:1 + 2 * n].view(ny, nx)
    assert ua.data_ptr() % 16 == 8 and ub.data_ptr() % 16 == 8
    ua.copy_(a)
    ub.copy_(b)
    for k in (1, 2, 3):
        plan.step(a, b, work, k)
        plan.step(ua, ub, work, k)
        torch.cuda.synchronize()
        assert torch.equal(a, ua) and torch.equal(b, ub)


def test_captured_steps_match_single_ones():
    import paper_2101_06550_gb300 as chx

    ny, nx = 40, 1411
    c0, cm = _fields(ny, nx)
    plan = chx.ChPlan(nx, ny, nx * DX, ny * DX, _gamma(50.0), DT, chx.PREC_F32_REFINE)
    work = plan.alloc_work()
    for steps in (2, 4, 5):
        a, b = torch.from_numpy(c0).cuda(), torch.from_numpy(cm).cuda()
        plan.step(a, b, work, steps)
        c, d = torch.from_numpy(c0).cuda(), torch.from_numpy(cm).cuda()
        plan.profile(True)  # no graphs
        for _ in range(steps):
            plan.step(c, d, work, 1)
        plan.profile(False)
        plan.profile_read(reset=True)
        torch.cuda.synchronize()
        assert torch.equal(a, c) and torch.equal(b, d), steps


@pytest.mark.parametrize("ny,nx", [(40, 1411), (32, 1408)])
def test_forced_steps(ny, nx):
    """Given deviates, and whole runs that draw them, against the oracle and the FP64 plan."""
    import paper_2101_06550_gb300 as chx

    lx, ly, gamma, sigma = nx * DX, ny * DX * 1.2, _gamma(50.0), 1e-8
    c0, cm = _fields(ny, nx)
    rho = oracle.noise_normals(nx, ny, 4, 2, 0)
    plan = chx.ChPlan(nx, ny, lx, ly, gamma, DT, chx.PREC_F32_REFINE)
    work = plan.alloc_work()
    a, b = torch.from_numpy(c0).cuda(), torch.from_numpy(cm).cuda()
    plan.step_noise(a, b, work, torch.from_numpy(rho.ravel()).cuda(), sigma)
    want, _ = oracle.ch_cook_step(c0, cm, rho, lx, ly, gamma, DT, sigma)
    assert _rel(a.cpu().numpy(), want) <= TOL
    outs = []
    for p in (plan, chx.ChPlan(nx, ny, lx, ly, gamma, DT)):
        a = torch.zeros(ny * nx, dtype=torch.float64, device="cuda")
        b, scratch = torch.zeros_like(a), torch.empty(2 * ny * nx, dtype=torch.float64, device="cuda")
        p.cook_run(a, b, p.alloc_work(), scratch, 5, sigma, seed=3)
        outs.append(a.cpu().numpy())
    assert not np.array_equal(*outs)
    assert _rel(outs[0], outs[1]) <= 5 * TOL


def test_mass_over_a_run():
    ny, nx = 40, 1411
    c0 = synth.field(0, ny, nx, -0.1, 0.1) + 0.02
    got, _ = _run_gpu(c0, c0, nx * DX, ny * DX, _gamma(50.0), DT, 200, precision=1)
    assert abs(got.sum() - c0.sum()) / np.abs(c0).sum() <= 1e-9  # as for the 256^2 run of tests/test_gpu_ch.py

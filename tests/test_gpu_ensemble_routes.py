"""FP64 ensembles whose slots take different solves: fixed point where the operators have circulant
tables, LU for no implicit part (gamma = 0) and for stiff operators (a' > 5e4)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, DT = 64, 1e-3
SIDE = N * 2 * np.pi / 256
DX = SIDE / N
ORDINARY = [0.005, 0.01, 0.02]
STIFF = 6e4 * DX**4 / (2 / 3 * DT)  # a' = 6e4


def _chx():
    import paper_2101_06550_gb300 as chx

    return chx


def _ic(seed):
    """A few long waves: the implicit part of a step is as large as the field, not a' times larger."""
    a, b = 2 * np.pi * synth.uniform(seed, 2, 0, 1)
    x = 2 * np.pi * np.arange(N) / N
    return torch.from_numpy(0.3 * np.cos(x + a)[None, :] * np.cos(2 * x + b)[:, None] + 0.1).cuda()


def _read(ens, gid, slot):
    out = torch.empty((N, N), dtype=torch.float64, device="cuda")
    ens.read(gid, slot, out)
    return out


def _lone(seed, gamma, steps):
    """The simulation as a plan of its own."""
    chx = _chx()
    plan = chx.ChPlan(N, N, SIDE, SIDE, gamma, DT, chx.PREC_F64)
    now = _ic(seed)
    prev = now.clone()
    plan.step(now, prev, plan.alloc_work(), steps)
    torch.cuda.synchronize()
    return now


def _close(a, b):
    # a step's two solves differ by rounding (1e-11, tests/test_gpu_ch.py) and a few steps carry it on
    assert torch.max(torch.abs(a - b)) <= 5e-11 * torch.max(torch.abs(b))


@pytest.mark.parametrize("gamma", [0.0, STIFF])
@pytest.mark.parametrize("steps", [2, 3])
def test_slot_moved_onto_an_active_one_after_capture(gamma, steps):
    """The captured steps belong to the slots' operators: a slot of the other kind moved onto an
    active one takes its own operator along, in pairs of steps (replayed) and single ones alike."""
    ens = _chx().Ensemble(DT, _chx().PREC_F64)
    gid = ens.group_create(N, SIDE, ORDINARY[1], 3)
    for s, g in enumerate([ORDINARY[0], ORDINARY[2], gamma]):
        ens.load(gid, s, _ic(10 + s), None, g)
    ens.set_active(gid, 2)
    ens.step(2)
    ens.move(gid, 2, 1)
    ens.step(steps)
    _close(_read(ens, gid, 0), _lone(10, ORDINARY[0], 2 + steps))
    _close(_read(ens, gid, 1), _lone(12, gamma, steps))
    # and back: an ordinary slot onto the one that LU serves
    ens.load(gid, 2, _ic(20), None, ORDINARY[2])
    ens.step(2)
    ens.move(gid, 2, 1)
    ens.step(steps)
    _close(_read(ens, gid, 0), _lone(10, ORDINARY[0], 4 + 2 * steps))
    _close(_read(ens, gid, 1), _lone(20, ORDINARY[2], steps))
    ens.sync_status()


@pytest.mark.parametrize("n,capacity", [(33, 128), (33, 129), (191, 129), (192, 129)])
def test_both_sides_of_the_rule_for_many_small_fields(n, capacity):
    """Fixed point up to 128 slots or from 192 points a side on, LU beyond."""
    chx = _chx()
    side = n * DX
    x = 2 * np.pi * np.arange(n) / n
    ens = chx.Ensemble(DT, chx.PREC_F64)
    gid = ens.group_create(n, side, 0.01, capacity)
    first = torch.from_numpy(0.3 * np.cos(x)[None, :] * np.sin(2 * x)[:, None] + 0.1).cuda()
    last = first.T.contiguous() - 0.2
    for s in range(capacity):
        ens.load(gid, s, first if s == 0 else last)
    ens.set_active(gid, capacity)
    ens.step(3)
    ens.sync_status()
    plan = chx.ChPlan(n, n, side, side, 0.01, DT, chx.PREC_F64)
    work = plan.alloc_work()
    for slot, c in ((0, first), (capacity - 1, last)):
        now, prev = c.clone(), c.clone()
        plan.step(now, prev, work, 3)
        out = torch.empty((n, n), dtype=torch.float64, device="cuda")
        ens.read(gid, slot, out)
        _close(out, now)


@pytest.mark.parametrize("sigma", [0.0, 1e-8])
@pytest.mark.parametrize("n", [64, 33])  # even: deviates drawn in the step; odd: before it
def test_neighbours_of_the_other_solve_change_no_bit(n, sigma):
    """A simulation alone and beside slots of either kind, in pairs of steps and single ones."""
    chx = _chx()
    x = 2 * np.pi * np.arange(n) / n
    c0 = torch.from_numpy(0.3 * np.cos(x)[None, :] * np.sin(2 * x)[:, None] + 0.1).cuda()

    def run(gammas, slot):
        ens = chx.Ensemble(DT, chx.PREC_F64)
        gid = ens.group_create(n, n * DX, 0.01, 5)
        for s, g in enumerate(gammas):
            ens.load(gid, s, c0, None, g)
        ens.set_active(gid, len(gammas))
        if sigma:
            ens.set_cook(gid, sigma, 7)
        ens.step(5)
        ens.sync_status()
        out = torch.empty((n, n), dtype=torch.float64, device="cuda")
        ens.read(gid, slot, out)
        return out

    # the same slot each time: the forcing goes by the slot
    mixed = [0.0, 0.013, STIFF, 0.02, 0.0]
    for slot in range(4):
        alone = run([0.01] * slot + mixed[slot:slot + 1], slot)
        assert torch.equal(run(mixed, slot), alone), slot
    assert torch.equal(run([STIFF, 0.013], 1), run([0.01, 0.013], 1))


def test_autotune_where_no_step_reads_the_segment_counts():
    """All active slots in fixed point: nothing to time, nothing to allocate (a budget without room for
    a copy of the state), counts and memory as they were.  With an LU slot the counts are chosen."""
    chx = _chx()
    free = chx.Ensemble(DT, chx.PREC_F64)
    free.group_create(N, SIDE, ORDINARY[1], 3)
    used = free.bytes_used
    ens = chx.Ensemble(DT, chx.PREC_F64, hbm_budget=used)
    gid = ens.group_create(N, SIDE, ORDINARY[1], 3)
    for s, g in enumerate([ORDINARY[0], ORDINARY[2], STIFF]):
        ens.load(gid, s, _ic(10 + s), None, g)
    ens.set_active(gid, 2)
    before = ens.info(gid)
    assert ens.autotune(gid, 1) == (before["px"], before["py"])
    assert ens.info(gid) == before and ens.bytes_used == used
    ens.step(3)
    _close(_read(ens, gid, 1), _lone(11, ORDINARY[2], 3))
    ens.set_active(gid, 3)
    with pytest.raises(chx.ChxError) as e:
        ens.autotune(gid, 1)
    assert e.value.status == -4  # the copy of the state is over the budget
    gid = free.group_create(N, SIDE, ORDINARY[1], 1)
    free.load(gid, 0, _ic(12), None, STIFF)
    free.set_active(gid, 1)
    counts = free.autotune(gid, 1)
    assert all(N % c == 0 for c in counts)
    free.step(2)
    _close(_read(free, gid, 0), _lone(12, STIFF, 2))

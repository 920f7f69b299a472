"""Accuracy of the exponential recurrence where its sums are hardest, against the
oracle: many templates (no chunk maps, so that a row run sums its last windows from
zero and sweeps on), tau steps of many SFTs, an outage longer than the windows of
most tau, a glitch behind the windows."""

import numpy as np
import pytest

import oracle
import synth
from synth import EXP, T_SFT, Grid
from tests.parity_util import TOL, check_map

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1805_05652_gb300 as fm  # noqa: E402

UNIQUE = 16


def _run(inst):
    """The map of the instance's templates and its oracle's, computed among 129 copies
    of them (two groups of 32 tau x 2064 templates take no chunk maps)."""
    assert inst.n_templates == UNIQUE and inst.grid.n_tau == 64
    dev = torch.device("cuda:0")
    t, a, x = (torch.from_numpy(v).to(dev) for v in (inst.t, inst.antenna, inst.fafb))
    p = fm.Plan(inst.grid, inst.n_sft, 129 * UNIQUE, "fp64", fm.FMAP_PLAN_EXP_RECURRENCE)
    p.set_refine(0)
    m, _ = p.compute(t, a, x.repeat(129, 1, 1))
    assert p.status() == fm.FMAP_OK
    got = m[-UNIQUE:].cpu().numpy().astype(np.float64)
    assert torch.equal(m[-UNIQUE:], m[:UNIQUE])
    p.close()
    ref, val, _ = oracle.fmap(inst.t, inst.antenna, inst.fafb, inst.grid.as_tuple(), mode="fast")
    return got, ref, val


def test_coarse_tau_steps_start():
    """The last rows of a run start from sums over up to 31 tau steps of 30 SFTs more
    than the shortest window.  With FP32 sums of at most 21 atoms E is off by about
    0.8e-7 rms, 2F of noise (four squares) by 1.4 times that; two roundings of each
    sum's difference give 0.5e-7, the quadratic form and the coefficients 0.4e-7 each:
    together 1.4e-7 of the map's rms, and half as much again is the bound.  (3.4e-7
    where the first sums of a run span up to 2800 atoms.)"""
    grid = Grid(0, T_SFT, 32, 100 * T_SFT, 30 * T_SFT, 64, EXP)
    inst = synth.make_instance(1201, n_det=2, n_slots=9000, n_templates=UNIQUE, grid=grid)
    got, ref, val = _run(inst)
    check_map(got, ref, val, TOL["rec"])
    d, r = (got - ref)[:, 24:, 20:32], ref[:, 24:, 20:32]
    rms = float(np.sqrt((d * d).mean() / (r * r).mean()))
    assert rms <= 2.1e-7, rms


def _outage(days, grid, n_templates=UNIQUE):
    """500 SFTs, an outage, 4000 SFTs."""
    inst = synth.make_instance(1203, n_det=2, n_slots=4500, n_templates=n_templates, grid=grid)
    t = inst.t.copy()
    t[500:] += days * 48 * T_SFT
    return synth.Instance(t, inst.antenna, inst.fafb, grid)


@pytest.mark.parametrize("days,tau_min,dtau,t0_min,dt0", [
    (62, 60, 2, 2900, 5), (73, 400, 10, 2700, 19), (73, 1000, 12, 900, 48), (52, 1000, 12, 400, 40)])
def test_windows_that_start_in_an_outage(days, tau_min, dtau, t0_min, dt0):
    """Windows whose t0 lies in an outage of two months hold the first atoms after
    it: their sum is a small part of what E carries past their end."""
    grid = Grid(t0_min * T_SFT, dt0 * T_SFT, 64, tau_min * T_SFT, dtau * T_SFT, 64, EXP)
    got, ref, val = _run(_outage(days, grid))
    check_map(got, ref, val, TOL["rec"])


def _batch_maps(insts):
    dev = torch.device("cuda:0")
    b = fm.Batch([(i.grid, *(torch.from_numpy(v).to(dev) for v in (i.t, i.antenna, i.fafb)))
                  for i in insts], autotune=False)
    b.run()
    assert b.status() == fm.FMAP_OK
    out = [m.cpu().numpy().astype(np.float64) for m in b.maps]
    b.close()
    return out


@pytest.mark.parametrize("n_templates", [1, 3, 8])
def test_outage_and_glitch_in_a_batch(n_templates):
    """The same in a batch (chunk maps or not), beside an instance with neither."""
    g1 = Grid(900 * T_SFT, 48 * T_SFT, 64, 1000 * T_SFT, 24 * T_SFT, 40, EXP)
    g2 = Grid(0, 3 * T_SFT, 200, 500 * T_SFT, 2 * T_SFT, 33, EXP)
    plain = synth.make_instance(1204, n_det=2, n_slots=3000, n_templates=n_templates, grid=g2)
    glitch = synth.Instance(plain.t, plain.antenna, plain.fafb.copy(), g2)
    glitch.fafb[0, :, 2050] *= np.float32(4e3)
    insts = [_outage(73, g1, n_templates), plain, glitch]
    for inst, got in zip(insts, _batch_maps(insts)):
        ref, val, _ = oracle.fmap(inst.t, inst.antenna, inst.fafb, inst.grid.as_tuple(), mode="fast")
        check_map(got, ref, val, TOL["rec"])


@pytest.mark.parametrize("cut8", [0, 4, 12])
@pytest.mark.parametrize("n_templates,own", [(1, False), (3, True), (6, False)])
def test_glitch_behind_an_outage(n_templates, own, cut8):
    """Windows whose t0 lies in an outage and whose end lies before a glitch, on a coarse
    grid: E at their ends is a thousand times their sums.  Windows of 3 tau and
    shorter ones, plans and batches."""
    n, first = 240, 90
    grid = Grid(0, 40 * T_SFT // 3, 50, 15 * T_SFT, 11 * T_SFT, 60, EXP, T_SFT, cut8)
    inst = synth.make_instance(1206, n_det=2, presence=0.9, n_merged=n, n_templates=n_templates, grid=grid,
                               shared_antenna=not own)
    t, x = inst.t.copy(), inst.fafb.copy()
    t[first:] += 300 * T_SFT
    x[:, :, first + 40] *= np.float32(1e3)
    inst = synth.Instance(t, inst.antenna, x, grid, not own)
    ref, val, _ = oracle.fmap(t, inst.antenna, x, grid.as_tuple(), mode="fast")
    d = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (t, inst.antenna, x)]
    p = fm.Plan(grid, n, n_templates, "fp64",
                fm.FMAP_PLAN_EXP_RECURRENCE | (fm.FMAP_PLAN_PER_TEMPLATE_ANTENNA if own else 0))
    p.set_refine(0)
    m, _ = p.compute(*d)
    assert p.status() == fm.FMAP_OK
    p.close()
    for got in (m.cpu().numpy().astype(np.float64), _batch_maps([inst])[0]):
        check_map(got, ref, val, TOL["rec"])


@pytest.mark.parametrize("n_templates", [1, 2, 7])
def test_care_over_steps_of_many_tau(n_templates):
    """Rows 150 SFTs apart and tau from one SFT: between two rows the decays of a cursor's
    atoms pass below the FP32 range and back."""
    grid = Grid(0, 150 * T_SFT, 12, T_SFT, 3 * T_SFT, 70, EXP)
    inst = synth.make_instance(1207, n_det=2, presence=0.9, n_merged=1900, n_templates=n_templates, grid=grid)
    t, x = inst.t.copy(), inst.fafb.copy()
    t[700:] += 60 * T_SFT
    x[:, :, 300::400] *= np.float32(1e3)
    inst = synth.Instance(t, inst.antenna, x, grid)
    ref, val, _ = oracle.fmap(t, inst.antenna, x, grid.as_tuple(), mode="fast")
    d = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (t, inst.antenna, x)]
    p = fm.Plan(grid, 1900, n_templates, "fp64", fm.FMAP_PLAN_EXP_RECURRENCE)
    p.set_refine(0)
    m, _ = p.compute(*d)
    assert p.status() == fm.FMAP_OK
    p.close()
    for got in (m.cpu().numpy().astype(np.float64), _batch_maps([inst])[0]):
        check_map(got, ref, val, TOL["rec"])


def test_level_of_one_call_is_not_the_next_ones():
    """A call on data with a glitch, and the same plan on data without: the second's map
    is bit for bit that of a plan that never saw the first."""
    grid = Grid(0, 3 * T_SFT, 100, 300 * T_SFT, 2 * T_SFT, 40, EXP)
    inst = synth.make_instance(1205, n_det=2, n_slots=2000, n_templates=5, grid=grid)
    dev = torch.device("cuda:0")
    t, a, x = (torch.from_numpy(v).to(dev) for v in (inst.t, inst.antenna, inst.fafb))
    bad = x.clone()
    bad[:, :, 1100] *= 1e4
    maps = []
    for first in (None, bad):
        p = fm.Plan(grid, inst.n_sft, 5, "fp64", fm.FMAP_PLAN_EXP_RECURRENCE)
        if first is not None:
            p.compute(t, a, first)
        m, _ = p.compute(t, a, x)
        assert p.status() == fm.FMAP_OK
        maps.append(m.cpu().numpy())
        p.close()
    assert np.array_equal(maps[0], maps[1])


def test_glitch_behind_the_windows():
    """One atom 4000 times the noise, up to 1350 SFTs behind the windows' ends: E at
    the window's end carries it through every step between, and the window's own sum
    is what remains of it.  Rounded once every 21 atoms (like E at the window's
    start), E's relative error is about 2^-23 and the cells keep their 1e-5; rounded
    at every step it is 3e-6, some 1e-5 of the window's sum and twice that of 2F."""
    grid = Grid(0, 3 * T_SFT, 500, 960 * T_SFT, 2 * T_SFT, 64, EXP)
    inst = synth.make_instance(1202, n_det=2, n_slots=5000, n_templates=UNIQUE, grid=grid)
    inst.fafb[:, :, 4350] *= np.float32(4e3)
    got, ref, val = _run(inst)
    check_map(got, ref, val, TOL["rec"])

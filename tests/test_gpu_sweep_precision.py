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

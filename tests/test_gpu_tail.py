"""The stages after the cells: compaction of the ill-conditioned entries, their
recomputation for groups of templates, the reductions and the refinement, at the
sizes where their work splits change, against the oracle."""

import numpy as np
import pytest

import oracle
import synth
from synth import EXP, RECT, T_SFT, Grid
from tests.parity_util import TOL, check_map

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1805_05652_gb300 as fm  # noqa: E402


def _run(inst, prec="fp64", flags=0, refine=None):
    dev = torch.device("cuda:0")
    t, a, x = (torch.from_numpy(v).to(dev) for v in (inst.t, inst.antenna, inst.fafb))
    p = fm.Plan(inst.grid, inst.n_sft, inst.n_templates, prec,
                flags | (0 if inst.shared_antenna else fm.FMAP_PLAN_PER_TEMPLATE_ANTENNA))
    if refine is not None:
        p.set_refine(refine)
    m, s = p.compute(t, a, x)
    assert p.status() == fm.FMAP_OK
    out = m.cpu().numpy(), fm.summary_to_numpy(s)
    p.close()
    return out


@pytest.mark.parametrize("shared", [True, False])
@pytest.mark.parametrize("n_templates", [1, 3, 4, 5, 6, 7, 9])
@pytest.mark.parametrize("window", [RECT, EXP])
def test_fixup_template_groups(window, n_templates, shared):
    """One detector's short windows are ill-conditioned: every template of a
    group (four, ragged) gets its own values, refined or not."""
    grid = Grid(-700, T_SFT, 61, 2 * T_SFT if window == RECT else T_SFT, T_SFT, 23, window)
    inst = synth.make_instance(910 + n_templates, n_det=1, presence=0.9, n_merged=70,
                               n_templates=n_templates, grid=grid, shared_antenna=shared,
                               injections=[(n_templates - 1, window, 9 * T_SFT, 12 * T_SFT, 90.0)])
    ref, val, _ = oracle.fmap(inst.t, inst.antenna, inst.fafb, grid.as_tuple(), mode="fast")
    rs = oracle.summary(ref, val)
    prec = "fp64"
    flags = fm.FMAP_PLAN_EXP_RECURRENCE if window == EXP else 0
    for refine in (0, 64):
        m, s = _run(inst, prec, flags, refine)
        check_map(m, ref, val, TOL[prec])
        assert np.array_equal(s["n_valid"], rs["n_valid"])
        np.testing.assert_allclose(s["max2F"], rs["max2F"], rtol=TOL[prec])
        np.testing.assert_allclose(s["logB"], rs["logB"], atol=1e-4)


def test_compaction_long_bitmask():
    """More marked-entry units than one launch compacts (per-template antenna
    rows) and fewer (shared rows) give the same map and summaries."""
    T = 70
    grid = Grid(0, T_SFT, 250, 2 * T_SFT, T_SFT, 250, RECT)
    inst = synth.make_instance(77, n_det=1, presence=0.9, n_merged=260, n_templates=T, grid=grid)
    assert T * grid.n_cells > 128 * 32768 > grid.n_cells
    one_m, one_s = _run(inst)
    own = synth.Instance(inst.t, np.broadcast_to(inst.antenna, (T, *inst.antenna.shape)).copy(),
                         inst.fafb, grid, False)
    own_m, own_s = _run(own)
    np.testing.assert_allclose(own_m, one_m, rtol=1e-6, atol=1e-6)
    for k in ("m", "n", "n_valid"):
        assert np.array_equal(own_s[k], one_s[k])

"""The first launch of a call: input checks, prefix scans and copies of the atoms."""

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
from paper_1805_05652_gb300 import binding as fb  # noqa: E402


@pytest.mark.parametrize("window", [RECT, EXP])
def test_no_templates_no_antenna_rows(window):
    """Antenna rows per template, and no template: there are no rows to check
    (what lies behind the pointer is not the call's)."""
    n = 40
    grid = Grid(0, T_SFT, 5, 2 * T_SFT, T_SFT, 6, window)
    t = torch.arange(n, device="cuda") * T_SFT
    behind = torch.full((3 * n,), float("nan"), device="cuda")
    p = fm.Plan(grid, n, 0, "fp64", fm.FMAP_PLAN_PER_TEMPLATE_ANTENNA)
    out = torch.zeros((1, 32), dtype=torch.uint8, device="cuda")
    a = fb.make_atoms(n, 0, False, t, behind, None)
    call = fb.fmap_compute_rect if window == RECT else fb.fmap_compute_exp
    call(p.handle, a, None, out, None)
    assert p.status() == fm.FMAP_OK
    p.close()


@pytest.mark.parametrize("n", [80, 1200, 9000])
@pytest.mark.parametrize("level", [1e9, 1e12, 1e15])
def test_prefix_sums_before_periodic_outliers(n, level):
    """One outlier in every 32 atoms: the windows before the first of them keep their
    sums, as they do before a single one.  The last atoms of the data alike, behind
    zeros."""
    grid = Grid(0, T_SFT, 20, 2 * T_SFT, T_SFT, 8, RECT)
    head = synth.make_instance(1301, n_det=2, n_slots=n, n_templates=2, grid=grid)
    head.fafb[:, :, 31::32] *= np.float32(level)
    last = (n - 1) // 32 * 32 - 32            # the last whole 32 atoms and the rest
    tail_grid = Grid(last * T_SFT, T_SFT, 20, 2 * T_SFT, T_SFT, 8, RECT)
    tail = synth.make_instance(1302, n_det=2, n_slots=n, n_templates=2, grid=tail_grid)
    tail.fafb[:, :, :last] = 0.0
    tail.fafb[:, :, last + 31:] *= np.float32(level)
    for inst in (head, tail):
        t, a, x = (torch.from_numpy(v).cuda() for v in (inst.t, inst.antenna, inst.fafb))
        p = fm.Plan(inst.grid, n, 2, "fp64")
        p.set_refine(0)
        m, _ = p.compute(t, a, x)
        assert p.status() == fm.FMAP_OK
        p.close()
        ref, val, _ = oracle.fmap(inst.t, inst.antenna, inst.fafb, inst.grid.as_tuple(), mode="direct")
        check_map(m.cpu().numpy().astype(np.float64), ref, val, TOL["fp64"])

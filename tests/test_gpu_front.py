"""The first launch of a call: input checks, prefix scans and copies of the atoms."""

import numpy as np
import pytest

from synth import EXP, RECT, T_SFT, Grid

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

"""Prefix scans and exponential sweeps at the edges of their work splits, against
the oracle: tile boundaries of the scans, ragged template groups, row runs that
start from chunk maps or from zero, SFTs off the T_sft lattice, coarse grids."""

import numpy as np
import pytest

import oracle
import synth
from synth import EXP, RECT, T_SFT, Grid
from tests.parity_util import TOL, check_map, check_summary, run_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


def _check(inst, prec):
    ref, val, _ = oracle.fmap(inst.t, inst.antenna, inst.fafb, inst.grid.as_tuple(), mode="fast")
    got, gs = run_gpu(inst, prec)
    check_map(got, ref, val, TOL[prec])
    # the cells within 16 of the maximum are refined: above 2F = 1e5 the fast
    # path's error bound is wider and the argmax flag is not promised
    if ref.max() < 1e5:
        check_summary(gs, ref, val, TOL[prec])


@pytest.mark.parametrize("n", [2, 31, 63, 64, 65, 257, 1023, 1024, 1025, 2049, 4100])
def test_rect_scan_lengths(n):
    """Data sets around the smallest integer scan (64 atoms) and the scan's tile
    of 1024 atoms; one template far smaller
    than the other, and a row of zeros."""
    grid = Grid(0, max(1, n // 40) * T_SFT, 40, 2 * T_SFT, max(1, n // 50) * T_SFT, 50, RECT)
    inst = synth.make_instance(300 + n, n_det=2, presence=0.9, n_merged=n, n_templates=3, grid=grid)
    inst.fafb[1] *= np.float32(1e-3)
    inst.fafb[2, 3] = 0.0
    _check(inst, "fp64")


@pytest.mark.parametrize("kind,level", [
    ("outlier", 1e4), ("outlier", 1e18), ("step", 1e15), ("all", 1e-19), ("all", 1e14)])
def test_rect_scan_levels(kind, level):
    """Rows whose level changes behind the windows of the grid, and rows of very
    small or large values: the windows keep their sums."""
    grid = Grid(0, 3 * T_SFT, 30, 2 * T_SFT, 2 * T_SFT, 40, RECT)
    inst = synth.make_instance(900, n_det=2, presence=0.9, n_merged=1200, n_templates=2, grid=grid)
    behind = int(np.searchsorted(inst.t, inst.t[0] + 250 * T_SFT))
    assert behind < 700
    part = {"outlier": slice(behind + 100, behind + 101), "step": slice(behind, None),
            "all": slice(None)}[kind]
    inst.fafb[..., part] *= np.float32(level)
    _check(inst, "fp64")


@pytest.mark.parametrize("n_templates", [1, 2, 3, 37, 38, 39, 40])
def test_rec_template_groups(n_templates):
    """63 groups of 32 tau: one, two or four templates per warp, the last
    group ragged."""
    grid = Grid(-900, T_SFT, 7, T_SFT, T_SFT // 2, 2000, EXP)
    _check(synth.make_instance(500 + n_templates, n_det=2, presence=0.9, n_merged=90,
                               n_templates=n_templates, grid=grid), "rec")


@pytest.mark.parametrize("n,n_t0,n_tau,dt0,dtau", [
    (17, 1, 1, 1, 1), (33, 3, 33, T_SFT, T_SFT), (700, 150, 64, T_SFT, T_SFT),
    (1500, 40, 31, 31 * T_SFT, 17 * T_SFT), (2500, 300, 40, 777, 12345)])
@pytest.mark.parametrize("own_rows", [False, True])
def test_rec_row_runs(n, n_t0, n_tau, dt0, dtau, own_rows):
    """Row runs that start from chunk maps, within and past the first tau group,
    on fine and coarse grids, with shared and per-template antenna rows."""
    grid = Grid(-2 * T_SFT, dt0, n_t0, T_SFT, dtau, n_tau, EXP)
    _check(synth.make_instance(700 + n, n_det=2, presence=0.8, n_merged=n, n_templates=3,
                               grid=grid, shared_antenna=not own_rows,
                               injections=[(1, EXP, 5 * T_SFT, 9 * T_SFT, 120.0)]), "rec")


@pytest.mark.parametrize("prec", ["rec", "fp64", "bf16x3"])
@pytest.mark.parametrize("kind", ["jitter", "outage", "mixed"])
def test_exp_off_lattice_times(prec, kind):
    """SFT starts off the T_sft lattice, and gaps longer than the tabulated
    powers of the decay."""
    grid = Grid(0, 2500, 45, 3000, 4100, 70, EXP)
    inst = synth.make_instance(40, n_det=2, presence=0.9, n_merged=400, n_templates=3, grid=grid)
    rng = np.random.default_rng(5)
    t = inst.t.copy()
    if kind != "outage":
        t = t + np.cumsum(rng.integers(0, 700, t.shape[0]) * (rng.random(t.shape[0]) < 0.3))
    if kind != "jitter":
        t[150:] += 40 * T_SFT
        t[260:] += 16 * T_SFT
    _check(synth.Instance(t, inst.antenna, inst.fafb, grid), prec)


@pytest.mark.parametrize("n_t0,n_tau", [(1, 1), (9, 33), (3, 64), (12, 65), (20, 129)])
@pytest.mark.parametrize("n_templates", [1, 2, 5])
def test_rect_wide_rows(n_t0, n_tau, n_templates):
    """Rows that start more atoms apart than a staged group takes, at the edges of
    the cells' tiles, by one, two and four template lanes per tile."""
    grid = Grid(-T_SFT, 4 * T_SFT, n_t0, 2 * T_SFT, T_SFT, n_tau, RECT)
    _check(synth.make_instance(950 + n_tau, n_det=2, presence=0.9, n_merged=500,
                               n_templates=n_templates, grid=grid), "fp64")


@pytest.mark.parametrize("at", [1, 2047, 2300, 4498])
def test_exp_one_irregular_gap(at):
    """One gap off the SFT lattice, in any of the parts the atoms are checked in."""
    grid = Grid(-T_SFT, 60 * T_SFT, 45, 3 * T_SFT, 23 * T_SFT, 40, EXP)
    inst = synth.make_instance(960, n_det=1, presence=0.9, n_merged=4500, n_templates=2, grid=grid)
    t = inst.t.copy()
    t[at:] += 777
    _check(synth.Instance(t, inst.antenna, inst.fafb, grid), "rec")


@pytest.mark.parametrize("n_tau", [1, 32, 33, 64, 65, 257])
def test_table_antenna_columns(n_tau):
    """Window tables at the edges of the antenna sums' 64 columns per warp and 256
    per block, with samples of both signs that end above zero."""
    x = np.linspace(0.0, 1.0, 37)
    table = (np.cos(5.0 * x) * np.exp(-x)).astype(np.float32)
    grid = Grid(-700, 1500, 7, 1200, 900, n_tau, synth.TABLE, T_SFT, 0, None, None, table)
    _check(synth.make_instance(970, n_det=2, presence=0.9, n_merged=300, n_templates=2, grid=grid),
           "fp64")

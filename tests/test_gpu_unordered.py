"""Timestamps that do not increase are reported (FMAP_ERR_DATA), and until the
caller asks for the status every kernel of the call still runs on them: window ends
that are not ordered stay inside every array, and the same plan or batch then
computes the ordered data as if nothing had happened."""

import numpy as np
import pytest

import synth
from synth import EXP, RECT, TABLE, T_SFT, Grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1805_05652_gb300 as fm  # noqa: E402


def _blocks(n, block, seed):
    """Times on the T_SFT lattice, the first in place, the others in blocks of
    `block` atoms in random order."""
    rng = np.random.default_rng(seed)
    t = np.arange(n, dtype=np.int64) * T_SFT
    q = np.arange(1, n) // block
    order = rng.permutation(q.max() + 1)
    t[1:] = t[1:][np.argsort(order[q], kind="stable")]
    return t


def _batch_recovers(inst, bad_t):
    dev = torch.device("cuda:0")
    t = torch.from_numpy(bad_t).to(dev)
    a, x = torch.from_numpy(inst.antenna).to(dev), torch.from_numpy(inst.fafb).to(dev)
    b = fm.Batch([(inst.grid, t, a, x)], autotune=False)
    b.run()
    assert b.status() == fm.FMAP_ERR_DATA
    t.copy_(torch.from_numpy(inst.t))
    b.run()
    assert b.status() == fm.FMAP_OK
    got = b.maps[0].cpu().numpy()
    b.close()
    c = fm.Batch([(inst.grid, t, a, x)], autotune=False)
    c.run()
    assert c.status() == fm.FMAP_OK
    assert np.array_equal(got, c.maps[0].cpu().numpy())
    c.close()


def _plan_recovers(inst, bad_t, prec, flags=0):
    dev = torch.device("cuda:0")
    a, x = torch.from_numpy(inst.antenna).to(dev), torch.from_numpy(inst.fafb).to(dev)
    good, bad = torch.from_numpy(inst.t).to(dev), torch.from_numpy(bad_t).to(dev)
    p = fm.Plan(inst.grid, inst.n_sft, inst.n_templates, prec, flags)
    first, s0 = p.compute(good, a, x)
    assert p.status() == fm.FMAP_OK
    first, s0 = first.cpu().numpy(), s0.cpu().numpy()
    p.compute(bad, a, x)
    assert p.status() == fm.FMAP_ERR_DATA
    again, s1 = p.compute(good, a, x)
    assert p.status() == fm.FMAP_OK
    assert np.array_equal(again.cpu().numpy(), first) and np.array_equal(s1.cpu().numpy(), s0)
    p.close()


def test_index_group_past_the_last_rows_range():
    """A group of t0 rows whose first rows' windows reach further than its last
    row's, with a union of ranges longer than the index step stages (8192)."""
    n = 9000
    grid = Grid(0, 100 * T_SFT, 24, 100 * T_SFT, 600 * T_SFT, 5, EXP)
    inst = synth.make_instance(990, n_slots=n, grid=grid)
    _batch_recovers(inst, _blocks(n, 300, 21))


@pytest.mark.parametrize("n_templates", [1, 2, 4])
@pytest.mark.parametrize("step", [1, 30])
@pytest.mark.parametrize("block", [1, 7, 60, 300])
def test_rect_window_ends_out_of_order(block, step, n_templates):
    """Rectangular cells whose group's window ends lie below its first one, over
    staged prefixes (steps of one SFT) and over global ones (30 SFTs)."""
    grid = Grid(0, step * T_SFT, 40, 2 * T_SFT, 3 * T_SFT, 70, RECT)
    inst = synth.make_instance(991, n_slots=1500, n_templates=n_templates, grid=grid)
    for seed in range(3):
        _plan_recovers(inst, _blocks(1500, block, seed), "fp64")
    _batch_recovers(inst, _blocks(1500, block, 3))


_X = np.linspace(0.0, 1.0, 257)
_TABLE = tuple((np.cos(5.0 * _X) * np.exp(-_X)).astype(np.float32).tolist())


@pytest.mark.parametrize("prec", ["fp64", "fp32", "tf32", "bf16x3"])
@pytest.mark.parametrize("kind", ["swap", 1, 7, 60])
def test_table_times_before_t0(kind, prec):
    """Sampled windows with atoms that start before the window's t0: one swapped
    neighbouring pair, and blocks out of order."""
    grid = Grid(0, T_SFT // 2, 60, 2 * T_SFT, T_SFT, 70, TABLE, T_SFT, 0, None, None, _TABLE)
    inst = synth.make_instance(992, n_slots=300, n_templates=2, grid=grid)
    if kind == "swap":
        bad = inst.t.copy()
        bad[[20, 21]] = bad[[21, 20]]
    else:
        bad = _blocks(300, kind, 5)
    _plan_recovers(inst, bad, prec)


@pytest.mark.parametrize("prec,rec", [("fp64", True), ("fp64", False), ("fp32", False),
                                      ("tf32", False), ("bf16x3", False)])
@pytest.mark.parametrize("block", [1, 60, 300])
def test_exp_times_out_of_order(block, prec, rec):
    grid = Grid(0, 3 * T_SFT, 60, T_SFT, 5 * T_SFT, 70, EXP)
    inst = synth.make_instance(993, n_slots=1200, n_templates=3, grid=grid)
    flags = fm.FMAP_PLAN_EXP_RECURRENCE if rec else 0
    _plan_recovers(inst, _blocks(1200, block, 6), prec, flags)
    if rec:
        _batch_recovers(inst, _blocks(1200, block, 7))

"""Planning a batch on the host: the work splits of any accepted grid are formed
without a fault (in a process of its own, on a machine with a GPU or without)."""

import subprocess
import sys

import pytest

import paper_1805_05652_gb300 as fm
from synth import T_SFT

_CODE = """
import paper_1805_05652_gb300 as fm
from paper_1805_05652_gb300 import binding as fb
fm.lib()
g = fb.make_grid((0, {dt0}, 1, {t_sft}, 0, 1, {t_sft}, fb.FMAP_EXP))
item = fb.fmap_batch_item(g, fb.make_atoms(0, 0, True, None, None, None), None, None)
try:
    fb.fmap_batch_destroy(fb.fmap_batch_plan([item], 0, 0))
except fm.FmapError as e:
    assert e.status in (fm.FMAP_ERR_NOMEM, fm.FMAP_ERR_CUDA), e
"""


@pytest.mark.parametrize("t_sft,dt0", [(T_SFT, 0), (T_SFT, -3 * T_SFT), (T_SFT, -1),
                                       (1, -3), (1, 2**63 - 1), (1, -2**63)])
def test_single_row_any_t0_step(t_sft, dt0):
    """dt0 of a grid with one t0 row is not restricted (nothing uses it)."""
    fm.build()
    r = subprocess.run([sys.executable, "-c", _CODE.format(dt0=dt0, t_sft=t_sft)],
                       capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])

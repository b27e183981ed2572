"""Sets of few tiles run 128-column output tiles (the ragged set and the single
matrices of the other GPU tests among them).  The edges of that rule: the
largest set that takes them, the smallest that does not, and frames whose
last tiles are ragged in 128, each against the oracle and bitwise equal under
both schedules."""
import pytest

import paper_2608_05088_gb300.malt as malt
from paper_2608_05088_gb300 import inputs
from tests.gpu_harness import Run
from tests.test_gpu_schedule import run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [
    ((768, 768),) * 8,                     # 48 symmetric tiles: the most that narrow tiles cover
    ((768, 768),) * 8 + ((8, 8),),         # 49: wide
    ((128, 256), (136, 264), (120, 392), (384, 128), (264, 520)),   # widths around 128 and 256
    ((256, 2120), (2184, 264)),            # grouped form, ragged, wide and tall
])
def test_edges(shapes):
    wl = inputs.Workload("narrow", 70, shapes, "f32", 1.0, 0.02, "malter", 2)
    run_both(wl, 2, schedules=[malt.MALT_NS_PHASED, malt.MALT_NS_PERSISTENT])
    run = Run(wl, check=[0, len(shapes) - 1])
    for s in range(wl.steps):
        run.step()
        assert run.status() == malt.MALT_OK, run.opt.timeout_site()
        for i in run.check:
            run.assert_close(i, f"step {s}")
    run.close()

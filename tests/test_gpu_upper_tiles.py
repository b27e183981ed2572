"""Symmetric products are stored as their upper triangle of 256 x 256 tiles and
read back across the diagonal, transposed.  Frames of one to five tile rows with
ragged last tiles, in wide and in narrow tiles and in both forms of the
iteration, against the oracle and bitwise equal under both schedules."""
import pytest

import paper_2608_05088_gb300.malt as malt
from paper_2608_05088_gb300 import inputs
from tests.gpu_harness import Run
from tests.test_gpu_schedule import run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [
    ((264, 264), (512, 520), (776, 520)),                    # narrow tiles, two and three tile rows
    ((776, 776),) * 9,                                       # wide, 4 tile rows, the last of 8 rows
    ((776, 1560),) * 5 + ((1560, 776),) * 4,                 # the same, grouped form, both orientations
    ((1032, 1096), (1280, 1288)) + ((520, 528),) * 12,       # five tile rows; several classes in one launch
])
def test_tile_rows(shapes):
    wl = inputs.Workload("upper", 71, shapes, "f32", 1.0, 0.02, "malter", 2)
    run_both(wl, 2, schedules=[malt.MALT_NS_PHASED, malt.MALT_NS_PERSISTENT])
    run = Run(wl, check=[0, len(shapes) - 1])
    for s in range(wl.steps):
        run.step()
        assert run.status() == malt.MALT_OK, run.opt.timeout_site()
        for i in run.check:
            run.assert_close(i, f"step {s}")
    run.close()

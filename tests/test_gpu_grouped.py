"""The grouped Newton-Schulz form (3 to 8 iterations of wide frames).

On frames whose rows and columns differ by many decades every row and column of
the direction keeps the accuracy that the iterated bf16 form has on it (a CPU
model of that form's arithmetic).  Each number of iterations, with its own list of
products and work table, matches the oracle, and one state takes them in turn."""
import dataclasses

import numpy as np
import pytest

import paper_2608_05088_gb300.malt as malt
from paper_2608_05088_gb300 import inputs
from tests.bf16_ns_model import newton_schulz_bf16
from tests.gpu_harness import Run
from tests.test_gpu_schedule import run_both
from tests.test_ns_plan import graded_frames, is_grouped

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [4, 5, 8])
def test_small_rows_and_columns(k):
    names, grads = zip(*graded_frames(256, 2048, True, k))
    grads = [g.astype(np.float32) if i % 2 else np.ascontiguousarray(g.T).astype(np.float32)
             for i, g in enumerate(grads)]
    shapes = tuple(g.shape for g in grads)
    wl = inputs.Workload("graded", 80, shapes, "f32", 1.0, 0.02, "muon", 1, ns_steps=k)
    run = Run(wl)
    assert is_grouped(malt.malt_ns_plan(256, 2048, len(shapes), run.hp, muon=True))
    run.step(grads)
    check_slices(run, names, k)
    run.close()


@pytest.mark.parametrize("k", [3, 5, 8])
def test_small_rows_and_columns_preconditioned(k):
    """The same frames as what remains after L M R: gradients whose statistics lie far
    below eps, so that L and R are constant."""
    names, grads = zip(*graded_frames(256, 2048, False, k))
    # (the last one, preconditioned scales, is preconditioned by the step itself)
    grads = [np.ascontiguousarray((g.T if i % 2 else g) * (1.0 if i == len(names) - 1 else 1e-9 / np.abs(g).max()))
             .astype(np.float32) for i, g in enumerate(grads)]
    shapes = tuple(g.shape for g in grads)
    wl = inputs.Workload("graded", 81, shapes, "f32", 1.0, 0.02, "malt", 1, ns_steps=k)
    run = Run(wl)
    assert is_grouped(malt.malt_ns_plan(256, 2048, len(shapes), run.hp))
    run.step(grads)
    check_slices(run, names, k)
    run.close()


def check_slices(run, names, k):
    assert run.status() == malt.MALT_OK, run.opt.timeout_site()
    for i, name in enumerate(names):
        want = run.info[i]["O"]
        new = run.host(run.opt.direction(i)) - want
        old = newton_schulz_bf16(run.info[i]["Mt"], k) - want
        for axis in (0, 1):
            size = np.linalg.norm(want, axis=axis)
            e_new, e_old = (np.linalg.norm(d, axis=axis) / size for d in (new, old))
            # bars of tests/test_ns_plan.py
            assert np.sqrt(np.mean(e_new ** 2)) < 1.1 * np.sqrt(np.mean(e_old ** 2)), (name, axis)
            assert e_new.max() < 2.0 * e_old.max(), (name, axis, e_new.max(), e_old.max())


# grouped (wide and tall, ragged) and iterated frames in one launch; the second set
# in 128-wide tiles
WIDE = ((776, 1560),) * 5 + ((1560, 776),) * 4 + ((520, 520),)
NARROW = ((256, 4096), (2184, 264), (136, 264))


@pytest.mark.parametrize("shapes", [WIDE, NARROW])
@pytest.mark.parametrize("k", [3, 4, 6, 7, 8])
def test_each_number_of_iterations_bitwise(shapes, k):
    wl = inputs.Workload("grouped_k", 82, shapes, "f32", 1.5, 0.02, "malter", 1, ns_steps=k)
    run_both(wl, 1, schedules=[malt.MALT_NS_PHASED, malt.MALT_NS_PERSISTENT])


@pytest.mark.parametrize("variant", ["malter", "muon"])
@pytest.mark.parametrize("schedule", [malt.MALT_NS_PERSISTENT, malt.MALT_NS_PHASED])
@pytest.mark.parametrize("shapes,check", [(WIDE, (0, 8, 9)), (NARROW, (0, 1, 2))])
def test_iterations_change_between_steps(shapes, check, schedule, variant):
    """One state stepped with every grouped number of iterations and two iterated ones
    in turn; every step matches the oracle run with the same sequence."""
    wl = inputs.Workload("grouped_switch", 83, shapes, "f32", 1.0, 0.02, variant, 8)
    run = Run(wl, check=check)
    run.opt.set_ns_schedule(schedule)
    base = run.hp_ref
    for s, k in enumerate((5, 3, 8, 2, 7, 4, 9, 6)):
        run.hp_ref = dataclasses.replace(base, ns_steps=k)
        run.hp = malt.hparams(lr=wl.lr, ns_steps=k)
        run.step()
        assert run.status() == malt.MALT_OK, run.opt.timeout_site()
        for i in check:
            run.assert_close(i, f"step {s} k={k}")
    run.close()

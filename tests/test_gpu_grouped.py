"""The grouped Newton-Schulz form on frames whose rows and columns differ by many
decades: every row and column of the direction keeps the accuracy that the
iterated bf16 form has on it (a CPU model of that form's arithmetic)."""
import numpy as np
import pytest

import paper_2608_05088_gb300.malt as malt
from paper_2608_05088_gb300 import inputs
from tests.bf16_ns_model import newton_schulz_bf16
from tests.gpu_harness import Run
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

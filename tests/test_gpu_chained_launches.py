"""Launches that overlap the one before them read what it wrote, never what the
launch before that did: steps queued back to back, with nothing between them, at
the start of a run, where every step's factors differ from the last one's by far
more than the tolerance."""
import numpy as np
import pytest

import oracle.adamw_ref as aref
import paper_2608_05088_gb300.malt as malt
from paper_2608_05088_gb300 import inputs
from tests.gpu_harness import Run
from tests.test_gpu_whole_optimizer import AdamRun

pytestmark = pytest.mark.gpu


def test_adamw_early_steps():
    """Under a constant gradient every step moves w by lr (m_hat = g, v_hat = g^2).
    With the factors of the step before, step t would move it by
    (1 - b1^t) / (1 - b1^(t-1)) sqrt((1 - b2^(t-1)) / (1 - b2^t)) of that: 1.36 at
    t = 2, 1.0006 at t = 20."""
    run = AdamRun([(5,), (1000,), (70001,)], [0.0, 0.1, 0.0], lr=0.01, seed=75)
    steps = 20
    grads = run.draw()
    for t, g in zip(run.g, grads):
        t.copy_(run.torch.from_numpy(g))
    run.torch.cuda.synchronize()
    for _ in range(steps):
        run.opt.step(run.hp)
    for i, g in enumerate(grads):
        w, wd = run.w0[i].astype(np.float64), float(np.float32(run.wds[i]))
        for _ in range(steps):
            w, _ = aref.adamw_step_ref(w, g.astype(np.float64), run.st_ref[i], run.hp_ref, weight_decay=wd)
        got = run.w[i].double().cpu().numpy()
        # per step 1e-5 of the step and two ulps of w (tests/test_gpu_whole_optimizer.py)
        ulp = np.spacing(np.maximum(np.abs(run.w0[i]), np.abs(got)).astype(np.float32))
        assert np.all(np.abs(got - w) <= steps * (1e-5 * run.lr + 2.0 * ulp)), i
    assert run.opt.get_step() == steps
    run.close()


def test_noalloc_calls_back_to_back():
    """Two matrices in turn through the one scratch array, nothing between the calls:
    bitwise the results of the same calls with the GPU idle before each.  (A finalize
    that read the partial sums of the call before would see the other matrix's.)"""
    import torch
    g = torch.Generator(device="cuda").manual_seed(76)

    def calls(wait):
        out = []
        for m, n, scale in ((392, 1000, 1.0), (1280, 776, 1e3)):
            G = torch.randn(m, n, generator=g, device="cuda").mul_(scale)
            out.append((G, torch.zeros_like(G), *(torch.zeros(s, device="cuda") for s in (m, n, m, n))))
        torch.cuda.synchronize()
        for _ in range(10):
            for a in out:
                assert malt.malt_stats_noalloc(*a) == malt.MALT_OK
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out

    plain = calls(True)
    g.manual_seed(76)
    for a, b in zip(plain, calls(False)):
        assert all(torch.equal(x, y) for x, y in zip(a, b))


def test_refused_launch_is_reported_once():
    """A launch that the runtime refuses (into a stream capture that a synchronize has
    invalidated) fails its own call and no later one."""
    import torch
    run = Run(inputs.Workload("refused", 77, ((128, 256),), "f32", 1.0, 0.02, "malt", 1))
    z = [torch.zeros(s, device="cuda") for s in ((128, 256), (128, 256), (128,), (256,), (128,), (256,))]
    side = torch.cuda.Stream()
    assert malt.malt_stats_noalloc(*z, stream=side) == malt.MALT_OK
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        graph.capture_begin()
        with pytest.raises(RuntimeError):
            side.synchronize()
        rc = malt.malt_stats_noalloc(*z, stream=side)
        with pytest.raises(RuntimeError):
            graph.capture_end()
    torch.cuda.synchronize()
    assert rc == malt.MALT_ERR_CUDA
    assert run.opt.guard_bytes_corrupted() == 0      # checks the last error after its launch
    run.step()
    assert run.status() == malt.MALT_OK
    run.assert_close(0)
    run.close()

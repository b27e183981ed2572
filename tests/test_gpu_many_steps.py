"""Thousands of persistent Newton-Schulz launches of a set whose tile rate the
epilogue and the signals bound (GPT-2 Small, short reductions): no wait may ever
run out.  (Reports of finished tiles that overtook the signalling warp by a whole
round of its barriers were once lost, about once in a thousand steps.)"""
import pytest

import paper_2608_05088_gb300.malt as malt
from paper_2608_05088_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_no_wait_runs_out():
    import torch
    shapes = inputs.WORKLOADS["gpt2_small"].shapes
    params = []
    for a, b in shapes:
        params.append((torch.randn(a, b, device="cuda").mul_(0.02).bfloat16(), torch.randn(a, b, device="cuda"),
                       *(torch.zeros(s, device="cuda") for s in ((a, b), (a,), (b,)))))
    opt = malt.MaltOptimizer(params)
    opt.set_ns_schedule(malt.MALT_NS_PERSISTENT)
    hp = malt.hparams(lr=1e-3)
    for block in range(8):
        for _ in range(750):
            opt.step(hp)
        assert opt.check() == malt.MALT_OK, (block, opt.timeout_site())
    assert opt.guard_bytes_corrupted() == 0
    opt.close()

"""The array that the AdamW binding hands to the library (host only): its fields are
those of one struct written per tensor, for everything the entry points take."""
import ctypes
import math

import numpy as np
import pytest
import torch

import paper_2608_05088_gb300.malt as malt


def entry(n=5, copy=True, g_dtype=torch.float32, wd=0.1, shape=None):
    s = shape or (n,)
    z = lambda dt: torch.zeros(s, dtype=dt)  # noqa: E731
    return (z(torch.float32), z(torch.bfloat16) if copy else None, z(g_dtype), z(torch.float32), z(torch.float32), wd)


def reference(params):
    arr = (malt.malt_adamw_param_t * max(len(params), 1))()
    for i, (w, c, g, m, v, wd) in enumerate(params):
        arr[i] = malt.malt_adamw_param_t(
            w.data_ptr(), None if c is None else c.data_ptr(), g.data_ptr(),
            malt.MALT_BF16 if g.dtype == torch.bfloat16 else malt.MALT_F32, m.data_ptr(), v.data_ptr(), w.numel(),
            float(wd))
    return arr


@pytest.mark.parametrize("wds", [
    (0.0, 0.1, -0.0, 1), (np.float32(0.1), np.float64(0.1), torch.tensor(0.1), True),
    (1e39, -1e39, math.inf, 1e-46), ("0.1", "1e3", 2, 0.5), (math.nan, 0.1, 0.1, 0.1),
])
def test_fields(wds):
    params = [entry(3, True, wd=wds[0]), entry(4097, False, torch.bfloat16, wds[1]),
              entry(copy=True, g_dtype=torch.bfloat16, wd=wds[2], shape=(3, 5)), entry(1, False, wd=wds[3])]
    for p in (params, tuple(params), [list(e) for e in params]):
        got, want = malt.adamw_params_array(p), reference(params)
        assert len(got) == len(want) and bytes(got) == bytes(want)
    assert ctypes.sizeof(malt.malt_adamw_param_t) == 64


def test_empty():
    assert len(malt.adamw_params_array([])) == 1


@pytest.mark.parametrize("bad", [
    lambda e: (e[0][::2],) + e[1:], lambda e: e[:2] + (torch.zeros(6),) + e[3:],
    lambda e: (e[0].double(),) + e[1:], lambda e: (e[0], e[1].float()) + e[2:],
    lambda e: e[:2] + (e[2].half(),) + e[3:], lambda e: e[:5], lambda e: e + (0.1,), lambda e: e[:5] + ("x",),
])
def test_refused(bad):
    with pytest.raises((ValueError, TypeError)):   # (a gradient of another dtype: TypeError)
        malt.adamw_params_array([entry(), bad(entry()), entry()])

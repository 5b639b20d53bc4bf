"""Which path a batch takes, and that what it computes does not depend on
things the caller did not ask for."""

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu


def _device(mats, dtype):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a.T)).to(dtype).cuda().T for a in mats]


def _kernels(gb, mats, dtype):
    import torch
    return [torch.zeros((a.shape[1], min(16, a.shape[1])), dtype=dtype, device="cuda").T for a in mats]


def test_fp32_batch_does_not_depend_on_the_workspace(gb):
    """FP32 results are the persistent kernel's, bit for bit, whatever room the
    workspace has: a pivot that is zero to FP32 rounding has one sign."""
    import torch
    shapes = [(2000, 256), (900, 40), (5003, 128), (700, 129), (301, 100), (64, 16), (400, 200)]
    mats = [workloads.gaussian(m, n, 500 + i) for i, (m, n) in enumerate(shapes)]
    out = []
    with gb.Context(0) as ctx:
        for ws in (None, torch.empty(64 << 20, dtype=torch.uint8, device="cuda")):
            A, T = _device(mats, torch.float32), _kernels(gb, mats, torch.float32)
            ctx.set_workspace(ws)
            ctx.factor_batched(A, T)
            assert ctx.sync()[0] == gb.GBQR_OK
            out.append((A, T))
        ctx.set_workspace(None)
    for (A, B) in zip(*[o[0] for o in out]):
        assert torch.equal(A, B)
    for (A, B) in zip(*[o[1] for o in out]):
        assert torch.equal(A, B)

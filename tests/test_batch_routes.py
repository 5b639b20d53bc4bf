"""Which path a batch takes, and that what it computes does not depend on
things the caller did not ask for."""

import ctypes

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


def _need(gb, shapes):
    I64 = ctypes.c_int64 * len(shapes)
    return gb.gbqr_batched_workspace_bytes(len(shapes), I64(*[s[0] for s in shapes]), I64(*[s[1] for s in shapes]), None)


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


def test_graphs_of_several_shape_sets_on_one_context(gb):
    """A captured batch keeps what it reads: after the context has planned
    other batches it replays to the bits that eager calls gave.  (The
    workspace is the caller's, so that nothing moves it.)"""
    import torch
    sets = [[(2000, 256), (900, 40), (5003, 128)], [(700, 64), (1300, 250), (600, 300), (64, 16)], [(4096, 96), (100, 60)]]
    stream = torch.cuda.Stream()
    with gb.Context(0, stream) as ctx:
        ws = torch.empty(1 << 30, dtype=torch.uint8, device="cuda")
        ctx.set_workspace(ws)
        assert max(_need(gb, s) for s in sets) <= ws.numel()     # (room for the grouped path)
        want, graphs, held = [], [], []
        for k, shapes in enumerate(sets):
            mats = [workloads.gaussian(m, n, 520 + 10 * k + i) for i, (m, n) in enumerate(shapes)]
            A, T = _device(mats, torch.float64), _kernels(gb, mats, torch.float64)
            torch.cuda.synchronize()
            ctx.factor_batched(A, T)
            torch.cuda.synchronize()
            want.append((A, T))
            A, T = _device(mats, torch.float64), _kernels(gb, mats, torch.float64)
            fresh = [a.clone() for a in A]
            torch.cuda.synchronize()
            graphs.append(ctx.capture(lambda: ctx.factor_batched(A, T)))
            held.append((A, T, fresh))
        for k in (0, 2, 1, 0):
            A, T, fresh = held[k]
            for a, t, f in zip(A, T, fresh):
                a.copy_(f)
                t.zero_()
            torch.cuda.synchronize()
            graphs[k].launch()
            torch.cuda.synchronize()
            assert ctx.sync()[0] == gb.GBQR_OK
            for got, exp in zip(A + T, want[k][0] + want[k][1]):
                assert torch.equal(got, exp)
        for g in graphs:
            g.close()
        ctx.set_workspace(None)


def test_panels_given_up_at_every_place(gb):
    """Matrices whose panels fail the condition check at different columns, in
    one batch: whichever CTA finds out first, the results are the same, and
    those of a workspace that only the persistent kernel fits."""
    import torch
    n, mats = 128, []
    for j in range(1, n, 3):
        a = workloads.gaussian(600 + j, n, 560 + j)
        a[:, j] = a[:, j // 2] + 1e-9 * a[:, j]
        mats.append(a)
    with gb.Context(0) as ctx:
        out = []
        for ws in (None, None, None, torch.empty(64 << 20, dtype=torch.uint8, device="cuda")):
            A, T = _device(mats, torch.float64), _kernels(gb, mats, torch.float64)
            if ws is not None:
                ctx.set_workspace(ws)
            ctx.factor_batched(A, T)
            assert ctx.sync()[0] == gb.GBQR_OK
            out.append(A + T)
        ctx.set_workspace(None)
    for other in out[1:]:
        for p, q in zip(out[0], other):
            assert torch.equal(p, q)


@pytest.mark.parametrize("few,many", [((300, 280), (2000, 64)), ((2000, 64), (300, 280))])
def test_ungrouped_matrices_beside_and_before_the_groups(gb, orc, few, many):
    """Few ungrouped matrices run beside the groups, many before them."""
    import torch
    shapes = [few] * 2 + [many] * 90
    mats = [workloads.gaussian(m, n, 580 + i % 5) for i, (m, n) in enumerate(shapes)]
    with gb.Context(0) as ctx:
        out = []
        for ws in (None, torch.empty(64 << 20, dtype=torch.uint8, device="cuda")):
            A, T = _device(mats, torch.float64), _kernels(gb, mats, torch.float64)
            ctx.set_workspace(ws)
            ctx.factor_batched(A, T)
            assert ctx.sync()[0] == gb.GBQR_OK
            out.append((A, T))
        ctx.set_workspace(None)
    for i in (0, 1, 2, 91):
        a = mats[i]
        _gpu.compare_factor(a, gb.to_numpy(out[0][0][i]), gb.to_numpy(out[0][1][i]), gb.GBQR_T_PANEL, 16, orc, f"{a.shape}")
        if a.shape[0] == 300:       # the persistent kernel's, in either place
            assert torch.equal(out[0][0][i], out[1][0][i]) and torch.equal(out[0][1][i], out[1][1][i])

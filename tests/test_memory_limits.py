"""Calls that fit without the scratch of the digit products and groups run
where that scratch does not fit: little free memory on the GPU, or matrices
whose digits alone would fill it."""

import ctypes

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu


class _Held:
    """All free memory of the GPU but `leave` bytes."""

    def __init__(self, leave):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.t = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        import torch
        del self.t
        torch.cuda.empty_cache()


def _plain(gb, m, n):
    return gb.workspace_bytes(m, n, gb.GBQR_T_PANEL, gb.opts(fp64_gemm=gb.GBQR_GEMM_DMMA))


def test_factor_without_room_for_digits(gb):
    import torch
    m, n = 2_000_000, 64
    with gb.Context(0) as roomy:
        a = torch.empty((n, m), dtype=torch.float64, device="cuda").normal_(generator=torch.Generator("cuda").manual_seed(1))
        A, B = a.clone().T, a.T
        T, U = gb.colmajor(n, n, fill=0.0), gb.colmajor(n, n, fill=0.0)
        roomy.factor(A, T, gb.GBQR_T_PANEL)
        assert roomy.sync()[0] == gb.GBQR_OK
    leave = _plain(gb, m, n) + (1 << 30)
    assert leave < gb.workspace_bytes(m, n)
    with gb.Context(0) as ctx, _Held(leave):
        ctx.factor(B, U, gb.GBQR_T_PANEL)
        assert ctx.sync()[0] == gb.GBQR_OK
    s = float(np.sqrt(m))
    assert float((torch.tril(A, -1) - torch.tril(B, -1)).abs().max()) <= 1e-11
    assert float((torch.triu(A[:n]) - torch.triu(B[:n])).abs().max()) <= 1e-11 * s
    assert float((T - U).abs().max()) <= 1e-11


def test_batch_without_room_for_groups(gb):
    import torch
    mats = [workloads.gaussian(4000, 128, 900 + i % 4) for i in range(200)]
    dev = lambda: [torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T for a in mats]
    out = []
    with gb.Context(0) as ctx:
        I64 = ctypes.c_int64 * 200
        assert gb.gbqr_batched_workspace_bytes(200, I64(*[4000] * 200), I64(*[128] * 200), None) > 1 << 30
        ctx.set_workspace(torch.empty(64 << 20, dtype=torch.uint8, device="cuda"))
        A, T = dev(), [gb.colmajor(16, 128, fill=0.0) for _ in mats]
        ctx.factor_batched(A, T)
        assert ctx.sync()[0] == gb.GBQR_OK
        out.append(A + T)
        ctx.set_workspace(None)
        A, T = dev(), [gb.colmajor(16, 128, fill=0.0) for _ in mats]
        with _Held(1 << 30):
            ctx.factor_batched(A, T)
            assert ctx.sync()[0] == gb.GBQR_OK
        out.append(A + T)
    for p, q in zip(*out):
        assert torch.equal(p, q)


def test_groups_hold_their_matrices(gb):
    """A matrix whose digits alone exceed a group's scratch (36 GB here) is not
    grouped: it asks for what one of 15 columns does, which never is."""
    I64 = ctypes.c_int64 * 2
    need = [gb.gbqr_batched_workspace_bytes(2, I64(20_000_000, 2000), I64(n, 64), None) for n in (16, 15)]
    assert need[0] <= need[1] + (1 << 30)


def test_more_rows_than_one_sum_splits(gb):
    """2^25 rows, more than a digit product sums in 65535 splits: the TSQR."""
    import torch
    m, n = 1 << 25, 16
    a = torch.empty((n, m), dtype=torch.float64, device="cuda").normal_(generator=torch.Generator("cuda").manual_seed(3))
    G = a @ a.T
    T = gb.colmajor(n, n, fill=0.0)
    with gb.Context(0) as ctx:
        ctx.factor(a.T, T, gb.GBQR_T_PANEL)
        assert ctx.sync()[0] == gb.GBQR_OK
    R = torch.triu(a.T[:n])
    assert float((R.T @ R - G).norm() / G.norm()) <= 1e-13


def test_digits_leave_room(gb):
    """The digits' share of the workspace is bounded, whatever the rows."""
    for m, n in [(100_000_000, 16), (20_000_000, 256)]:
        assert gb.workspace_bytes(m, n) - _plain(gb, m, n) <= 64 << 30


def test_server_cap_without_room_for_digits(gb, orc):
    """A cap that holds a request only without the digit products admits it."""
    import torch
    m, n = 20000, 300
    a, _, b = workloads.ls_problem(m, n, 2.0, 910)
    A, bd, x = _gpu.device_matrix(a), torch.from_numpy(b).cuda(), torch.zeros(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    cap = _plain(gb, m, n) + (1 << 20) + 8 * (m * n + m + n)
    assert cap < gb.workspace_bytes(m, n)
    with gb.Context(0) as ctx:
        ctx.serve(2, cap)
        r = ctx.poll(ctx.submit(A, bd, x, gb.GBQR_FP64), wait=True)
        with pytest.raises(gb.GbqrError):
            ctx.submit(_gpu.device_matrix(workloads.gaussian(m, n + 8, 911)), bd,
                       torch.zeros(n + 8, dtype=torch.float64, device="cuda"), gb.GBQR_FP64)
        ctx.stop_serving()
    assert r.status == gb.GBQR_OK and r.footprint_bytes == cap
    x_o, _ = orc.ls_solve(a, b)
    assert np.linalg.norm(x.cpu().numpy() - x_o) <= 1e-11 * np.linalg.norm(x_o)

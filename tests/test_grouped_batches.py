"""Batches factored group by group from their Gram matrices: shapes at the
edges of what the grouped path takes, matrices that it hands to the persistent
kernel midway, and a workspace that only the persistent kernel fits."""

import ctypes

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu

# around 4 rows a column of the first and of a later panel, around the 128
# column panel and its narrower splits, 16-wide T blocks that end ragged
EDGES = [(63, 16), (64, 16), (68, 17), (511, 128), (512, 128), (520, 129), (700, 129), (768, 256), (639, 255),
         (1200, 250), (301, 100), (40, 30), (2000, 1), (4097, 33)]


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


def _need(gb, shapes):
    I64 = ctypes.c_int64 * len(shapes)
    return gb.gbqr_batched_workspace_bytes(len(shapes), I64(*[s[0] for s in shapes]), I64(*[s[1] for s in shapes]), None)


def _run(gb, ctx, mats, dtype=np.float64, workspace=None):
    import torch
    tt = torch.float64 if dtype == np.float64 else torch.float32
    As, Ts = [], []
    for i, a in enumerate(mats):
        m, n = a.shape
        buf = torch.full((n, m + i % 3), float("nan"), dtype=tt, device="cuda")     # odd leading dimensions too
        buf[:, :m] = torch.from_numpy(np.ascontiguousarray(a.T).astype(dtype)).cuda()
        As.append(buf.T[:m])
        Ts.append(torch.full((n, 16), float("nan"), dtype=tt, device="cuda").T)
    ctx.set_workspace(workspace)
    ctx.factor_batched(As, Ts)
    torch.cuda.synchronize()
    st, _ = ctx.sync()
    ctx.set_workspace(None)
    return st, [A.cpu().numpy().astype(np.float64) for A in As], [T.cpu().numpy().astype(np.float64) for T in Ts]


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_shapes_at_the_edges(gb, ctx, orc, dtype):
    mats = [workloads.gaussian(m, n, 300 + i).astype(dtype) for i, (m, n) in enumerate(EDGES)]
    st, VR, T = _run(gb, ctx, mats, dtype)
    assert st == gb.GBQR_OK
    for a, vr, t in zip(mats, VR, T):
        nb = min(_gpu.BATCH_B, a.shape[1])
        _gpu.compare_factor(a, vr, t[:nb], gb.GBQR_T_PANEL, nb, orc, f"{a.shape}", fp32=dtype == np.float32)


def _parallel(a, j, k):
    """Column j nearly column k: the panel that holds both is ill-conditioned,
    and so is every trailing block that holds both."""
    a[:, j] = a[:, k] + 1e-9 * a[:, j]
    return a


def test_ill_conditioned_panels_go_to_the_persistent_kernel(gb, ctx):
    import torch
    shapes = [(2000, 256), (2000, 256), (1500, 256), (900, 40)]
    mats = [workloads.gaussian(m, n, 330 + i) for i, (m, n) in enumerate(shapes)]
    _parallel(mats[0], 100, 3)                  # the first panel
    _parallel(mats[1], 255, 130)                # the second
    st, VR, T = _run(gb, ctx, mats)
    assert st == gb.GBQR_OK
    # a workspace one block short of the grouped path's: the persistent kernel alone
    need = _need(gb, shapes)
    st2, VR2, T2 = _run(gb, ctx, mats, workspace=torch.empty(need - 256, dtype=torch.uint8, device="cuda"))
    assert st2 == gb.GBQR_OK
    assert np.array_equal(VR[0], VR2[0]) and np.array_equal(T[0], T2[0])
    assert not np.array_equal(VR[2], VR2[2])    # (the grouped path did run)
    for a, vr, t in list(zip(mats, VR, T)) + list(zip(mats, VR2, T2)):
        n = a.shape[1]
        Q = _gpu.q_from_panels(vr, t, _gpu.BATCH_B)
        assert np.linalg.norm(a - Q @ np.triu(vr[:n])) <= _gpu.TOL_BACKWARD * np.linalg.norm(a)
        assert np.linalg.norm(Q.T @ Q - np.eye(n), 2) <= _gpu.TOL_BACKWARD


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("col", [5, 200])
def test_nonfinite_matrices_stay_apart(gb, ctx, col, value):
    mats = [workloads.gaussian(m, n, 350 + i) for i, (m, n) in enumerate([(1300, 250), (1300, 250), (600, 64)])]
    st, VR, T = _run(gb, ctx, mats)
    assert st == gb.GBQR_OK
    mats[1][700, col] = value
    st, VR2, T2 = _run(gb, ctx, mats)
    assert st == gb.GBQR_ENONFINITE
    for i in (0, 2):
        assert np.array_equal(VR[i], VR2[i]) and np.array_equal(T[i], T2[i])


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_sums_of_the_largest_digits(gb, ctx, dtype):
    """Tall matrices whose columns have one sign and nearly one magnitude, just
    below a power of two: the digit products' integer sums at their largest."""
    mats = []
    for i, (m, n) in enumerate([(45001, 33), (21000, 20), (66000, 130)]):
        a = workloads.gaussian(m, n, 370 + i)
        a[:, 0] = 0.9999                        # (the other columns keep it well-conditioned)
        mats.append(a.astype(dtype))
    st, VR, T = _run(gb, ctx, mats, dtype)
    assert st == gb.GBQR_OK
    tol = _gpu.TOL_BACKWARD if dtype == np.float64 else _gpu.TOL32_BACKWARD
    for a, vr, t in zip(mats, VR, T):
        n = a.shape[1]
        a = a.astype(np.float64)
        Q = _gpu.q_from_panels(vr, t, _gpu.BATCH_B)
        assert np.linalg.norm(a - Q @ np.triu(vr[:n])) <= tol * np.linalg.norm(a)
        assert np.linalg.norm(Q.T @ Q - np.eye(n), 2) <= tol

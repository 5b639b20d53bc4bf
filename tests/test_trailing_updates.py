"""The fused trailing update (W = Y^T C, C -= V W from digits cut once) in both
types, at the edges of its 128 x 64 tiles, of its panels and of the row count
it starts at, against the oracle."""

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


# one column behind the panel; a ragged last panel; the least number of rows
# and one row less; tile remainders of 1 and 63; n > m / 4 (its last panels
# are a TSQR's); panels narrower than 128
SHAPES = [(700, 129, 128), (1300, 300, 128), (256, 192, 64), (255, 192, 64), (641, 257, 128), (1023, 383, 128),
          (400, 400, 128), (900, 200, 48)]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("m,n,nb", SHAPES)
def test_panel_layout_matches_oracle(gb, ctx, orc, m, n, nb, dtype):
    import torch
    f32 = dtype == "f32"
    tt = torch.float32 if f32 else torch.float64
    a = workloads.graded(m, n, 400 + n, 2.0)
    if f32:
        a = a.astype(np.float32)
    buf = torch.full((n, m + 5), float("nan"), dtype=tt, device="cuda")
    buf[:, :m] = torch.from_numpy(np.ascontiguousarray(a.T)).cuda()
    A, T = buf.T[:m], torch.full((n, nb), float("nan"), dtype=tt, device="cuda").T
    assert ctx.factor(A, T, gb.GBQR_T_PANEL, gb.opts(panel_nb=nb)) == gb.GBQR_OK
    torch.cuda.synchronize()
    assert ctx.sync()[0] == gb.GBQR_OK
    if m == n:      # the last columns' V is as ill-conditioned as the matrix
        Q = _gpu.q_from_panels(A.cpu().numpy(), T.cpu().numpy(), nb)
        tol = _gpu.TOL32_BACKWARD if f32 else _gpu.TOL_BACKWARD
        a = np.asarray(a, dtype=np.float64)
        assert np.linalg.norm(a - Q @ np.triu(A.cpu().numpy()[:n])) <= tol * np.linalg.norm(a)
        assert np.linalg.norm(Q.T @ Q - np.eye(n), 2) <= tol
    else:
        _gpu.compare_factor(a, A.cpu().numpy(), T.cpu().numpy(), gb.GBQR_T_PANEL, nb, orc, f"{m}x{n}", fp32=f32)
    assert bool(torch.isnan(buf[:, m:]).all())      # the padding stays


@pytest.mark.parametrize("m,n,nb", [(20000, 512, 256), (9001, 450, 200)])
def test_wide_panels_merge_t(gb, ctx, orc, m, n, nb):
    """Panels of two Gram-matrix halves: the T merge's product with the second
    half's unit lower trapezoid, in column chunks where the scratch of the
    look-ahead lane holds no more."""
    a = workloads.gaussian(m, n, 430 + nb)
    VR, T, _ = _gpu.factor_gpu(ctx, a, gb.GBQR_T_PANEL, gb.opts(panel_nb=nb))
    _gpu.compare_factor(a, VR, T, gb.GBQR_T_PANEL, nb, orc, f"{m}x{n} nb {nb}")
    # and with the full T, whose merge products are the widest
    VR, T, nb = _gpu.factor_gpu(ctx, a, gb.GBQR_T_FULL)
    _gpu.compare_factor(a, VR, T, gb.GBQR_T_FULL, nb, orc, f"{m}x{n} full")

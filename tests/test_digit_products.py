"""Large FP64 products by exact digit splitting on the tensor cores: applying
Q through them against the oracle's reflector-by-reflector application, at
tile edges, remainders and extreme column scales."""

import numpy as np
import pytest

import workloads
from tests import _gpu

pytestmark = pytest.mark.gpu

U = np.finfo(float).eps / 2


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


def _problem(gb, ctx, m, n, layout, seed):
    a = workloads.graded(m, n, seed, 2.0)
    VR, T, nb = _gpu.factor_gpu(ctx, a, layout)
    return a, VR, T, nb


# rows, reflectors and columns around the 128 x 64 tile and the 32-, 256- and
# 512-wide steps in K, and products split over K and not
SHAPES = [(1025, 130, 65, "panel"), (512, 128, 256, "panel"), (4099, 127, 63, "panel"), (2047, 257, 129, "full"),
          (1500, 700, 300, "full"), (33000, 33, 64, "panel")]


@pytest.mark.parametrize("m,n,nrhs,layout_name", SHAPES)
def test_apply_matches_oracle(gb, ctx, orc, m, n, nrhs, layout_name):
    layout = gb.GBQR_T_FULL if layout_name == "full" else gb.GBQR_T_PANEL
    a, VR, T, nb = _problem(gb, ctx, m, n, layout, 40 + n)
    b = workloads.gaussian(m, nrhs, 41)
    b *= (10.0 ** np.linspace(-290, 290, nrhs))[None, :]     # columns are scaled independently
    b[:, nrhs // 2] = 0.0
    B = gb.to_colmajor(b)
    ctx.apply_qt(gb.to_colmajor(VR), gb.to_colmajor(T), B, layout, nb)
    got = gb.to_numpy(B)
    vr_o, tau_o = orc.house_qr(a)
    s = np.maximum(np.abs(b).max(axis=0), np.finfo(float).tiny)
    want = np.column_stack([orc.apply_qt(vr_o, tau_o, np.ascontiguousarray(b[:, j] / s[j])) for j in range(nrhs)])
    err = np.linalg.norm(got / s - want, axis=0) / np.maximum(np.linalg.norm(b / s, axis=0), 1e-300)
    # n reflections on either side, each within a few u of the column's norm
    assert err.max() <= 6 * n * U, err.max()
    assert not got[:, nrhs // 2].any()


def test_nonfinite_columns_stay_apart(gb, ctx):
    layout = gb.GBQR_T_PANEL
    _, VR, T, nb = _problem(gb, ctx, 2000, 128, layout, 50)
    b = workloads.gaussian(2000, 200, 51)
    bad = b.copy()
    bad[1999, 3] = np.nan
    bad[0, 70] = np.inf
    out = []
    for x in (b, bad):
        B = gb.to_colmajor(x)
        ctx.apply_qt(gb.to_colmajor(VR), gb.to_colmajor(T), B, layout, nb)
        out.append(gb.to_numpy(B))
    keep = [j for j in range(200) if j not in (3, 70)]
    assert np.array_equal(out[0][:, keep], out[1][:, keep])
    assert np.isnan(out[1][:, 3]).all() and not np.isfinite(out[1][:, 70]).any()


def test_workspace_without_room_for_digits(gb, orc):
    """A caller's workspace of the FMA engines' size still serves the call."""
    import torch
    a = workloads.gaussian(1500, 900, 52)
    with gb.Context(0) as c:
        nbytes = gb.workspace_bytes(1500, 900, gb.GBQR_T_PANEL, gb.opts(fp64_gemm=gb.GBQR_GEMM_DMMA))
        assert nbytes < gb.workspace_bytes(1500, 900)
        c.set_workspace(torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
        VR, T, nb = _gpu.factor_gpu(c, a, gb.GBQR_T_PANEL)
        _gpu.compare_factor(a, VR, T, gb.GBQR_T_PANEL, nb, orc, "small workspace")
        c.set_workspace(None)

"""Panels that the Gram-matrix base case gives up (odd columns close to the even
ones: each column's part apart from the others is 3 % of its length): the
recursion on TSQRs in one launch, against the oracle, from the narrowest panel
to the widest, at one leaf and at several merge levels, with Y = V T for the
fused update, and twice (its counters are left zero)."""

import numpy as np
import pytest

import workloads
from tests import _gpu
from tests.test_parity_factor import _near_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gb):
    with gb.Context(0) as c:
        yield c


@pytest.mark.parametrize("m,n,layout_name,nb", [
    (64, 16, "full", 0), (68, 17, "full", 0), (101, 25, "full", 0), (133, 33, "full", 0), (512, 128, "full", 0),
    (4099, 127, "full", 0), (20001, 48, "full", 0), (33001, 96, "full", 0), (70001, 20, "panel", 0),
    (3000, 300, "panel", 128), (1300, 290, "panel", 96), (900, 200, "panel", 48), (2000, 257, "full", 0)])
def test_given_up_panels_match_oracle(gb, ctx, orc, m, n, layout_name, nb):
    layout = gb.GBQR_T_FULL if layout_name == "full" else gb.GBQR_T_PANEL
    a = _near_pairs(m, n, 700 + n, 3e-2)
    o = gb.opts(panel_nb=nb) if nb else None
    VR, T, nbr = _gpu.factor_gpu(ctx, a, layout, o, lda_pad=n % 3)
    _gpu.compare_factor(a, VR, T, layout, nbr, orc, f"{m}x{n}")
    VR2, T2, _ = _gpu.factor_gpu(ctx, a, layout, o, lda_pad=n % 3)
    assert np.array_equal(VR, VR2) and np.array_equal(T, T2)


@pytest.mark.parametrize("m,n,nb", [(2000, 40, 40), (3000, 300, 128), (512, 128, 128)])
def test_given_up_panels_fp32(gb, ctx, orc, m, n, nb):
    import torch
    a = _near_pairs(m, n, 730 + n, 3e-2).astype(np.float32)
    A = torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T
    T = torch.full((n, nb), float("nan"), dtype=torch.float32, device="cuda").T
    ctx.factor(A, T, gb.GBQR_T_PANEL, gb.opts(panel_nb=nb))
    torch.cuda.synchronize()
    _gpu.compare_factor(a.astype(np.float64), A.cpu().numpy(), T.cpu().numpy(), gb.GBQR_T_PANEL, nb, orc, f"fp32 {m}x{n}", fp32=True)


def test_mixed_least_squares_with_given_up_panels(gb, ctx, orc):
    import torch
    a = _near_pairs(4000, 320, 740, 3e-2)
    x = np.random.default_rng(741).standard_normal(320)
    b = a @ x
    xd = torch.zeros(320, dtype=torch.float64, device="cuda")
    st, _ = ctx.ls_solve(_gpu.device_matrix(a), torch.from_numpy(b).cuda(), xd, gb.GBQR_MIXED_SPLITBF16)
    assert st == gb.GBQR_OK
    # columns' condition about 1 / 3e-2, times the square for a residual near zero
    assert np.linalg.norm(xd.cpu().numpy() - x) <= 1e-11 * np.linalg.norm(x)


def test_given_up_panels_in_a_graph(gb):
    import torch
    a = _near_pairs(3000, 300, 750, 3e-2)
    stream = torch.cuda.Stream()
    with gb.Context(0, stream) as ctx:
        A, T = _gpu.device_matrix(a), gb.colmajor(128, 300, fill=0.0)
        torch.cuda.synchronize()
        ctx.factor(A, T, gb.GBQR_T_PANEL)
        torch.cuda.synchronize()
        B, U, fresh = _gpu.device_matrix(a), gb.colmajor(128, 300, fill=0.0), _gpu.device_matrix(a)
        torch.cuda.synchronize()
        graph = ctx.capture(lambda: ctx.factor(B, U, gb.GBQR_T_PANEL))
        for _ in range(2):
            B.copy_(fresh)
            torch.cuda.synchronize()
            graph.launch()
            torch.cuda.synchronize()
            assert torch.equal(A, B) and torch.equal(T, U)
        graph.close()

"""Solves with deep factors (natural elimination order: many dependency levels) --
the level pipeline with C_a over a cluster of CTAs, and the panels of exact
factors -- against the launch per level, over cluster sizes and problems: levels
of less than a slice, ragged grids, fill, blocks of less than a panel and with a
partial last one, FP64 and FP32, the Chebyshev solve's D_a.  The pipeline sums a
row's entries in the order of the levels and agrees to a few roundings; the
panels multiply by inverse triangles of 32 rows, so there the bound is the A0
solve's own: n eps cond(A0), below 1e-12 (FP64) on these problems."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

PROBLEMS = {
    "2d_64_exact": ((64, 64), (2, 2), dict(factor=1)),
    "2d_27x23_exact": ((27, 23), (2, 3), dict(factor=1)),
    "2d_16x9_exact": ((16, 9), (2, 2), dict(factor=1)),
    "3d_12x11x10_exact": ((12, 11, 10), (2, 2, 1), dict(factor=1)),
    "2d_40x30_exact_multicolour": ((40, 30), (3, 2), dict(factor=1, b_order=1, c_order=1)),
    "2d_37x50_ic0": ((37, 50), (3, 2), dict()),
    "3d_20": ((20, 20, 20), (2, 2, 2), dict()),
    "3d_33x17x21": ((33, 17, 21), (3, 2, 2), dict()),
    "3d_24_ic2": ((24, 24, 24), (2, 2, 2), dict(fill_level=2)),
    "3d_24_ic1_multicolour": ((24, 24, 24), (2, 3, 2), dict(fill_level=1, b_order=1, c_order=1)),
    "3d_48": ((48, 48, 48), (3, 3, 3), dict()),
    "3d_40_multicolour_b": ((40, 30, 35), (3, 2, 3), dict(b_order=1)),
    "3d_24_cheb": ((24, 24, 24), (3, 3, 3), dict(c_solver=1)),
}


def _solve(name, monkeypatch, ctas, precision):
    shape, boxes, kw = PROBLEMS[name]
    monkeypatch.setenv("DDLR_DEEP", "0" if ctas == 0 else "1")
    monkeypatch.setenv("DDLR_DEEP_CTAS", str(max(1, ctas)))
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, boxes)
    h = pkg.DDLR(A, part, p, rank_k=4, precision=precision, **kw)
    y = h.a0_solve(W.rhs(A[0], 3))
    _, info = h.pcg(W.rhs(A[0], 4), tol=1e-8)
    h.close()
    return y, info[0]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_cluster_solve_matches_levels(name, precision, monkeypatch):
    ref, iref = _solve(name, monkeypatch, 0, precision)
    eps = np.finfo(np.float64 if precision == 0 else np.float32).eps
    for ctas in (1, 2, 4, 8, 16):
        y, inf = _solve(name, monkeypatch, ctas, precision)
        tol = 5000 * eps if PROBLEMS[name][2].get("factor") else 8 * eps
        assert np.abs(y - ref).max() <= tol * np.abs(ref).max(), ctas
        assert inf["status"] == "OK" and abs(inf["its"] - iref["its"]) <= 1

"""The persistent kernels' reductions (block sums by four warps, column folds,
four-column Gram-Schmidt products, row dots with and without 16-byte loads) over
ranks that divide no warp evenly, against the per-phase kernels (DDLR_PERSIST=0):
the same solution to the accuracy that a change of summation order leaves in a
solve to 1e-8 (1e-10), the same Ritz values (1e-9), the same iterations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("variant", [1, 2])
@pytest.mark.parametrize("k", [1, 3, 7, 20, 33, 64, 70, 130])
def test_ranks(k, variant, precision, monkeypatch):
    shape = (21, 18, 19)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 2))
    b = W.rhs(A[0], 1)
    got = []
    for persist in ("1", "0"):
        monkeypatch.setenv("DDLR_PERSIST", persist)
        h = pkg.DDLR(A, part, p, variant=variant, rank_k=k, c_order=1, b_order=1, precision=precision)
        assert (h.info()["persistent"] != 0) == (persist == "1")
        x, info = h.pcg(b, tol=1e-8)
        got.append((x, info[0]["its"], h.ritz()[:k]))
        h.close()
    (x1, i1, r1), (x0, i0, r0) = got
    assert i1 == i0
    assert np.linalg.norm(x1 - x0) <= 1e-10 * np.linalg.norm(x0)
    assert np.abs(r1 - r0).max() <= 1e-9 * np.abs(r0).max()

"""Column reductions of the block PCG in their two forms -- a CTA per group of ranges
for narrow blocks with few rows, else a CTA per range -- on both sides of the line
between them: 25 and 27 reduced columns (mixed precision reduces two per right-hand
side), 4,864 row blocks, less than one row block per range and the last one ragged.
Both add in the same order, so a column's solution has the same bits in every block
whose kernels are otherwise the same (odd widths: the scalar forms)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape, widths", [((9, 7, 5), (3, 25, 27)), ((24, 25, 23), (3, 13, 25, 27, 31)),
                                           ((67, 68, 68), (3, 13, 27)), ((68, 68, 68), (3, 13))])
@pytest.mark.parametrize("kw", [{}, dict(precision=1), dict(scale_diag=1)], ids=str)
def test_columns_have_the_same_bits(shape, widths, kw):
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 2))
    B = np.stack([W.rhs(A[0], s) for s in range(max(widths))], axis=1)
    ref = None
    for R in sorted(widths, reverse=True):
        h = pkg.DDLR(A, part, p, rank_k=4, c_order=1, b_order=1, max_nrhs=R, **kw)
        X, info = h.pcg(np.asfortranarray(B[:, :R]), tol=1e-8)
        h.close()
        assert all(i["status"] == "OK" for i in info)
        if ref is None:
            ref = X, info
        assert np.array_equal(X, ref[0][:, :R])
        assert [i["its"] for i in info] == [i["its"] for i in ref[1][:R]]

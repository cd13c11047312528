"""First solves restricted to the rows that E^T reads where C_a is solved with
approximately (Chebyshev steps, the approximate inverse): the tail after the sweeps
reads interface rows alone, which are all kept, so the bits are those of the solve
over all rows (DDLR_E_ROWS=0)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kw", [dict(c_solver=1), dict(c_solver=2), dict(c_solver=2, variant=2)], ids=str)
def test_same_bits(kw, precision, monkeypatch):
    shape, boxes = (33, 17, 21), (3, 2, 2)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, boxes)
    B = np.asfortranarray(np.stack([W.rhs(A[0], 3 + j) for j in range(5)], axis=1))
    got = []
    for all_rows in (True, False):
        if all_rows:
            monkeypatch.setenv("DDLR_E_ROWS", "0")
        else:
            monkeypatch.delenv("DDLR_E_ROWS")
        h = pkg.DDLR(A, part, p, rank_k=4, c_order=1, b_order=1, max_nrhs=5, precision=precision, **kw)
        assert h.info()["levels_interior"] == 2
        got.append([h.apply(B[:, 0].copy()), h.pcg(B[:, 1].copy(), tol=1e-8)[0], h.apply(B), h.pcg(B, tol=1e-8)[0]])
        h.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)

"""Solves that only E^T reads (the first of a DDLR-1 apply, the Lanczos operator),
restricted to the rows it needs, against the same solves over all rows
(DDLR_E_ROWS=0): every row kept has the same arithmetic, so the bits are the same.
Boxes one node wide (every interior row next to the interface, or none left) to
boxes with a deep inside, both kernel paths, every precision, narrow and wide blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

GRIDS = {"7x5": ((7, 5), (3, 2)), "40x33": ((40, 33), (2, 2)), "9x9x9": ((9, 9, 9), (4, 4, 4)),
         "33x17x21": ((33, 17, 21), (3, 2, 2)), "24x25x26": ((24, 25, 26), (1, 1, 2))}


@pytest.mark.parametrize("kw", [{}, dict(variant=2), dict(precision=1), dict(precision=1, uk_bf16=1, scale_diag=1)], ids=str)
@pytest.mark.parametrize("persist", ["0", "1"])
@pytest.mark.parametrize("grid", GRIDS)
def test_same_bits(grid, persist, kw, monkeypatch):
    monkeypatch.setenv("DDLR_PERSIST", persist)
    shape, boxes = GRIDS[grid]
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, boxes)
    n = A[0]
    got = []
    for all_rows in (True, False):
        if all_rows:
            monkeypatch.setenv("DDLR_E_ROWS", "0")
        else:
            monkeypatch.delenv("DDLR_E_ROWS")
        h = pkg.DDLR(A, part, p, rank_k=4, c_order=1, b_order=1, max_nrhs=6, **kw)
        if grid in ("33x17x21", "40x33"):
            assert h.info()["levels_interior"] == 2
        out = [h.apply(W.rhs(n, 1)), h.pcg(W.rhs(n, 2), tol=1e-8)[0]]
        for r in (5, 6):                       # scalar and 16-byte column forms
            B = np.asfortranarray(np.stack([W.rhs(n, 3 + j) for j in range(r)], axis=1))
            out += [h.apply(B), h.pcg(B, tol=1e-8)[0]]
        got.append(out)
        h.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)

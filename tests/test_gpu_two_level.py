"""FP32 solves with two-level factors: the grouped-entry kernel against the
entry-by-entry one (DDLR_CHUNK_ROWS=4).  The arithmetic of a row is the same, so
the bits are; rows of 0 to 14 entries (a group holds 6) and ragged last CTAs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def stars(leaves, per_part, parts):
    """Disjoint stars (any first-fit colouring has two colours): hub rows of up to
    `leaves` entries; the first leaf of a star couples to that of its like in the next part."""
    size = leaves + 1
    n = size * per_part * parts
    e = [(h, h + 1 + q) for h in range(0, n, size) for q in range(leaves)]
    e += [(h + 1, h + size * per_part + 1) for h in range(0, n - size * per_part, size)]
    D = (leaves + 2.0) * np.eye(n)
    for i, j in e:
        D[i, j] = D[j, i] = -1.0
    rows, cols = np.nonzero(D)
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))])
    part = (np.arange(n) // (size * per_part)).astype(np.int32)
    return (n, rp.astype(np.int32), cols.astype(np.int32), D[rows, cols]), part


@pytest.mark.parametrize("kw", [{}, dict(scale_diag=1), dict(variant=2)], ids=str)
@pytest.mark.parametrize("case", ["s1", "s5", "s7", "s14", "lap2d", "lap3d", "jump"])
def test_same_bits(case, kw, monkeypatch):
    monkeypatch.setenv("DDLR_PERSIST", "0")
    if case[0] == "s":
        p = 3
        A, part = stars(int(case[1:]), 25, p)
    else:
        shape = {"lap2d": (41, 37), "lap3d": (17, 13, 19), "jump": (16, 16, 16)}[case]
        A = W.jump_coefficient_fv(16, 4, 0) if case == "jump" else W.laplacian(shape)
        part, p = W.box_partition(shape, (2,) * len(shape))
    b = W.rhs(A[0], 1)
    got = []
    for rows in (None, "4"):
        if rows:
            monkeypatch.setenv("DDLR_CHUNK_ROWS", rows)
        h = pkg.DDLR(A, part, p, rank_k=4, c_order=1, b_order=1, precision=1, **kw)
        assert h.info()["levels_interior"] <= 2
        got.append((h.a0_solve(b), h.apply(b), h.pcg(b, tol=1e-8)[0]))
        h.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)

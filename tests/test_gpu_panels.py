"""Accuracy of the panel solves of exact factors, which multiply by the inverse
triangles of 32 rows, on factors that are badly scaled or badly conditioned: the
error of A0 z = x against the same factor solved in extended precision is that of
the level sweeps (at most twice theirs, and four roundings for entries that both
get right).  The panels took the solve: C_a in one launch that is not the
pipeline's, and other last bits than the levels'."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPE = (37, 41)


def _matrix(kind):
    A = W.to_scipy(W.laplacian(SHAPE)).tocsr()
    n = A.shape[0]
    u = np.random.default_rng(5).uniform(-1, 1, n)
    if kind == "scaled":                       # D A D, entries over twelve decades
        D = sp.diags(10.0 ** (3 * u))
        A = D @ A @ D
    elif kind == "jump":                       # couplings of cells whose coefficients span eight decades
        k = 10.0 ** (4 * u)
        C = sp.triu(A, 1).tocoo()
        w = 2 * k[C.row] * k[C.col] / (k[C.row] + k[C.col])
        G = sp.coo_matrix((w, (C.row, C.col)), shape=A.shape)
        G = G + G.T
        A = sp.diags(np.asarray(G.sum(1)).ravel() + k) - G
    elif kind == "squared":                    # 13 points, positive and negative couplings
        A = A @ A
    A = sp.csr_matrix(A)
    A = (A + A.T) * 0.5                        # the same bits on both sides
    A.sort_indices()
    return n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data.astype(np.float64)


def _solve_extended(r, c, v, x):
    """(L L^T)^-1 x from the factor's entries, in extended precision."""
    n = len(x)
    assert (c <= r).all()
    z = x.astype(np.longdouble)
    L = sp.csr_matrix((v, (r, c)), shape=(n, n))
    L.sort_indices()
    rows = [(L.indices[a:b], L.data[a:b].astype(np.longdouble)) for a, b in zip(L.indptr, L.indptr[1:])]
    for i, (ci, vi) in enumerate(rows):
        z[i] = (z[i] - (vi[:-1] * z[ci[:-1]]).sum()) / vi[-1]
    for i in range(n - 1, -1, -1):
        ci, vi = rows[i]
        z[i] /= vi[-1]
        z[ci[:-1]] -= vi[:-1] * z[i]
    return z


@pytest.mark.parametrize("kind", ["laplacian", "scaled", "jump", "squared"])
def test_panels_are_as_accurate_as_levels(kind, monkeypatch):
    A = _matrix(kind)
    part, p = W.box_partition(SHAPE, (2, 2))
    got = []
    for deep in ("0", "1"):
        monkeypatch.setenv("DDLR_DEEP", deep)
        h = pkg.DDLR(A, part, p, rank_k=2, lanczos_max=4, factor=1)
        xs = [W.rhs(A[0], 1), W.to_scipy(A) @ W.rhs(A[0], 2)]
        if deep == "1":
            monkeypatch.setenv("DDLR_TEST_DEEP_GIVE_UP", "0")     # the pipeline would time out
        h.reset_counters()
        ys = [h.a0_solve(x) for x in xs]
        monkeypatch.delenv("DDLR_TEST_DEEP_GIVE_UP", raising=False)
        launches = h.counters()["families"]["sptrsv_c"]["launches"]
        assert launches == 2 if deep == "1" else launches > 2
        got.append(ys)
        fac = h.factor_coo()
        h.close()
    eps = np.finfo(np.float64).eps
    for x, lev, pan in zip(xs, *got):
        z = _solve_extended(*fac, x)
        err = [float(np.abs(y - z).max() / np.abs(z).max()) for y in (lev, pan)]
        assert not np.array_equal(lev, pan)
        assert err[1] <= 2 * err[0] + 4 * eps, err

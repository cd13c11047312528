"""Which DDLR-2 applies and GMRES solves of shallow factors go in one launch: on
both sides of the rule's lines (elements of U_k, its type, vector loads or not) the
route is the expected one and the result that of the per-phase kernels, to the
bounds of test_gpu_persist_apply.py (the same sums in another order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

FP32, BF16 = dict(precision=1), dict(precision=1, uk_bf16=1)


def _families(h):
    return {f for f, v in h.counters()["families"].items() if v["launches"]}


# n k against 6e6 (n >= 100000) in mixed precision, 12e6 (k <= 32) in FP64; GMRES
# against 14e6 + 0.24e6 m in mixed precision
@pytest.mark.parametrize("edge, k, kw, one_apply, one_gmres",
                         [(48, 32, BF16, True, True), (48, 64, FP32, False, True), (48, 60, BF16, True, True),
                          (48, 256, BF16, False, False), (45, 128, FP32, True, True), (48, 128, {}, True, True),
                          (74, 32, {}, False, True), (74, 24, {}, True, True)])
def test_route(edge, k, kw, one_apply, one_gmres, monkeypatch):
    shape = (edge, edge, edge)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (3, 3, 3))
    h = pkg.DDLR(A, part, p, variant=2, rank_k=k, lanczos_max=k, c_order=1, b_order=1, **kw)
    U, _, _, Hk = h.lowrank()
    x = W.rhs(A[0], 3)
    h.reset_counters()
    y = h.apply(x)
    assert ("apply_persist" in _families(h)) == one_apply
    h.reset_counters()
    z, i1 = h.gmres(x, tol=1e-30, maxit=6, restart=10, check=False)
    assert ("gmres_persist" in _families(h)) == one_gmres
    h.close()
    monkeypatch.setenv("DDLR_PERSIST", "0")
    h = pkg.DDLR(A, part, p, variant=2, rank_k=k, lanczos_max=k, c_order=1, b_order=1, **kw)
    h.set_lowrank(U, Hk=Hk)
    tol = 1e-12 if not kw else (1e-4 if kw.get("uk_bf16") else 1e-5)
    y0, (z0, i0) = h.apply(x), h.gmres(x, tol=1e-30, maxit=6, restart=10, check=False)
    assert np.linalg.norm(y - y0) <= tol * np.linalg.norm(y0)
    assert i1["its"] == i0["its"]
    assert np.linalg.norm(z - z0) <= 10 * tol * np.linalg.norm(z0)
    h.close()

"""DDLR-2's H_k = (I - U_k^T E V_k)^-1 (lemma 1) at the sizes where the kernels
that form it change shape: one column, the widths around a warp and around the
shared-memory and batched-solve limit of 64 columns, odd ranks, SPD (Cholesky)
and indefinite (Gauss-Jordan) problems, deep and shallow factors.

With exact local factors U_k = A0^-1 E V_k, so U_k^T E V_k = U_k^T A0 U_k: the
reference is formed from the returned U_k and the dense A0 of the definitions.
Tolerance: the sums of k products over n rows carry at most about n eps of
their size and the inversion amplifies them by cond(I - K): 4 n eps cond."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402
from dense_ddlr import DenseDDLR  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lowrank", [0, 2])
@pytest.mark.parametrize("indefinite", [0, 1])
@pytest.mark.parametrize("k", [1, 2, 31, 33, 64, 65, 79])
def test_hk_matches_definition(k, indefinite, lowrank):
    shape = (27, 23)
    A = W.shifted_laplacian(shape, 0.08) if indefinite else W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2))
    h = pkg.DDLR(A, part, p, variant=2, rank_k=k, factor=1, indefinite=indefinite, lowrank_method=lowrank)
    U, _, _, Hk = h.lowrank()
    h.close()
    D = DenseDDLR(A, part, p)
    K = U.T @ D.to_original(D.A0) @ U
    G = np.eye(k) - 0.5 * (K + K.T)
    ref = np.linalg.inv(G)
    tol = 4 * A[0] * np.finfo(float).eps * np.linalg.cond(G)
    assert np.abs(Hk - ref).max() <= tol * np.abs(ref).max()

"""Bytes per kernel family of deep A0 solves: the launches of one solve, each with
the bytes its family is said to move, make up the bytes of the solve, whichever
kernels take C_a -- the level pipeline, the panels or a launch per level."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape, boxes, kw, deep, launches_c",
                         [((20, 20, 20), (2, 2, 2), {}, "1", 1), ((48, 40), (2, 2), dict(factor=1), "1", 1),
                          ((20, 20, 20), (2, 2, 2), {}, "0", None)])
def test_families_add_up(shape, boxes, kw, deep, launches_c, precision, monkeypatch):
    monkeypatch.setenv("DDLR_DEEP", deep)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, boxes)
    h = pkg.DDLR(A, part, p, rank_k=4, precision=precision, **kw)
    h.reset_counters()
    h.a0_solve(W.rhs(A[0], 1))
    fam = {f: v["launches"] for f, v in h.counters()["families"].items() if f.startswith("sptrsv")}
    t = h.traffic()
    assert fam["sptrsv_c"] == (launches_c or 2 * h.info()["levels_c"] - 1)
    total = sum(n * t["family_bytes"][f] for f, n in fam.items())
    assert total == pytest.approx(t["a0_bytes"], rel=1e-12)
    h.close()

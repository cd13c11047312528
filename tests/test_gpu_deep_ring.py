"""Deep solves with few stages of the factor in shared memory at a time: rings of
one stage (DDLR_DEEP_STAGES) up against the launch per level, and the blocks that
leave room for few -- wide ones, and several to an SM.  That the pipeline serves
them is seen from DDLR_TEST_DEEP_GIVE_UP, which only its kernel knows.  A row's
entries are summed in the order of the levels: a few roundings apart at most."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _solve(shape, boxes, monkeypatch, deep, served=None, **kw):
    monkeypatch.setenv("DDLR_DEEP", "1" if deep else "0")
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, boxes)
    h = pkg.DDLR(A, part, p, rank_k=2, lanczos_max=4, **kw)
    x = W.rhs(A[0], 3)
    if served is not None:
        monkeypatch.setenv("DDLR_TEST_DEEP_GIVE_UP", "0")
        if served:
            with pytest.raises(pkg.DdlrError) as e:
                h.a0_solve(x)
            assert e.value.status == "TIMEOUT"
        else:
            h.a0_solve(x)
        monkeypatch.delenv("DDLR_TEST_DEEP_GIVE_UP")
    y = h.a0_solve(x)
    h.close()
    return y


def _close(y, ref, precision):
    eps = np.finfo(np.float64 if precision == 0 else np.float32).eps
    assert np.abs(y - ref).max() <= 8 * eps * np.abs(ref).max()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ctas", [1, 2, 8])
@pytest.mark.parametrize("kw", [dict(), dict(fill_level=2)], ids=str)
def test_short_rings(kw, ctas, precision, monkeypatch):
    shape, boxes = (33, 26, 21), (3, 2, 2)
    ref = _solve(shape, boxes, monkeypatch, False, precision=precision, **kw)
    monkeypatch.setenv("DDLR_DEEP_CTAS", str(ctas))
    for stages in (1, 2, 3, 5):
        monkeypatch.setenv("DDLR_DEEP_STAGES", str(stages))
        _close(_solve(shape, boxes, monkeypatch, True, served=True, precision=precision, **kw), ref, precision)


# interior blocks alone (C_a in a multicolour order): edges of 23 and 28 nodes (the
# widest in FP64), of 35 (the widest in FP32), four to an SM, one past the widest
@pytest.mark.parametrize("shape, boxes, precision, served",
                         [((48, 48, 48), (2, 2, 2), 0, True), ((58, 58, 58), (2, 2, 2), 0, True),
                          ((72, 72, 72), (2, 2, 2), 1, True), ((96, 96, 96), (8, 8, 8), 0, True),
                          ((128, 128, 128), (8, 8, 8), 0, True), ((128, 128, 128), (8, 8, 8), 1, True),
                          ((62, 62, 62), (2, 2, 2), 0, False)])
def test_wide_blocks_are_served(shape, boxes, precision, served, monkeypatch):
    kw = dict(precision=precision, c_order=1)
    ref = _solve(shape, boxes, monkeypatch, False, **kw)
    _close(_solve(shape, boxes, monkeypatch, True, served=served, **kw), ref, precision)

"""The one-launch preconditioner apply and GMRES of shallow factors against the
per-phase kernels (DDLR_PERSIST=0).  Both evaluate the same sums in another
order: an apply agrees to the rounding of its type times the condition of its
few steps (1e-12 in FP64, 1e-5 in FP32), a GMRES solve to 1e-6 in the residual
to 1e-9 in its iterate (FP64; mixed 1e-6, one rounding of M^-1 v per step), with
the same iterations in FP64 and at most one apart in mixed precision.  Also:
repeated calls give the same bits (the kernels reset their own barriers), a
captured apply replays, and a wait that runs out is reported and recovered
from."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

MC = dict(c_order=1, b_order=1)


def handles(A, part, p, monkeypatch, **kw):
    out = []
    for persist in ("1", "0"):
        monkeypatch.setenv("DDLR_PERSIST", persist)
        out.append(pkg.DDLR(A, part, p, **MC, **kw))
    assert out[0].info()["persistent"] and not out[1].info()["persistent"]
    return out


def close(a, b, tol):
    return np.linalg.norm(a - b) <= tol * np.linalg.norm(b)


# one CTA (n < 256), a ragged last CTA, more than 152 CTAs' worth of rows
@pytest.mark.parametrize("shape", [(7, 5, 6), (21, 18, 19), (35, 34, 36)])
@pytest.mark.parametrize("kw", [dict(variant=1, rank_k=1), dict(variant=1, rank_k=7, precision=1),
                                dict(variant=1, rank_k=8, precision=1, uk_bf16=1), dict(variant=2, rank_k=9),
                                dict(variant=2, rank_k=6, precision=1), dict(variant=1, rank_k=5, scale_diag=1)],
                         ids=str)
def test_apply(shape, kw, monkeypatch):
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 1))
    h1, h0 = handles(A, part, p, monkeypatch, **kw)
    x = W.rhs(A[0], 3)
    tol = 1e-5 if kw.get("precision") else 1e-12
    y = h1.apply(x)
    assert close(y, h0.apply(x), tol if not kw.get("uk_bf16") else 1e-4)
    for _ in range(3):
        assert np.array_equal(h1.apply(x), y)
    xd = torch.tensor(x, device="cuda")
    s = torch.cuda.Stream()
    h1.set_stream(s)
    yd = torch.zeros_like(xd)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        h1.apply(xd, yd)
    for _ in range(2):
        yd.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(yd.cpu().numpy(), y)
    xd2 = xd.clone()                                   # in place
    torch.cuda.synchronize()
    h1.apply(xd2, xd2)
    torch.cuda.synchronize()
    assert np.array_equal(xd2.cpu().numpy(), y)
    h1.close(); h0.close()


@pytest.mark.parametrize("restart", [1, 2, 31, 33, 128, 129])
@pytest.mark.parametrize("kw", [dict(rank_k=6), dict(rank_k=5, precision=1), dict(rank_k=4, scale_diag=1)], ids=str)
def test_gmres(restart, kw, monkeypatch):
    shape = (17, 14, 15)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 1))
    h1, h0 = handles(A, part, p, monkeypatch, **kw)
    b = W.rhs(A[0], 2)
    mixed = bool(kw.get("precision"))
    x1, i1 = h1.gmres(b, tol=1e-6, maxit=300, restart=restart, check=False)
    x0, i0 = h0.gmres(b, tol=1e-6, maxit=300, restart=restart, check=False)
    assert i1["status"] == i0["status"] and abs(i1["its"] - i0["its"]) <= int(mixed)
    assert close(x1, x0, 1e-5 if mixed else 1e-9)
    assert np.array_equal(h1.gmres(b, tol=1e-6, maxit=300, restart=restart, check=False)[0], x1)
    for maxit in (1, 5):                             # unfinished: within a cycle and at its end
        x1, i1 = h1.gmres(b, tol=1e-12, maxit=maxit, restart=restart, check=False)
        x0, i0 = h0.gmres(b, tol=1e-12, maxit=maxit, restart=restart, check=False)
        assert (i1["its"], i1["status"]) == (i0["its"], i0["status"]) == (maxit, "NOCONV")
        assert np.linalg.norm(x1 - x0) <= (1e-5 if mixed else 1e-11) * np.linalg.norm(x0)
    x1, i1 = h1.gmres(np.zeros_like(b), tol=1e-6, restart=restart)
    assert not x1.any() and i1["its"] == 0 and i1["status"] == "OK"
    bad = b.copy()
    bad[7] = np.inf
    assert h1.gmres(bad, restart=restart, check=False)[1]["status"] == "NAN"
    h1.close(); h0.close()


def test_timeout(monkeypatch):
    shape = (21, 18, 19)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 2))
    h = pkg.DDLR(A, part, p, rank_k=4, **MC)
    x = W.rhs(A[0], 1)
    y, (z, _) = h.apply(x), h.gmres(x, tol=1e-6)
    h.set_wait_limit(1e-3)
    for call in (lambda: h.apply(x), lambda: h.gmres(x, tol=1e-6)):
        monkeypatch.setenv("DDLR_TEST_UNMET_BARRIER", "1")
        with pytest.raises(pkg.DdlrError) as e:
            call()
        assert e.value.status == "TIMEOUT"
        monkeypatch.delenv("DDLR_TEST_UNMET_BARRIER")
        h.set_wait_limit(2.0)
        assert np.array_equal(h.apply(x), y)
        assert np.array_equal(h.gmres(x, tol=1e-6)[0], z)
        h.set_wait_limit(1e-3)
    h.close()

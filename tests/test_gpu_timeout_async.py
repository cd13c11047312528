"""A wait that runs out in an apply into device memory, which does not read the
timeout flag: the launches after it find the barrier's counters as they should be
and give the same bits as before, and the next call that waits for the device
reports the timeout, once.

The wait is made to run out as in test_gpu_timeout.py: DDLR_TEST_UNMET_BARRIER=1
lets the first grid barrier of a launch wait for an arrival that nothing provides,
for 1 ms."""
import time

import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1505_04341_gb300 as pkg  # noqa: E402
import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _handle(shape=(21, 18, 19), **kw):
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 2))
    h = pkg.DDLR(A, part, p, rank_k=4, c_order=1, b_order=1, **kw)
    return h, torch.tensor(W.rhs(A[0], 1), device="cuda")


def _unmet_apply(h, x, y, monkeypatch):
    """An apply whose wait runs out; nothing is reported yet."""
    h.set_wait_limit(1e-3)
    monkeypatch.setenv("DDLR_TEST_UNMET_BARRIER", "1")
    h.apply(x, y)
    torch.cuda.synchronize()
    monkeypatch.delenv("DDLR_TEST_UNMET_BARRIER")
    h.set_wait_limit(2.0)


def _times_out(call):
    with pytest.raises(pkg.DdlrError) as e:
        call()
    assert e.value.status == "TIMEOUT"


@pytest.mark.parametrize("kw", [{}, dict(variant=2), dict(precision=1, uk_bf16=1)], ids=str)
def test_later_launches_are_not_affected(kw, monkeypatch):
    h, x = _handle(**kw)
    y0 = h.apply(x).clone()
    z0, _ = h.gmres(x, tol=1e-6)
    z0 = z0.clone()
    for _ in range(2):                      # the second: after a launch that left its counters in order
        y = torch.full_like(x, 7.0)
        _unmet_apply(h, x, y, monkeypatch)
        for _ in range(3):
            y = torch.full_like(x, 7.0)
            h.apply(x, y)
            torch.cuda.synchronize()
            assert torch.equal(y, y0)
        _times_out(lambda: h.apply(x.cpu().numpy()))       # the first call that waits
        assert (h.apply(x.cpu().numpy()) == y0.cpu().numpy()).all()
        assert torch.equal(h.gmres(x, tol=1e-6)[0], z0)
    h.close()


@pytest.mark.parametrize("call", ["refactor", "set_lowrank", "batch"])
def test_pending_timeout_is_reported(call, monkeypatch):
    """No call that waits clears the flag without reporting it, and the call
    repeated then leaves the handle as it was."""
    h, x = _handle(max_nrhs=3)
    U, lam, theta, _ = h.lowrank()
    X = torch.stack([x, 2 * x, -x]).T

    def run():
        if call == "refactor":
            h.refactor()
        elif call == "set_lowrank":
            h.set_lowrank(U, lam, theta)
        else:
            return h.apply(X.cpu().numpy())

    run()
    y0 = h.apply(x).clone()
    _unmet_apply(h, x, torch.empty_like(x), monkeypatch)
    _times_out(run)
    run()
    assert torch.equal(h.apply(x), y0)
    h.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ctas", [1, 2, 8])
def test_deep_solve_gives_up(ctas, precision, monkeypatch):
    """A part of a deep solve that gives up after some stage (DDLR_TEST_DEEP_GIVE_UP)
    leaves when the transfers into its shared memory have arrived, well before
    the limit of that wait, and so do its peers."""
    monkeypatch.setenv("DDLR_DEEP_CTAS", str(ctas))
    shape = (30, 29, 31)
    A = W.laplacian(shape)
    part, p = W.box_partition(shape, (2, 2, 3))
    h = pkg.DDLR(A, part, p, rank_k=4, precision=precision)
    x = W.rhs(A[0], 1)
    y0 = h.a0_solve(x)
    levels = h.info()["levels_c"]
    for at in (0, 1, 7, levels // 2, levels - 1, levels, levels + 9, 2 * levels - 1):
        monkeypatch.setenv("DDLR_TEST_DEEP_GIVE_UP", str(at))
        t = time.perf_counter()
        if at <= 7:                        # a stage that every part has
            _times_out(lambda: h.a0_solve(x))
        else:
            try:
                h.a0_solve(x)
            except pkg.DdlrError as e:
                assert e.status == "TIMEOUT"
        assert time.perf_counter() - t < 0.5
        monkeypatch.delenv("DDLR_TEST_DEEP_GIVE_UP")
        assert (h.a0_solve(x) == y0).all()
    h.close()

"""A context replays captured graphs of its solves; a call that differs in anything the captured
launches hold must not get the old graph.  Every solve on the shared context is compared with the same
solve on a context of its own.

Tolerance: both solves end below a relative residual of 1e-10 with the same kernels: 1e-9 of the
largest component (the preconditioned operator's condition number is below ~10)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(gbi, ctx, R, p, a, trunc, precision, repeats=1):
    i = ctx.trap_inputs(R.shape[0], trunc, 0.01, 0.1, 0.05, 0.02, R, p)
    prm = gbi.params(a=a, eta=0.05, trunc=trunc, precision=precision, rtol=1e-10)
    for _ in range(repeats):
        out = ctx.solve(prm, R, i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"])
    ctx.synchronize()
    return out[:3]


def _inputs(N, seed):
    import torch
    import workloads
    s = workloads.small_cloud(N, seed, phi=0.05, dmin=2.3)
    return [torch.tensor(np.ascontiguousarray(s[k]), dtype=torch.float64, device="cuda") for k in ("R", "p")]


def _same(got, ref):
    for x, y in zip(got, ref):
        assert float((x - y).abs().max()) <= 1e-9 * max(float(y.abs().max()), 1e-6)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("N", [60, 400])   # one-cluster step, separate kernels
def test_another_radius(N, precision):
    """The same suspension with spheres of another radius (no two overlap)."""
    import torch
    import paper_1411_0278_gb300 as gbi
    R, p = _inputs(N, 3)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = gbi.Context(0, stream=stream)
    for a in (1.0, 0.5, 1.1, 1.0):
        got = _solve(gbi, ctx, R, p, a, 2, precision)
        own = gbi.Context(0, stream=stream)
        _same(got, _solve(gbi, own, R, p, a, 2, precision))
        own.close()
    ctx.close()


@pytest.mark.parametrize("N,trunc,precision,wpt", [(642, 3, 2, 0), (1000, 3, 2, 0), (1000, 3, 3, 0), (1024, 3, 1, 0),
                                                   (300, 2, 1, 1), (300, 2, 1, 3), (300, 2, 3, 1)])
def test_scratch_before_the_capture(N, trunc, precision, wpt):
    """A fresh context captures the FP32 pass of its first solve before that pass has run; the split
    tail's and the balanced forms' scratch has to be there (forced forms, and sizes at which the
    FP32 pass needs more of it than the double-float one)."""
    import torch
    import paper_1411_0278_gb300 as gbi
    R, p = _inputs(N, 5)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    plain = gbi.Context(0, stream=stream)
    ref = _solve(gbi, plain, R, p, 1.0, trunc, precision)
    plain.close()
    ctx = gbi.Context(0, stream=stream)
    ctx.set_split_tail(1)
    ctx.set_wpt(wpt)
    for _ in range(3):       # direct, capture, replay
        got = _solve(gbi, ctx, R, p, 1.0, trunc, precision)
        for x, y in zip(got, ref):
            tol = 1e-9 if precision < 3 else 1e-5
            assert float((x - y).abs().max()) <= tol * float(y.abs().max())
    assert ctx.solve_graph_replays() >= 1
    ctx.close()


def test_scratch_that_moves_between_solves():
    """A larger pass grows (and moves) the split tail's scratch while every other buffer stays: the next
    solve's steps must use the new one."""
    import torch
    import paper_1411_0278_gb300 as gbi
    N, trunc = 1000, 3
    R, p = _inputs(N, 6)
    big, _ = _inputs(3040, 7)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        torch.cuda.synchronize()
        ctx = gbi.Context(0, stream=stream)
        ctx.set_split_tail(1)
        x = torch.randn(25, 3040, dtype=torch.float64, device="cuda")
        y = torch.zeros_like(x)
        ctx.apply(3040, trunc, 1.0, 2, 2, 1, big, x, y)      # five full waves: buffers for 3040, no split
        ref = _solve(gbi, ctx, R, p, 1.0, trunc, 2)
        ctx.apply(2900, trunc, 1.0, 2, 2, 1, big, x, y)      # a tail of 468 targets in five parts
        for _ in range(3):
            _same(_solve(gbi, ctx, R, p, 1.0, trunc, 2), ref)
        ctx.close()


@pytest.mark.parametrize("precision", [1, 2])
def test_wait_limit_of_a_replayed_solve(precision):
    """gbi_set_wait_limit holds for later solves of captured sizes too: with no rounds every stage wait of
    the tiled passes gives up, with the default restored the results are back."""
    import torch
    import paper_1411_0278_gb300 as gbi
    R, p = _inputs(100, 8)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = gbi.Context(0, stream=stream)
    ctx.set_wpt(1)
    ref = _solve(gbi, ctx, R, p, 1.0, 2, precision, repeats=3)
    i = ctx.trap_inputs(100, 2, 0.01, 0.1, 0.05, 0.02, R, p)
    prm = gbi.params(a=1.0, eta=0.05, trunc=2, precision=precision, rtol=1e-10, max_iter=60, max_refine=3)
    short = lambda: ctx.solve(prm, R, i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"], allow_not_converged=True)
    for _ in range(3):
        short()
    ctx.set_wait_limit(0)
    for _ in range(3):
        with pytest.raises(gbi.GbiError) as err:
            short()
        assert err.value.status == gbi.GBI_ERR_TIMEOUT
    ctx.set_wait_limit(-1)
    for _ in range(3):
        _same(_solve(gbi, ctx, R, p, 1.0, 2, precision), ref)
    ctx.close()

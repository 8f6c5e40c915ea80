"""Solves of one small system, whose Arnoldi steps run on one cluster of blocks: against the dense
oracle solve at sizes around the slices (fewer elements than blocks, ragged slices) and around the
limits of the form (n = 1536 in one round, 4096 in two).

Tolerance: the residual is below 1e-10 and the operator's condition number below ~10: 1e-8 of the
largest component (as the parity tests of the solver); precision 3 carries FP32 outputs, 1e-5."""
import numpy as np
import pytest

from oracle import dynamics, galerkin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,trunc", [(1, 2), (2, 3), (3, 4), (13, 2), (61, 3), (62, 3), (32, 4), (192, 2), (193, 2)])
@pytest.mark.parametrize("precision", [0, 2, 3])
def test_small_solves(N, trunc, precision):
    import torch
    import paper_1411_0278_gb300 as gbi
    import workloads
    s = workloads.small_cloud(N, 60 + N, phi=0.05, dmin=2.3)
    inp = dynamics.trap_inputs(s["R"], s["p"], dict(a=s["a"], eta=s["eta"], k=s["k"], vs=s["vs"], s0=s["s0"], d0=0.02),
                               trunc)
    ref = galerkin.solve(s["R"], inp["Va"], inp["Oa"], inp["VH"], inp["Fe"], inp["Te"], s["a"], s["eta"], trunc)
    t = {k: torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda") for k, v in inp.items()}
    R = torch.tensor(s["R"], dtype=torch.float64, device="cuda")
    tol = 1e-5 if precision == 3 else 1e-8
    for stream in (None, torch.cuda.Stream()):
        torch.cuda.synchronize()
        ctx = gbi.Context(0, stream=stream)
        for restart in (40, 3):      # 3: several cycles
            prm = gbi.params(a=s["a"], eta=s["eta"], trunc=trunc, precision=precision, rtol=1e-10, restart=restart)
            for _ in range(3):       # direct, capture, replay
                got = ctx.solve(prm, R, t["Va"], t["Oa"], t["VH"], t["Fe"], t["Te"])
            ctx.synchronize()
            for x, y in zip(got[:3], ref):
                assert np.abs(x.cpu().numpy() - y).max() <= tol * max(np.abs(y).max(), 1e-6)
        ctx.close()


@pytest.mark.parametrize("N", [511, 512, 513])
def test_two_round_limit(N):
    """FP64 solves on both sides of n = 4096 against the refined mixed solve."""
    import torch
    import paper_1411_0278_gb300 as gbi
    import workloads
    s = workloads.small_cloud(N, 5, phi=0.05, dmin=2.3)
    R = torch.tensor(s["R"], dtype=torch.float64, device="cuda")
    p = torch.tensor(s["p"], dtype=torch.float64, device="cuda")
    ctx = gbi.Context(0)
    i = ctx.trap_inputs(N, 2, s["k"], s["vs"], s["s0"], 0.02, R, p)
    out = []
    for precision in (0, 2):
        prm = gbi.params(a=s["a"], eta=s["eta"], trunc=2, precision=precision, rtol=1e-11)
        out.append(ctx.solve(prm, R, i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"])[:3])
    for x, y in zip(*out):
        assert float((x - y).abs().max()) <= 1e-9 * float(y.abs().max())
    ctx.close()

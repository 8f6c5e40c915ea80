"""Wall images at the edges of the kernel's blocks, tiles and source slices (one sphere, fewer
spheres than a slice, a block and a tile plus one), with torques: sampled spheres against the
oracle, FP64 within 1e-12 and FP32 within 1e-5 of the largest velocity."""
import numpy as np
import pytest

from oracle import dynamics, wall

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
@pytest.mark.parametrize("N", [1, 7, 9, 33, 129, 263])
def test_wall_edges(N, precision, tol):
    import torch
    import paper_1411_0278_gb300 as gbi
    import workloads
    s = workloads.small_cloud(N, 40 + N, phi=0.05, dmin=2.2)
    R = s["R"].copy()
    R[:, 2] += 1.3 - R[:, 2].min()
    prm = dict(a=s["a"], eta=s["eta"], k=s["k"], vs=s["vs"], s0=s["s0"], d0=0.03)
    inp = dynamics.trap_inputs(R, s["p"], prm, 2)
    inp["Te"] = 0.1 * np.random.default_rng(N).normal(size=(N, 3))
    tgt = sorted({0, N // 2, N - 1})
    V_o, O_o = wall.wall_superpose(R, inp["Va"], inp["Oa"], inp["VH"], inp["Fe"], inp["Te"], s["a"], s["eta"],
                                   targets=tgt)
    t = {k: torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda") for k, v in inp.items()}
    ctx = gbi.Context(0)
    p = gbi.params(a=s["a"], eta=s["eta"], trunc=2, precision=precision)
    V, O = ctx.wall_superpose(p, torch.tensor(R, dtype=torch.float64, device="cuda"), t["Va"], t["Oa"], t["VH"],
                              t["Fe"], t["Te"])
    torch.cuda.synchronize()
    for got, ref in ((V, V_o), (O, O_o)):
        assert np.abs(got.cpu().numpy()[tgt] - ref).max() <= tol * max(np.abs(ref).max(), 1e-3)
    ctx.close()

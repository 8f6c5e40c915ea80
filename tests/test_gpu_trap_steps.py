"""Superposition trap steps in FP32 (one block for small suspensions, two kernels a step above)
against FP64 steps of the same call, which run the general sequence.

Tolerance: a step moves R by dt V and turns p by dt Omega; the FP32 pair sums are within 1e-5 of
their largest value (the parity bound of the FP32 kernels), so after a few steps R and p differ by less
than nsteps dt 1e-5 max|V - Va|, max|Omega|, both below 1 here."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# the block form's lanes per target change at powers of two; 72 / 73 is its limit, 512 a target
# block, 2048 / 2049 the change of the split rule, 128 a source tile
SIZES = [1, 2, 3, 8, 31, 64, 72, 73, 129, 511, 513, 2048, 2049]


def suspension(n, seed):
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    R = 4.0 * (g - (m - 1) / 2) + rng.uniform(-0.5, 0.5, size=(n, 3))
    p = rng.normal(size=(n, 3))
    return R, p / np.linalg.norm(p, axis=1, keepdims=True)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("squirmer", [False, True])
def test_steps_against_fp64(n, squirmer):
    import torch
    import paper_1411_0278_gb300 as gbi
    R0, p0 = suspension(n, n)
    out = []
    dt, steps = 0.05, 3
    ctx = gbi.Context(0)
    for precision in (0, 1, 3):
        R = torch.tensor(R0, dtype=torch.float64, device="cuda")
        p = torch.tensor(p0, dtype=torch.float64, device="cuda")
        prm = gbi.params(a=1.0, eta=1 / (6 * math.pi), trunc=2, precision=precision)
        if squirmer:
            info = ctx.squirmer_step(prm, R, p, dt, 0.002, 0.15, -1 / 12, True, steps)
        else:
            info = ctx.trap_step(prm, R, p, dt, 0.002, 0.1, 0.05, 0.0, True, steps)
        torch.cuda.synchronize()
        assert info.pair_interactions == steps * n * (n - 1)
        assert (info.matvecs_f32, info.matvecs_f64) == ((0, steps) if precision == 0 else (steps, 0))
        out.append((R.cpu().numpy(), p.cpu().numpy()))
    tol = steps * dt * 1e-5
    for R, p in out[1:]:
        assert np.abs(R - out[0][0]).max() < tol and np.abs(p - out[0][1]).max() < tol
        assert np.abs(np.linalg.norm(p, axis=1) - 1).max() < 1e-14
    ctx.close()


def test_steps_in_one_call_or_many():
    """The state between calls is all there is: 7 steps in one call and in seven are the same."""
    import torch
    import paper_1411_0278_gb300 as gbi
    ctx = gbi.Context(0)
    prm = gbi.params(a=1.0, eta=0.3, trunc=2, precision=1)
    for n in (5, 200):
        R0, p0 = suspension(n, 3)
        got = []
        for calls in (1, 7):
            R = torch.tensor(R0, dtype=torch.float64, device="cuda")
            p = torch.tensor(p0, dtype=torch.float64, device="cuda")
            for _ in range(calls):
                ctx.trap_step(prm, R, p, 0.05, 0.002, 0.1, 0.05, 0.01, True, 7 // calls)
            got.append(torch.cat([R, p]).cpu())
        assert torch.equal(*got)
    ctx.close()

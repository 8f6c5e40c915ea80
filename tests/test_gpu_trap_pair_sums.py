"""The pair sums of the superposition trap steps in FP32 (one block up to 72 spheres, two kernels a step
above), isolated from the one-body motion, at spacings down to 2.1 radii and with strong modes.

One step with dt = 1: R1 - R0 - (vs p + mt F) is the pair velocity to FP64 rounding; p1 is compared with the
normalised p + Omega x p, whose error is at most that of Omega."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# 72 / 73: one block or two kernels; 2048 / 2049: narrow or wide pair blocks; 128: a source tile; 64 and 128: a
# second split of a target's sources
SIZES = [1, 2, 3, 8, 64, 65, 72, 73, 127, 129, 511, 513, 2048, 2049]


def suspension(n, seed):
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    R = 2.3 * (g - (m - 1) / 2) + rng.uniform(-0.1, 0.1, size=(n, 3))
    p = rng.normal(size=(n, 3))
    return R, p / np.linalg.norm(p, axis=1, keepdims=True)


def dev(x):
    import torch
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def one_step(ctx, gbi, R0, p0, eta, k, vs, s0, d0, precision):
    """R1, p1 of one step, and what the general kernels' V and Omega in FP32 and FP64 make of it."""
    prm = gbi.params(a=1.0, eta=eta, trunc=2, precision=precision)
    R, p = dev(R0), dev(p0)
    ctx.trap_step(prm, R, p, 1.0, k, vs, s0, d0, True, 1)
    out = [(R.cpu().numpy(), p.cpu().numpy())]
    R, p = dev(R0), dev(p0)
    i = ctx.trap_inputs(len(R0), 2, k, vs, s0, d0, R, p)
    one = vs * p0 + (-k * R0) / (6 * math.pi * eta)
    scale = None
    for precision in (1, 0):
        V, Om = (t.cpu().numpy() for t in ctx.superpose(gbi.params(a=1.0, eta=eta, trunc=2, precision=precision), R,
                                                         i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"]))
        q = p0 + np.cross(Om, p0)
        out.append((R0 + V, q / np.linalg.norm(q, axis=1, keepdims=True)))
        scale = np.abs(V - one).max(), np.abs(Om).max()
    return out, scale


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("d0", [0.0, 0.3])
@pytest.mark.parametrize("precision", [1, 3])
def test_pair_sums(n, d0, precision):
    """Against FP64: 1e-5 of the largest pair velocity and angular velocity (the parity bound of the
    FP32 kernels) and FP64 rounding of R1 and p1.  Against the general FP32 kernels, whose terms and order
    of summation these are: rounding of the FP64 update alone, some six of 2^-53 of the largest |R1|, |V| each
    (2e-15 of them), and as much of the unit vector p1 with the normalisation's (4e-15)."""
    import paper_1411_0278_gb300 as gbi
    R0, p0 = suspension(n, n)
    ctx = gbi.Context(0)
    (got, f32, f64), (dv, dw) = one_step(ctx, gbi, R0, p0, 0.07, 0.05, 0.1, 0.4, d0, precision)
    ctx.close()
    ulp = 2e-15 * max(np.abs(R0).max(), np.abs(f64[0] - R0).max())
    assert np.abs(got[0] - f64[0]).max() <= 1e-5 * dv + ulp
    assert np.abs(got[1] - f64[1]).max() <= 1e-5 * dw + 4e-15
    assert np.abs(got[0] - f32[0]).max() <= ulp
    assert np.abs(got[1] - f32[1]).max() <= 4e-15


@pytest.mark.parametrize("n", [2, 72, 73])
def test_profiled_steps_are_the_same(n):
    """Profiling times the kernels of an ordinary call: the same bits, launches and steps."""
    import torch
    import paper_1411_0278_gb300 as gbi
    ctx = gbi.Context(0)
    prm = gbi.params(a=1.0, eta=0.07, trunc=2, precision=1)
    got, launches = [], []
    steps = 5
    for prof in (False, True):
        ctx.set_profiling(prof)
        R, p = (dev(x) for x in suspension(n, 4))
        before = ctx.kernel_launches()
        ctx.trap_step(prm, R, p, 0.01, 0.05, 0.1, 0.4, 0.0, True, steps)
        launches.append(ctx.kernel_launches() - before)
        got.append(torch.cat([R, p]).cpu())
    st = ctx.kernel_stats(gbi._native.TRAP_F32)
    ctx.set_profiling(False)
    assert torch.equal(*got) and launches[0] == launches[1]
    assert st["launches"] == (1 if n <= 72 else steps)
    assert st["flops"] == pytest.approx(103.0 * n * (n - 1) * steps, rel=1e-12)
    ctx.close()

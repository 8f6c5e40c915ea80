"""Rounding of the FP64 superposition sums against extended precision (numpy's long double: 64 bits of
significand or more on the machines used).

Bound: with 64 sources per split and the splits added in order, the form before sources were split finer, the rms
error over all spheres of these suspensions measured 0.82e-16 and 0.84e-16 of the largest velocity; 400 of the
1500 spheres are sampled here (their rms is known to some 3%), so 0.95e-16 is asked.  Angular velocities: 0.70e-16
of the largest, 0.80e-16 is asked."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = np.longdouble


def reference(R, p, T, targets, eta, k, vs, s0):
    """V and Omega of the targets: forces -k R, torques T, V^(2s) = s0 (pp - I/3), a = 1."""
    pi = L("3.14159265358979323846264338327950288")
    R, p, T, eta = R.astype(L), p.astype(L), T.astype(L), L(eta)
    F = -L(k) * R
    S = -(L(5) / 6) * L(s0) * (p[:, :, None] * p[:, None, :] - np.eye(3, dtype=L) / 3)
    F8, T8 = F / (8 * pi * eta), T / (8 * pi * eta)
    V, Om = [], []
    for t in targets:
        x = R[t] - R
        r2 = (x * x).sum(1)
        r2[t] = L("inf")
        r1 = 1 / np.sqrt(r2)
        r3 = r1 ** 3
        r5, r7 = r3 * r1 ** 2, r3 * r1 ** 4
        Sx = (S * x[:, None, :]).sum(2)
        cx = (r3 - 2 * r5) * (x * F8).sum(1) + (8 * r7 - 3 * r5) * (x * Sx).sum(1)
        v = (r1 + L(2) / 3 * r3)[:, None] * F8 + cx[:, None] * x + r3[:, None] * np.cross(T8, x) - (L(16) / 5 * r5)[:, None] * Sx
        w = r3[:, None] * np.cross(F8, x) + (L(3) / 2 * (x * T8).sum(1) * r5)[:, None] * x - (r3 / 2)[:, None] * T8
        w = w + (3 * r5)[:, None] * np.cross(x, Sx)
        V.append(L(vs) * p[t] + F[t] / (6 * pi * eta) + v.sum(0))
        Om.append(T[t] / (8 * pi * eta) + w.sum(0))
    return np.array(V), np.array(Om)


@pytest.mark.parametrize("seed", [1, 2])
def test_superposition_rounding(seed):
    import torch
    import paper_1411_0278_gb300 as gbi
    n, eta, k, vs, s0 = 1500, 1 / (6 * math.pi), 0.01, 0.1, 0.05
    rng = np.random.default_rng(seed)
    side = (n * 4 * math.pi / 3 / 0.02) ** (1 / 3)
    m = int(np.ceil(n ** (1 / 3)))
    g = (np.arange(m) + 0.5) * side / m - side / 2
    R = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)[rng.choice(m ** 3, size=n, replace=False)]
    R = R + rng.uniform(-1, 1, size=(n, 3)) * (side / m - 2.1) / 2 / math.sqrt(3)
    R[:, 2] += 2.0 - R[:, 2].min()
    p = rng.normal(size=(n, 3))
    p /= np.linalg.norm(p, axis=1, keepdims=True)
    T = 0.02 * rng.normal(size=(n, 3))
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")
    ctx = gbi.Context(0)
    i = ctx.trap_inputs(n, 2, k, vs, s0, 0.0, dev(R), dev(p))
    got = ctx.superpose(gbi.params(a=1.0, eta=eta, trunc=2, precision=0), dev(R), i["Va"], i["Oa"], i["VH"], i["Fe"], dev(T))
    got = [t.cpu().numpy() for t in got]
    ctx.close()
    targets = rng.choice(n, size=400, replace=False)
    for x, ref, bound in zip(got, reference(R, p, T, targets, eta, k, vs, s0), (0.95e-16, 0.80e-16)):
        err = (x[targets] - ref).astype(float)
        assert math.sqrt((err ** 2).mean()) <= bound * np.abs(x).max()

"""Neighbour search of one large system far from the origin, with pairs whose separation along one axis is
the last FP64 number below the cut-off (the case in which rounded cell numbers could part them)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [0, 31, 34, 37, 41, 45, 49])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_pairs_at_the_cutoff(exponent, sign):
    import torch
    import paper_1411_0278_gb300 as gbi
    rc, n = 4.0, 2500
    rng = np.random.default_rng(exponent)
    base = sign * 2.0 ** exponent * np.array([1.0, 1.5, -1.25])
    grid = np.stack(np.meshgrid(*[np.arange(14.0)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    # 24 radii between the pairs; the fraction of a cell is arbitrary as far as FP64 resolves it
    first = base + 24.0 * grid + rng.uniform(0.0, 4.0, size=(n, 3))
    axis = rng.integers(0, 3, size=n)
    second = first.copy()
    ulp = np.maximum(np.spacing(np.abs(first[np.arange(n), axis])), np.spacing(np.abs(first[np.arange(n), axis]) + rc))
    step = np.where(ulp < rc, (np.ceil(rc / ulp) - 1.0) * ulp, 0.0)
    second[np.arange(n), axis] += step
    R = np.concatenate([first, second])
    d = R[n:] - R[:n]
    close = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2] < rc * rc
    assert close.mean() > 0.9
    ctx = gbi.Context(0)
    tg, sr = ctx.pairs(torch.tensor(R, dtype=torch.float64, device="cuda"), 1.0, rc)
    torch.cuda.synchronize()
    got = set(zip(tg.cpu().tolist(), sr.cpu().tolist()))
    ctx.close()
    k = np.flatnonzero(close)
    assert got == set(zip(k, k + n)) | set(zip(k + n, k))

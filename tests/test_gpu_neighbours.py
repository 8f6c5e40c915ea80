"""Neighbour lists of every search form against the definition, (dx dx + dy dy) + dz dz < (rcut a)^2
evaluated in FP64 pair by pair: whole numbers, so they are equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def brute(R, rc, offsets=None):
    n = len(R)
    sys = np.zeros(n, dtype=np.int64) if offsets is None else np.repeat(np.arange(len(offsets) - 1), np.diff(offsets))
    tg, sr = [], []
    for b in range(0, n, 512):
        d = R[b:b + 512, None] - R[None]
        d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
        ok = (d2 < rc * rc) & (sys[b:b + 512, None] == sys[None])
        i, j = np.nonzero(ok)
        keep = i + b != j
        tg.append(i[keep] + b)
        sr.append(j[keep])
    return np.concatenate(tg), np.concatenate(sr)


def lattice(n, sp, rng, jitter):
    m = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    return sp * g + jitter * rng.uniform(-1, 1, size=(n, 3))


# n: the scan by warps (33, 4096) and the bucket search from its smallest size, with and without
# more cells than buckets; spacing 2 puts thousands of pairs exactly at the cut-off of 4 a
@pytest.mark.parametrize("n,sp,jitter,shift", [(1, 2.0, 0.0, 0.0), (33, 2.0, 0.0, 0.0), (4096, 3.4, 0.5, 0.0),
                                               (4097, 2.0, 0.0, 0.0), (5000, 3.4, 0.5, 3.0e5), (6007, 9.0, 4.0, 0.0),
                                               (5000, 3.4, 0.5, -1.0e9), (9001, 2.2, 0.1, 17.0)])
def test_single_system(ctx, n, sp, jitter, shift):
    import torch
    rng = np.random.default_rng(n)
    R = lattice(n, sp, rng, jitter) + shift
    if sp == 9.0:
        R[:, 0] *= 40.0   # a long box: far more cells than buckets along x
    R = R[rng.permutation(n)]
    for a, rcut in ((1.0, 4.0), (0.5, 5.0)):
        tg, sr = ctx.pairs(torch.tensor(R, device="cuda"), a, rcut)
        t, s = brute(R, rcut * a)
        assert np.array_equal(tg.cpu().numpy(), t) and np.array_equal(sr.cpu().numpy(), s)


@pytest.mark.parametrize("sizes", [(2, 3, 2), (40, 1, 7, 300), (16, 16), (4097, 5)])
def test_batch(ctx, sizes):
    import torch
    rng = np.random.default_rng(len(sizes))
    R = np.concatenate([lattice(k, 2.0, rng, 0.3) for k in sizes])
    offs = [0] + list(np.cumsum(sizes))
    tg, sr = ctx.pairs(torch.tensor(R, device="cuda"), 1.0, 4.0, offs)
    t, s = brute(R, 4.0, offs)
    assert np.array_equal(tg.cpu().numpy(), t) and np.array_equal(sr.cpu().numpy(), s)


def test_crowded_spheres(ctx):
    """More than 64 neighbours: an error in the bucket search, a longer list below its size."""
    import torch
    import paper_1411_0278_gb300 as gbi
    rng = np.random.default_rng(3)
    R = lattice(4097, 5.0, rng, 0.0)
    R[:80] = rng.uniform(0, 1, size=(80, 3))
    with pytest.raises(gbi.GbiError) as e:
        ctx.pairs(torch.tensor(R, device="cuda"), 1.0, 4.0)
    assert e.value.status == gbi.GBI_ERR_ARG
    tg, sr = ctx.pairs(torch.tensor(R[:300], device="cuda"), 1.0, 4.0)
    t, s = brute(R[:300], 4.0)
    assert np.array_equal(tg.cpu().numpy(), t) and np.array_equal(sr.cpu().numpy(), s)


@pytest.fixture(scope="module")
def ctx():
    import paper_1411_0278_gb300 as gbi
    c = gbi.Context(0)
    yield c
    c.close()

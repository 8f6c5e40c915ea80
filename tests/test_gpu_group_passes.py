"""Batches large enough for the grouped pair passes and the warp-per-system Arnoldi step in their
solves (1600 spheres and more, systems of at most 17, at l <= 3 of at most 9), and one sphere below: against the
streaming kernels (a forced choice) and an independent smallest distance.

Tolerances: both solves meet a residual of 1e-10 and the system's condition number is below ~10: 1e-8 of the
largest component, 1e-5 where the outputs are FP32 sums (precision 3).  The smallest squared distance is
an FP32 number formed from differences exact to 2^-24: 1e-6."""
import numpy as np
import pytest

from test_gpu_small_systems import close, dev, systems

pytestmark = pytest.mark.gpu

# (trunc, sizes): groups of 1, 2, 4, 8, 16 lanes; systems above 256 vector elements (no warp per system):
# l <= 4 from 6 spheres; 1599 spheres
CASES = [(2, [17, 16, 1] * 50), (2, [2, 1] * 534), (2, [17] * 94 + [1]), (3, [9, 4, 2] * 110), (3, [3, 3, 2] * 200),
         (4, [5, 2, 1] * 200), (4, [17, 3] * 80), (4, [9, 8] * 95)]


@pytest.fixture(autouse=True)
def stream():
    import torch
    with torch.cuda.stream(torch.cuda.Stream()):
        yield


def _case(trunc, sizes):
    import torch
    import paper_1411_0278_gb300 as gbi
    R, p, offs = systems(sizes, trunc)
    ctx = gbi.Context(0, stream=torch.cuda.current_stream())
    R, p = dev(R), dev(p)
    i = ctx.trap_inputs(len(R), trunc, 0.01, 0.1, 0.05, 0.02, R, p)
    return gbi, ctx, R, offs, (i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"])


def _closest(R, offs):
    R, best = R.cpu().numpy(), np.inf
    for b, e in zip(offs[:-1], offs[1:]):
        if e - b > 1:
            d = np.linalg.norm(R[b:e, None] - R[None, b:e], axis=-1)
            best = min(best, d[np.triu_indices(e - b, 1)].min())
    return best


@pytest.mark.parametrize("trunc,sizes", CASES)
@pytest.mark.parametrize("precision", [1, 2, 3])
def test_solves_and_smallest_distance(trunc, sizes, precision):
    import torch
    gbi, ctx, R, offs, a = _case(trunc, sizes)
    prm = gbi.params(a=1.0, eta=0.7, trunc=trunc, precision=precision, rtol=1e-10, max_iter=4000)
    ctx.set_wpt(4)
    ref = ctx.batch_solve(prm, offs, R, *a)[:3]
    ctx.set_wpt(0)
    for _ in range(3):       # direct launches, graph capture, replay
        V, Om, Q, info, _ = ctx.batch_solve(prm, offs, R, *a)
        assert abs(info.min_separation / _closest(R, offs) - 1) < 1e-6
    torch.cuda.current_stream().synchronize()
    for x, y in zip((V, Om, Q), ref):
        close(x, y, 1e-8 if precision < 3 else 1e-5)
    ctx.close()


@pytest.mark.parametrize("trunc,sizes", [(2, [17, 16, 1] * 50), (4, [5, 2, 1] * 200)])
@pytest.mark.parametrize("precision", [1, 2])
def test_overlap_guard(trunc, sizes, precision):
    gbi, ctx, R, offs, a = _case(trunc, sizes)
    d = _closest(R, offs)
    ctx.batch_solve(gbi.params(a=1.0, eta=0.7, trunc=trunc, precision=precision, min_sep=d * 0.9999), offs, R, *a)
    for _ in range(3):
        with pytest.raises(gbi.GbiError):
            ctx.batch_solve(gbi.params(a=1.0, eta=0.7, trunc=trunc, precision=precision, min_sep=d * 1.0001), offs, R, *a)
    ctx.close()


@pytest.mark.parametrize("trunc,sizes", [(2, [17, 16, 1] * 50), (3, [3, 3, 2] * 200), (4, [5, 2, 1] * 200), (4, [17, 3] * 80)])
@pytest.mark.parametrize("precision", [1, 2, 3])
def test_warm_start(trunc, sizes, precision):
    """From a guess with every coefficient off by up to a tenth, and from the solution itself."""
    import torch
    gbi, ctx, R, offs, a = _case(trunc, sizes)
    prm = gbi.params(a=1.0, eta=0.7, trunc=trunc, precision=precision, rtol=1e-10, max_iter=4000)
    ref = ctx.batch_solve(prm, offs, R, *a)[:3]
    torch.manual_seed(3)
    for scale in (0.1, 0.0):
        guess = ref[2] * (1.0 + scale * torch.rand_like(ref[2]))
        for _ in range(3):
            got = ctx.batch_solve(prm, offs, R, *a, QH=guess.clone(), warm_start=True)
            assert got[3].rel_residual <= 1e-10
            for x, y in zip(got[:3], ref):
                close(x, y, 1e-8 if precision < 3 else 1e-5)
    ctx.close()


def test_tuned_choice_is_kept():
    """What gbi_tune chose for a batch's passes serves every later batch of that size class: the pass
    gives the bits of the same choice forced (sums of 16 sources in another order differ)."""
    gbi, ctx, R, offs, a = _case(2, [17] * 130)
    prm = gbi.params(a=1.0, eta=0.7, trunc=2, precision=1)
    chosen = ctx.tune(2, [130 * k for k in range(18)], reps=2)   # 17 systems of 130: streaming forms only
    assert all(w in (2, 4, 8, 16) for w in chosen)
    assert ctx.pass_wpt(2, 1, 0, 1, offs[-1], batched=True) == chosen[5]
    got = ctx.batch_superpose(prm, offs, R, *a)
    ctx.set_wpt(chosen[5])
    for x, y in zip(got, ctx.batch_superpose(prm, offs, R, *a)):
        assert bool((x == y).all())
    ctx.close()


@pytest.mark.parametrize("trunc,sizes", [(2, [17] * 130), (4, [3, 2] * 400), (4, [17, 20] * 10)])
def test_tuning_a_batch_of_small_systems(trunc, sizes):
    """The grouped form is a candidate, reported as 32 and kept; results stay."""
    gbi, ctx, R, offs, a = _case(trunc, sizes)
    prm = gbi.params(a=1.0, eta=0.7, trunc=trunc, precision=2, rtol=1e-10)
    ref = ctx.batch_solve(prm, offs, R, *a)[:3]
    chosen = ctx.tune(trunc, offs, reps=2)
    assert all(w in (2, 4, 8, 16, 32) for w in chosen)
    passes = [(2, 2, 1), (2, 2, 2), (2, 1, 2), (1, 0, 2), (2, 1, 1), (1, 0, 1)]
    for (rows, cols, precision), w in zip(passes, chosen):
        assert ctx.pass_wpt(trunc, rows, cols, precision, offs[-1], batched=True) == w
    for _ in range(3):
        got = ctx.batch_solve(prm, offs, R, *a)[:3]
    for x, y in zip(got, ref):
        close(x, y, 1e-8)
    ctx.close()


def test_layout_follows_the_choice():
    """A forced warps-per-target choice between calls changes kernels and vector layouts together."""
    gbi, ctx, R, offs, a = _case(3, [2, 3] * 400)
    prm = gbi.params(a=1.0, eta=0.7, trunc=3, precision=2, rtol=1e-10)
    first = None
    for w in (0, 0, 4, 4, 0, 8, 0):
        ctx.set_wpt(w)
        got = ctx.batch_solve(prm, offs, R, *a)[:3]
        first = first or got
        for x, y in zip(got, first):
            close(x, y, 1e-8)
    ctx.close()

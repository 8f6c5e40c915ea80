"""The calls that users of this framework make, as measurable cases.

Each case goes through the Python binding of the C ABI (``paper_1411_0278_gb300.Context``) the
way the programs of this repository call it: superposition dynamics of a few squirmers and of a
large cloud in a trap, one step of the fully coupled dynamics, refined and FP64 Galerkin solves,
a batch of suspensions of uneven size, label generation and a training gradient of the near-field
network, its evaluation in a large suspension, the periodic and wall Green's functions and the
flow field.  Sizes are those of the workloads and the benchmark of this repository; ``draw``
spreads them over the ranges those stand for.

``exact`` states each result in 64 bits from the definitions alone: the pair elements from the
derivatives of r and 1/r (a recursion over the derivative order), the linear system by conjugate
gradients on those elements, Ewald sums, forward-mode derivatives of the wall's Green's function
and the network in torch.
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_1411_0278_gb300 as gbi

A = 1.0                                # sphere radius of every workload
ETA = 1.0 / (6.0 * math.pi)            # viscosity: unit Stokes mobility at a = 1
K_TRAP, VS, S0 = 0.01, 0.1, 0.05       # trap stiffness, self-propulsion, strain mode of the workloads
B1, B2 = 0.15, -1.0 / 12.0             # squirmer slip of the two-squirmer orbits
R_ORBIT = 12.56                        # their orbit radius
R_CLOUD = 1256.6                       # radius of the 10^4-squirmer trap

_stream = None


def listed():
    return [
        # two squirmers orbiting in a trap, 50 Euler steps between samples: the smallest call,
        # bound by launches and latency
        {"name": "orbit_n2", "kind": "orbit", "n": 2, "steps": 50},
        # 10^4 squirmers on the trap radius, FP32 superposition: a few steps of a long trajectory
        {"name": "cloud_n10000", "kind": "cloud", "n": 10000, "steps": 4},
        # the benchmark's headline: one step (inputs, refined l <= 3 solve, Euler update)
        {"name": "step_mixed_l3_n1024", "kind": "step", "n": 1024, "trunc": 3},
        # the plain solve at the highest mixed truncation, every output kept to 1e-10 (a
        # reference for the learned correction); a size that fills no power of two
        {"name": "solve_mixed_l4_n1000", "kind": "solve", "n": 1000, "trunc": 4, "precision": 2},
        # the plain FP64 method on the smallest workload
        {"name": "solve_f64_l2_n64", "kind": "solve", "n": 64, "trunc": 2, "precision": 0},
        # independent suspensions of uneven size in one lock-step solve
        {"name": "batch_l2_48", "kind": "batch", "systems": 48, "largest": 1024},
        # two- and three-sphere systems solved at l <= 4: labels of the near-field network
        {"name": "labels_l4_4000", "kind": "labels", "systems": 4000},
        # one minibatch of the network's training: pairs, features, forward, loss, backward
        {"name": "gradient_1024", "kind": "gradient", "systems": 1024},
        # the network's correction of a large dense suspension
        {"name": "nearfield_n100000", "kind": "nearfield", "n": 100000},
        # point forces in a periodic cube, the plan left to the library
        {"name": "periodic_n100000", "kind": "periodic", "n": 100000},
        # the flow on a grid of points through a solved suspension
        {"name": "flow_l3_n1024", "kind": "flow", "n": 1024, "trunc": 3, "points": 262144},
        # swimmers above a no-slip wall, evaluated in FP64
        {"name": "wall_f64_n1500", "kind": "wall", "n": 1500},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["orbit", "cloud", "step", "solve", "solve", "batch", "labels", "gradient", "nearfield",
                       "periodic", "flow", "wall"])
    if kind == "orbit":
        return {"kind": kind, "n": log(2, 64), "steps": rng.choice([20, 50])}
    if kind == "cloud":
        return {"kind": kind, "n": log(100, 10000), "steps": rng.randint(1, 4)}
    if kind == "step":
        return {"kind": kind, "n": log(100, 1100), "trunc": rng.choice([2, 3])}
    if kind == "solve":
        if rng.random() < 0.4:
            return {"kind": kind, "n": log(8, 200), "trunc": rng.choice([2, 3]), "precision": 0}
        return {"kind": kind, "n": log(60, 1000), "trunc": rng.choice([2, 3, 4]), "precision": 2}
    if kind == "batch":
        return {"kind": kind, "systems": log(3, 48), "largest": log(100, 1024)}
    if kind == "labels":
        return {"kind": kind, "systems": log(100, 4000)}
    if kind == "gradient":
        return {"kind": kind, "systems": log(60, 4000)}
    if kind == "nearfield":
        return {"kind": kind, "n": log(1000, 100000)}
    if kind == "periodic":
        return {"kind": kind, "n": log(2000, 100000)}
    if kind == "flow":
        return {"kind": kind, "n": log(30, 1024), "trunc": rng.choice([2, 3]), "points": log(500, 200000)}
    return {"kind": kind, "n": log(50, 1500)}


# ------------------------------------------------------------------------------------ inputs


def _unit(rng, n):
    v = rng.normal(size=(n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _lattice(rng, n, phi, dmin):
    """n centres at volume fraction phi, no two closer than dmin: sites of a cubic lattice, jittered."""
    side = (n * 4.0 * math.pi * A ** 3 / 3.0 / phi) ** (1.0 / 3.0)
    m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    sp = side / m
    g = (np.arange(m) + 0.5) * sp - side / 2
    sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    sel = rng.choice(len(sites), size=n, replace=False)
    return sites[sel] + rng.uniform(-1.0, 1.0, size=(n, 3)) * (max(0.0, sp - dmin) / 2.0 / math.sqrt(3.0)), side


def _small_systems(rng, count):
    """count systems of two or three spheres, each sphere within [2.05 a, 4 a) of an earlier one
    and none closer than 2.05 a; two-sphere systems first."""
    n3 = count // 2
    n2 = count - n3
    r0 = rng.uniform(-5.0, 5.0, size=(count, 3))
    r1 = r0 + rng.uniform(2.05, 4.0, size=(count, 1)) * _unit(rng, count)
    r2 = np.full((n3, 3), np.nan)
    todo = np.arange(n3)
    while len(todo):
        base = np.where(rng.random(len(todo))[:, None] < 0.5, r0[n2 + todo], r1[n2 + todo])
        q = base + rng.uniform(2.05, 4.0, size=(len(todo), 1)) * _unit(rng, len(todo))
        ok = np.minimum(np.linalg.norm(q - r0[n2 + todo], axis=1), np.linalg.norm(q - r1[n2 + todo], axis=1)) >= 2.05
        r2[todo[ok]] = q[ok]
        todo = todo[~ok]
    two = np.stack([r0[:n2], r1[:n2]], 1).reshape(-1, 3)
    three = np.stack([r0[n2:], r1[n2:], r2], 1).reshape(-1, 3)
    offs = [2 * i for i in range(n2 + 1)] + [2 * n2 + 3 * i for i in range(1, n3 + 1)]
    return np.concatenate([two, three]), offs


def _theta(rng):
    """Network weights in the flat layout of gbi_mlp_set: uniform in the Glorot range, small biases."""
    parts = []
    for fo, fi in ((128, 9), (128, 128), (128, 128), (6, 128)):
        lim = math.sqrt(6.0 / (fi + fo))
        parts += [rng.uniform(-lim, lim, size=fo * fi), rng.uniform(-0.1, 0.1, size=fo)]
    return np.concatenate(parts).astype(np.float32)


def _raw(case, seed):
    """The seeded inputs of a case as numpy arrays."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("orbit", "cloud"):
        n = case["n"]
        if kind == "orbit":
            # evenly spread directions (a golden-angle spiral) turned at random
            i = np.arange(n) + 0.5
            z, phi = 1.0 - 2.0 * i / n, math.pi * (1.0 + math.sqrt(5.0)) * i
            s = np.sqrt(1.0 - z * z)
            u = np.stack([s * np.cos(phi), s * np.sin(phi), z], 1) + 0.05 * rng.normal(size=(n, 3))
            u = u @ np.linalg.qr(rng.normal(size=(3, 3)))[0]
            u /= np.linalg.norm(u, axis=1, keepdims=True)
            return dict(R=u * R_ORBIT * math.sqrt(n / 2.0), p=u.copy())
        u = _unit(rng, n)
        return dict(R=R_CLOUD * u, p=u.copy())
    if kind in ("step", "solve"):
        R, _ = _lattice(rng, case["n"], 0.05, 2.5)
        return dict(R=R, p=_unit(rng, case["n"]))
    if kind == "batch":
        # log-uniform sizes in [32, largest], the same for every seed (a layout that a program keeps)
        lay = np.random.default_rng(case["systems"])
        lo = math.log(min(32, case["largest"]))
        ns = np.round(np.exp(lay.uniform(lo, math.log(case["largest"]), case["systems"]))).astype(int)
        ns[0] = case["largest"]
        R = [_lattice(rng, int(n), rng.uniform(0.01, 0.15), 2.5)[0] for n in ns]
        return dict(R=np.concatenate(R), p=_unit(rng, int(ns.sum())), offsets=[0] + [int(v) for v in np.cumsum(ns)])
    if kind in ("labels", "gradient"):
        R, offs = _small_systems(rng, case["systems"])
        d = dict(R=R, p=_unit(rng, len(R)), offsets=offs)
        if kind == "gradient":
            d.update(theta=_theta(rng), labels=rng.normal(size=(len(R), 6)))
        return d
    if kind == "nearfield":
        n = case["n"]
        R, _ = _lattice(rng, n, 0.1, 2.05)
        p = _unit(rng, n)
        return dict(R=R, p=p, theta=_theta(rng), V=VS * p + 0.01 * rng.normal(size=(n, 3)),
                    Om=0.01 * rng.normal(size=(n, 3)))
    if kind == "periodic":
        n = case["n"]
        L = (n * 4.0 * math.pi / 3.0 / 0.1) ** (1.0 / 3.0)
        return dict(R=rng.uniform(0.0, L, size=(n, 3)), F=0.1 * rng.normal(size=(n, 3)), Va=VS * _unit(rng, n), L=L)
    if kind == "flow":
        n, t = case["n"], case["trunc"]
        R, side = _lattice(rng, n, 0.05, 2.5)
        p = _unit(rng, n)
        # coefficients of a trapped active suspension: one-body values with every mode excited
        QH = np.concatenate([0.3 * rng.normal(size=(n, k)) / (1 + j) for j, k in enumerate(_ranks(t))], 1)
        X = rng.uniform(-side / 2, side / 2, size=(case["points"], 3))
        return dict(R=R, p=p, QH=QH, X=X, Fe=-K_TRAP * R, Te=0.05 * rng.normal(size=(n, 3)))
    n = case["n"]
    R, _ = _lattice(rng, n, 0.02, 2.1)
    R[:, 2] += 2.0 * A - R[:, 2].min()
    return dict(R=R, p=_unit(rng, n), Te=0.02 * rng.normal(size=(n, 3)))


def prepare(case, seed):
    global _stream
    if _stream is None:
        # a user's stream (the library replays repeated solves as graphs on one)
        _stream = torch.cuda.Stream()
        torch.cuda.set_stream(_stream)
    dev = torch.device("cuda")
    raw = _raw(case, seed)
    s = {k: torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)
         for k, v in raw.items() if isinstance(v, np.ndarray) and k != "theta"}
    s.update({k: v for k, v in raw.items() if not isinstance(v, np.ndarray)})
    kind = case["kind"]
    s["case"] = case
    s["ctx"] = ctx = gbi.Context(0, stream=_stream)
    n = len(raw["R"])
    if kind in ("orbit", "cloud"):
        s["prm"] = gbi.params(a=A, eta=ETA, trunc=2, precision=1)
    elif kind == "step":
        s["prm"] = gbi.params(a=A, eta=ETA, trunc=case["trunc"], precision=3, rtol=1e-10, restart=40,
                              inner_rtol=1e-5, min_sep=2.0)
        ctx.tune(case["trunc"], [0, n])
        s["R1"], s["p1"] = torch.empty_like(s["R"]), torch.empty_like(s["p"])
    elif kind in ("solve", "batch", "labels"):
        trunc = {"batch": 2, "labels": 4}.get(kind) or case["trunc"]
        s["prm"] = gbi.params(a=A, eta=ETA, trunc=trunc, precision=case.get("precision", 2), rtol=1e-10, restart=40,
                              max_iter=4000, inner_rtol=1e-5)
        s["inp"] = ctx.trap_inputs(n, trunc, 0.0 if kind == "labels" else K_TRAP, VS, S0, 0.0, s["R"], s["p"])
    elif kind in ("gradient", "nearfield"):
        ctx.mlp_set(raw["theta"], 2.0)
    elif kind == "periodic":
        s["prm"] = gbi.params(a=A, eta=ETA, trunc=2, precision=1)
    elif kind == "flow":
        s["prm"] = gbi.params(a=A, eta=ETA, trunc=case["trunc"], precision=1)
    else:
        s["prm"] = gbi.params(a=A, eta=ETA, trunc=2, precision=0)
        s["inp"] = ctx.trap_inputs(n, 2, K_TRAP, VS, S0, 0.02, s["R"], s["p"])
        s["inp"]["Te"] = s["Te"]
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "orbit":
        ctx.squirmer_step(s["prm"], s["R"], s["p"], 0.5, _k_orbit(), B1, B2, True, case["steps"])
        return [s["R"], s["p"]]
    if kind == "cloud":
        ctx.trap_step(s["prm"], s["R"], s["p"], 0.05, _k_cloud(), VS, S0, 0.0, True, case["steps"])
        return [s["R"], s["p"]]
    if kind == "step":
        # a step from a stored configuration (repeated steps would run into contacts, which
        # the trap model does not resolve)
        s["R1"].copy_(s["R"])
        s["p1"].copy_(s["p"])
        ctx.trap_step(s["prm"], s["R1"], s["p1"], 0.1, K_TRAP, VS, S0, 0.0, False, 1)
        return [s["R1"], s["p1"]]
    if kind == "solve":
        i = s["inp"]
        return list(ctx.solve(s["prm"], s["R"], i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"])[:3])
    if kind in ("batch", "labels"):
        i = s["inp"]
        return list(ctx.batch_solve(s["prm"], s["offsets"], s["R"], i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"])[:3])
    if kind == "gradient":
        return list(ctx.mlp_loss_grad(s["R"], s["p"], A, s["labels"], s["offsets"]))
    if kind == "nearfield":
        V, Om = s["V"].clone(), s["Om"].clone()
        n = ctx.mlp_correct(s["R"], s["p"], A, S0, V, Om)
        return [V, Om, n]
    if kind == "periodic":
        return [ctx.periodic_superpose(s["prm"], s["L"], s["R"], s["Va"], s["F"])[0]]
    if kind == "flow":
        U, inside = ctx.flow(s["prm"], s["R"], s["Fe"], s["Te"], s["QH"], s["X"])
        return [U, inside]
    i = s["inp"]
    return list(ctx.wall_superpose(s["prm"], s["R"], i["Va"], i["Oa"], i["VH"], i["Fe"], i["Te"]))


def _k_orbit():
    return 6 * math.pi * ETA * (2 * B1 / 3) / R_ORBIT


def _k_cloud():
    return 6 * math.pi * ETA * VS / R_CLOUD


def work(case):
    """Arithmetic per ordered pair from the closed forms (superposition without torques and
    dipoles; the pair elements in the pair frame), network products, mesh sums."""
    kind = case["kind"]
    hh = {2: 273.0, 3: 894.0, 4: 2013.0}
    h = {2: 8, 3: 25, 4: 48}
    if kind in ("orbit", "cloud"):
        n, st = case["n"], case["steps"]
        return {"bytes": 96.0 * n * st, "flops": 130.0 * n * (n - 1) * st}
    if kind in ("step", "solve"):
        n, t = case["n"], case["trunc"]
        return {"bytes": 8.0 * n * (18 + 2 * h[t]), "flops": 16 * hh[t] * n * (n - 1)}
    if kind == "batch":
        hi = case["largest"]
        pairs = case["systems"] * (hi * hi - 32.0 * 32.0) / 2 / math.log(hi / 32.0)
        return {"bytes": 8.0 * 34 * case["systems"] * (hi - 32.0) / math.log(hi / 32.0), "flops": 16 * hh[2] * pairs}
    if kind == "labels":
        n = 2.5 * case["systems"]
        return {"bytes": 8.0 * n * (18 + 96), "flops": 12 * hh[4] * 4 * case["systems"]}
    net = 2.0 * (9 * 128 + 2 * 128 * 128 + 128 * 6)
    if kind == "gradient":
        pairs = 3.5 * case["systems"]
        return {"bytes": 2.5 * case["systems"] * 96 + 35078 * 8.0, "flops": 3 * net * pairs}
    if kind == "nearfield":
        return {"bytes": case["n"] * 192.0, "flops": net * 5.6 * case["n"]}
    if kind == "periodic":
        n = case["n"]
        return {"bytes": n * 96.0, "flops": n * (240 * 60 + 2 * 512 * 8.0) + 168.0 * n * 30 * math.log2(168.0 * n)}
    if kind == "flow":
        n, t, m = case["n"], case["trunc"], case["points"]
        return {"bytes": m * 48.0 + n * 8.0 * (9 + h[t]), "flops": {2: 250.0, 3: 531.0}[t] * n * m}
    n = case["n"]
    return {"bytes": n * 240.0, "flops": 500.0 * n * n}


# ----------------------------------------------------------------- results in 64 bits: modes

_H_MODES = [(2, 0), (3, 2), (3, 1), (3, 0), (4, 2), (4, 1), (4, 0), (5, 2)]   # (rank L, sigma)


def _modes(trunc):
    return [(1, 0), (2, 1)] + _H_MODES[:{2: 2, 3: 5, 4: 8}[trunc]]


def _ranks(trunc):
    """Components of the higher modes, in order."""
    return [2 * (L - sg) + 1 for L, sg in _modes(trunc)[2:]]


@functools.lru_cache(None)
def _stf(k):
    """Orthonormal basis [2k+1, 3, ..., 3] of the symmetric traceless tensors of rank k whose
    polynomials are the real solid harmonics, mu = -k..k."""
    leg = np.polynomial.legendre.Legendre.basis(k).convert(kind=np.polynomial.Polynomial)
    out = []
    for mu in range(-k, k + 1):
        m = abs(mu)
        d = leg.deriv(m).coef if m else leg.coef      # in z; homogenised with r^2 below
        poly = {}
        for j, c in enumerate(d):
            if abs(c) < 1e-15:
                continue
            h = (k - m - j) // 2                      # z^j (x^2+y^2+z^2)^h
            for a, b in itertools.product(range(h + 1), repeat=2):
                if a + b > h:
                    continue
                w = math.factorial(h) // (math.factorial(a) * math.factorial(b) * math.factorial(h - a - b))
                for t in range(m + 1):                # (x + i y)^m: cos part t even, sin part t odd
                    if (t % 2 == 0) != (mu >= 0):
                        continue
                    sg = (-1) ** (t // 2)
                    key = (2 * a + m - t, 2 * b + t, j + 2 * (h - a - b))
                    poly[key] = poly.get(key, 0.0) + c * w * sg * math.comb(m, t)
        T = np.zeros((3,) * k)
        for idx in itertools.product(range(3), repeat=k):
            e = tuple(idx.count(i) for i in range(3))
            T[idx] = poly.get(e, 0.0) * math.factorial(e[0]) * math.factorial(e[1]) * math.factorial(e[2]) / math.factorial(k)
        out.append(T / math.sqrt((T ** 2).sum()))
    return np.stack(out)


def _tail(X):
    """Symmetric traceless part in every index of X but the first."""
    k = X.ndim - 1
    if k <= 1:
        return X
    U = _stf(k).reshape(2 * k + 1, -1)
    return (X.reshape(3, -1) @ U.T @ U).reshape(X.shape)


@functools.lru_cache(None)
def _basis(trunc):
    """Embedded tensors e_p (unit norm), their norms c, their ranks L."""
    levi = np.zeros((3, 3, 3))
    for i, j, k in itertools.permutations(range(3)):
        levi[i, j, k] = (j - i) * (k - i) * (k - j) / 2
    es, cs, ls = [], [], []
    for L, sg in _modes(trunc):
        for T in _stf(L - sg):
            if sg == 0:
                E = T
            elif sg == 1:
                E = -(L - 1) / L * _tail(np.tensordot(levi, T, axes=([2], [0])))
            else:
                E = L * (L - 1) / (2 * (2 * L - 1)) * _tail(np.multiply.outer(np.eye(3), T))
            c = math.sqrt((E ** 2).sum())
            es.append(E / c)
            cs.append(c)
            ls.append(L)
    return es, np.array(cs), ls


def _poly(T):
    """sum over the indices of T of T[i..] x_i...: {exponents: coefficient}."""
    out = {}
    for idx in itertools.product(range(3), repeat=T.ndim):
        if T[idx] != 0.0:
            e = tuple(idx.count(i) for i in range(3))
            out[e] = out.get(e, 0.0) + float(T[idx])
    return out


def _mul(p, q, out, f):
    for (a, b, c), u in p.items():
        for (d, e, g), v in q.items():
            k = (a + d, b + e, c + g)
            out[k] = out.get(k, 0.0) + f * u * v


@functools.lru_cache(None)
def _self(trunc):
    """One-body scalars: (2l+1)/(2 pi) of the integral of Y (I - nn) Y over the unit sphere."""
    x, w = np.polynomial.legendre.leggauss(12)
    phi = 2 * np.pi * np.arange(26) / 26
    st = np.sqrt(1 - x * x)
    n = np.stack([np.outer(st, np.cos(phi)), np.outer(st, np.sin(phi)), np.outer(x, np.ones(26))], -1).reshape(-1, 3)
    wt = np.repeat(w * 2 * np.pi / 26, 26)
    es, _, ls = _basis(trunc)
    out = []
    for E, L in zip(es, ls):
        df = 1.0
        for j in range(1, L):
            df *= 2 * j - 1
        v = np.zeros((len(n), 3))
        for i in range(3):
            for e, c in _poly(E[i]).items():
                v[:, i] += c * n[:, 0] ** e[0] * n[:, 1] ** e[1] * n[:, 2] ** e[2]
        v *= df
        out.append((2 * L - 1) / (2 * np.pi) * float(np.sum(wt * ((v * v).sum(1) - (v * n).sum(1) ** 2))))
    return np.array(out)


def _monomials(lo, hi):
    return [(a, b, n - a - b) for n in range(lo, hi + 1) for a in range(n + 1) for b in range(n - a + 1)]


@functools.lru_cache(None)
def _weights(trunc, point):
    """W [monomials, q, p]: block[p, q] = sum over the monomials of W d^n(r or 1/r); the first
    monomials are those of r (degrees 2..K), then those of 1/r (0..K).  point: the velocity
    rows of a target of radius zero instead of every row."""
    es, _, ls = _basis(trunc)
    top = max(ls) - 1
    K = (0 if point else top) + top + 2
    mr = {e: i for i, e in enumerate(_monomials(2, K))}
    m1 = {e: i + len(mr) for i, e in enumerate(_monomials(0, K))}
    rows = range(3) if point else range(len(es))
    W = np.zeros((len(mr) + len(m1), len(es), len(rows)))
    pv = [[_poly(E[i]) if E.ndim > 1 else {(0, 0, 0): float(E[i])} for i in range(3)] for E in es]
    ps = [_poly(E) for E in es]
    for p in rows:
        for q in range(len(es)):
            lp, lq = ls[p] - 1, ls[q] - 1
            pref = A ** (lp + lq) * (-1) ** lq
            c = A * A * ((0.0 if point else 1.0 / (4 * lp + 6)) + 1.0 / (4 * lq + 6))
            w, wd = {}, {}
            _mul(ps[p], ps[q], w, 1.0)
            for i in range(3):
                _mul(pv[p][i], pv[q][i], wd, 1.0)
            for e, v in w.items():
                W[mr[e], q, p] -= pref * v
                W[m1[e], q, p] -= 2.0 * c * pref * v
            for e, v in wd.items():
                W[m1[e], q, p] += 2.0 * pref * v
    return torch.tensor(W, dtype=torch.float64, device="cuda"), K


def _derivatives(d, K):
    """Derivatives of r (degrees 2..K) and of 1/r (0..K) at d [..., 3], stacked last.  With
    f_m = ((1/r) d/dr)^m r, D[a + e_i, m] = x_i D[a, m+1] + a_i D[a - e_i, m+1]."""
    x = [d[..., i] for i in range(3)]
    r2 = x[0] ** 2 + x[1] ** 2 + x[2] ** 2
    ir2 = 1.0 / r2
    f = [r2.sqrt()]
    f.append(f[0] * ir2)
    for m in range(2, K + 2):
        f.append(f[-1] * ir2 * (-(2 * m - 3)))
    below, cur = None, [{(0, 0, 0): f[m]} for m in range(K + 2)]
    out_r, out_1 = [], [cur[1][0, 0, 0]]
    for n in range(1, K + 1):
        nxt = []
        for m in range(0, K + 2 - n):
            lev = {}
            for e in _monomials(n, n):
                i = next(j for j in range(3) if e[j] > 0)
                b = tuple(v - (j == i) for j, v in enumerate(e))
                t = x[i] * cur[m + 1][b]
                if b[i] > 0:
                    t = t + b[i] * below[m + 1][tuple(v - (j == i) for j, v in enumerate(b))]
                lev[e] = t
            nxt.append(lev)
        below, cur = cur, nxt
        if n >= 2:
            out_r += [cur[0][e] for e in _monomials(n, n)]
        out_1 += [cur[1][e] for e in _monomials(n, n)]
    return out_r, out_1


def _pair_derivs(X, R, K, skip):
    """[targets, sources, monomials] of X - R; skip: targets are the sources, no self pairs."""
    d = X[:, None, :] - R[None, :, :]
    if skip is not None:
        i = torch.arange(len(X), device=X.device)
        d[i, skip + i] = 1.0e3       # any finite value; the row is cleared below
    r, i1 = _derivatives(d, K)
    D = torch.stack(r + i1, -1)
    if skip is not None:
        D[i, skip + i] = 0.0
    return D


class _Pairs:
    """The pair operator of one suspension in 64 bits: y[n, p] = sum_m G_nm[p, q] x[m, q]."""

    def __init__(self, R, trunc, keep=True):
        self.R, self.trunc = R, trunc
        self.W, self.K = _weights(trunc, False)
        n = len(R)
        self.step = max(1, int(3.0e8 / (n * self.W.shape[0] * 8)) if n else 1)
        self.D = None
        if keep:
            self.D = [self._chunk(k) for k in range(0, n, self.step)]

    def _chunk(self, k):
        X = self.R[k:k + self.step]
        return _pair_derivs(X, self.R, self.K, k).reshape(len(X), -1)

    def __call__(self, x, cols, rows):
        n = len(self.R)
        W = self.W[:, cols][:, :, rows]
        B = torch.einsum("aqp,mq->map", W, x).reshape(n * W.shape[0], W.shape[2])
        chunks = self.D if self.D is not None else (self._chunk(k) for k in range(0, n, self.step))
        return torch.cat([D @ B for D in chunks])


def _to_x(F, T, VH, trunc):
    """Internal coordinates of -F, -T/a and of packed higher coefficients."""
    _, c, _ = _basis(trunc)
    c = torch.tensor(c, dtype=torch.float64, device=F.device)
    i = [1, 2, 0]
    return torch.cat([-F[:, i], -T[:, i] / A * c[3]], 1), VH * c[6:], c


def _from_x(y, Va, Oa, c):
    i = [2, 0, 1]
    return Va + y[:, :3][:, i], Oa + y[:, 3:][:, i] / c[3] / (2 * A)


def _galerkin(R, Va, Oa, VH, F, T, trunc):
    """V, Omega, Q^H of the Galerkin system of one suspension (conjugate gradients to rounding)."""
    xF, xV, c = _to_x(F, T, VH, trunc)
    G = _Pairs(R, trunc)
    g = torch.tensor(_self(trunc) / A, dtype=torch.float64, device=R.device)
    D = len(g)
    L, H = slice(0, 6), slice(6, D)
    b = -8 * math.pi * ETA * xV - G(xF, L, H)
    q = b / g[6:]
    r = b - G(q, H, H) - g[6:] * q
    z = r / g[6:]
    p, rz = z.clone(), (r * z).sum()
    for _ in range(80):
        w = G(p, H, H) + g[6:] * p
        al = rz / (p * w).sum()
        q = q + al * p
        r = r - al * w
        if float(r.norm()) <= 2e-15 * float(b.norm()):
            break
        z = r / g[6:]
        new = (r * z).sum()
        p, rz = z + (new / rz) * p, new
    x = torch.cat([xF, q], 1)
    y = -(G(x, slice(0, D), L) + g[:6] * xF) / (8 * math.pi * ETA)
    V, Om = _from_x(y, Va, Oa, c)
    return V, Om, q / c[6:]


def _trap(R, p, trunc, k, vs, s0, d0):
    U = torch.tensor(_stf(2), dtype=torch.float64, device=R.device)
    VH = torch.zeros(len(R), sum(_ranks(trunc)), dtype=torch.float64, device=R.device)
    VH[:, :5] = s0 * torch.einsum("uij,ni,nj->nu", U, p, p)
    VH[:, 5:8] = d0 * p[:, [1, 2, 0]]
    z = torch.zeros_like(R)
    return dict(F=-k * R, T=z, Va=vs * p, Oa=z, VH=VH)


def _euler(R, p, V, Om, dt):
    q = p + dt * torch.cross(Om, p, dim=1)
    return R + dt * V, q / q.norm(dim=1, keepdim=True)


def _superpose(R, F, T, S, d, Va, Oa):
    """Closed form at l <= 2: S = V^(2s) as a tensor [n, 3, 3], d = V^(3t)."""
    n = len(R)
    F8, T8 = F / (8 * math.pi * ETA), T / (8 * math.pi * ETA)
    S = -(5.0 / 6.0) * A * A * S
    d = A ** 3 / 10.0 * d
    V = Va + F / (6 * math.pi * ETA * A)
    Om = Oa + T / (8 * math.pi * ETA * A ** 3)
    step = max(1, int(2.0e7 / n))
    dot = lambda u, v: (u * v).sum(-1)  # noqa: E731
    for k in range(0, n, step):
        x = R[k:k + step, None] - R[None]
        i = torch.arange(len(x), device=R.device)
        r2 = dot(x, x)
        r2[i, k + i] = math.inf
        ri = r2.rsqrt()
        r3, r5 = ri ** 3, ri ** 5
        Sx = torch.einsum("mij,nmj->nmi", S, x)
        xSx = dot(x, Sx)
        cr = lambda u: torch.cross(u[None].expand_as(x), x, dim=-1)  # noqa: E731
        v = (ri + 2 * A * A / 3 * r3)[..., None] * F8 + (((r3 - 2 * A * A * r5) * dot(x, F8))[..., None] * x)
        v = v + r3[..., None] * cr(T8) + ((-3 * r5 + 8 * A * A * ri ** 7) * xSx)[..., None] * x
        v = v - (16.0 / 5.0 * A * A * r5)[..., None] * Sx + (3 * dot(x, d) * r5)[..., None] * x - r3[..., None] * d
        V[k:k + step] += v.sum(1)
        w = r3[..., None] * cr(F8) + 0.5 * ((3 * dot(x, T8) * r5)[..., None] * x - r3[..., None] * T8)
        w = w + (3 * r5)[..., None] * torch.cross(x, Sx, dim=-1)
        Om[k:k + step] += w.sum(1)
    return V, Om


def _strain(p, s0):
    return s0 * (p[:, :, None] * p[:, None, :] - torch.eye(3, dtype=p.dtype, device=p.device) / 3)


# ------------------------------------------------- results in 64 bits: other Green's functions


def _wall(R, F, T, S):
    """Image flow of forces, torques and stresslets above the wall z = 0 and half its curl."""
    n = len(R)
    eye = torch.eye(3, dtype=R.dtype, device=R.device)
    levi = torch.zeros(3, 3, 3, dtype=R.dtype, device=R.device)
    for i, j, k in itertools.permutations(range(3)):
        levi[i, j, k] = (j - i) * (k - i) * (k - j) / 2
    Dp = 20.0 / 3.0 * math.pi * ETA * A * A * S + 0.5 * torch.einsum("kjl,ml->mjk", levi, T)
    sgn = torch.tensor([1.0, 1.0, -1.0], dtype=R.dtype, device=R.device)
    V, Om = torch.zeros_like(R), torch.zeros_like(R)
    for k in range(0, n, 64):
        X = R[k:k + 64]
        x0 = X[:, None].expand(len(X), n, 3).contiguous()
        y0 = R[None].expand(len(X), n, 3).contiguous()

        def image(x, y):
            h = y[..., 2][..., None, None]
            r = x - y * sgn
            ir = (r * r).sum(-1).rsqrt()[..., None, None]
            rr = r[..., :, None] * r[..., None, :]
            r3, ri, rj = r[..., 2][..., None, None], r[..., :, None], r[..., None, :]
            t = h * (eye * ir ** 3 - 3 * rr * ir ** 5) + eye[:, 2][:, None] * rj * ir ** 3
            t = t - (eye * r3 + ri * eye[2]) * ir ** 3 + 3 * rr * r3 * ir ** 5
            return -(eye * ir + rr * ir ** 3) + 2 * h * sgn * t

        def flow(x):
            u = torch.einsum("nmij,mj->nmi", image(x, y0), F)
            for q in range(3):
                _, dw = torch.func.jvp(lambda y: image(x, y), (y0,), (eye[q].expand_as(y0).contiguous(),))
                u = u + torch.einsum("nmij,mj->nmi", dw, Dp[:, :, q])
            return u

        V[k:k + 64] = flow(x0).sum(1)
        for ax in range(3):
            _, du = torch.func.jvp(flow, (x0,), (eye[ax].expand_as(x0).contiguous(),))     # d u_i / d x_ax
            Om[k:k + 64] += 0.5 * torch.einsum("ki,ni->nk", levi[:, ax, :], du.sum(1))
    return V / (8 * math.pi * ETA), Om / (8 * math.pi * ETA)


def _periodic(R, F, Va, L):
    n = len(R)
    rc = L / 2
    xi = 5.8 / rc
    u = torch.zeros_like(R)
    step = max(1, int(4.0e7 / n))
    for k in range(0, n, step):
        x = R[k:k + step, None] - R[None]
        x = x - L * torch.round(x / L)
        r2 = (x * x).sum(-1)
        i = torch.arange(len(x), device=R.device)
        r2[i, k + i] = math.inf
        r2 = torch.where(r2 < rc * rc, r2, math.inf)
        r = r2.sqrt()
        rf = torch.where(r2 < math.inf, r, 1.0)
        e = torch.exp(-xi * xi * r2)
        f1 = torch.erfc(xi * r) - 2 * xi / math.sqrt(math.pi) * rf * e
        f2 = 4 * xi / math.sqrt(math.pi) * (xi * xi * rf * rf - 1) * e
        a, b = f2 + f1 / r, (f2 - f1 / r) / r2
        u[k:k + step] = a @ F - ((b * (x * F).sum(-1))[..., None] * x).sum(1)
        del x, r2, r, rf, e, f1, f2, a, b
    mm = int(2 * xi * math.sqrt(42.0) * L / (2 * math.pi))
    m = torch.arange(-mm, mm + 1, dtype=torch.float64, device=R.device)
    s = R / L - torch.floor(R / L)
    ex = [torch.polar(torch.ones_like(t), t) for t in (2 * math.pi * ((s[:, d, None] * m) % 1.0) for d in range(3))]
    kk = 2 * math.pi / L * m
    for ix in range(mm, 2 * mm + 1):
        P = ex[0][:, ix, None] * ex[1]                                          # [n, my]
        S = torch.stack([P.conj().T @ (F[:, d, None] * ex[2].conj()) for d in range(3)])   # [3, my, mz]
        k = torch.stack(torch.broadcast_tensors(kk[ix], kk[:, None], kk[None, :]))
        k2 = (k * k).sum(0)
        q = k2 / (4 * xi * xi)
        pref = (2.0 if ix > mm else 1.0) / L ** 3 * 8 * math.pi / k2 * (1 + q + 2 * q * q) * torch.exp(-q)
        pref = torch.where((k2 > 0) & (q < 42.0), pref, 0.0)
        ik2 = torch.where(k2 > 0, 1.0 / k2, 0.0)
        W = pref * (S - k * (k * S).sum(0) * ik2)
        for d in range(3):
            u[:, d] += ((P @ W[d]) * ex[2]).sum(1).real
    u = u - 8 * xi / math.sqrt(math.pi) * F
    return Va + F / (6 * math.pi * ETA * A) + u / (8 * math.pi * ETA)


def _flow(R, F, T, QH, X, trunc):
    xF, xQ, _ = _to_x(F, T, QH, trunc)
    W, K = _weights(trunc, True)
    x = torch.cat([xF, xQ], 1)
    n = len(R)
    B = torch.einsum("aqp,mq->map", W, x).reshape(n * W.shape[0], 3)
    U = torch.empty_like(X)
    inside = torch.zeros(len(X), dtype=torch.bool, device=X.device)
    step = max(1, int(6.0e8 / (n * W.shape[0] * 8)))
    for k in range(0, len(X), step):
        Y = X[k:k + step]
        inside[k:k + step] = (((Y[:, None] - R[None]) ** 2).sum(-1) < A * A).any(1)
        U[k:k + step] = (_pair_derivs(Y, R, K, None).reshape(len(Y), -1) @ B)[:, [2, 0, 1]]
    U = -U / (8 * math.pi * ETA)
    U[inside] = math.nan
    return U, int(inside.sum())


def _close_pairs(R, offsets):
    """Ordered pairs closer than 4 a, within each system if offsets are given."""
    n = len(R)
    if offsets is not None:
        o = torch.tensor(offsets, device=R.device)
        cnt = o[1:] - o[:-1]
        sysid = torch.repeat_interleave(torch.arange(len(cnt), device=R.device), cnt)
        tg, sr = [], []
        for sh in (-2, -1, 1, 2):
            i = torch.arange(max(0, -sh), min(n, n - sh), device=R.device)
            i = i[(sysid[i] == sysid[i + sh]) & (((R[i] - R[i + sh]) ** 2).sum(1) < 16.0 * A * A)]
            tg.append(i)
            sr.append(i + sh)
        return torch.cat(tg), torch.cat(sr)
    out = []
    step = max(1, int(1.0e8 / n))
    for k in range(0, n, step):
        d2 = sum((R[k:k + step, None, i] - R[None, :, i]) ** 2 for i in range(3))
        i, j = torch.nonzero(d2 < 16.0 * A * A, as_tuple=True)
        keep = (i + k) != j
        out.append(((i + k)[keep], j[keep]))
    return torch.cat([t for t, _ in out]), torch.cat([s for _, s in out])


def _network(theta, R, p, tg, sr):
    """Per-sphere sums [n, 6] of the rotated outputs."""
    rho = R[tg] - R[sr]
    r = rho.norm(dim=1, keepdim=True)
    ez = rho / r
    pn, pm = p[tg], p[sr]
    t = pn - (pn * ez).sum(1, keepdim=True) * ez
    exx = t / t.norm(dim=1, keepdim=True)
    ey = torch.cross(ez, exx, dim=1)
    dot = lambda u, v: (u * v).sum(1, keepdim=True)  # noqa: E731
    u, d = 2 * A / r, torch.clamp(r / A - 2.0, min=0.01)
    f = torch.cat([u, u ** 3, d, d.log(), dot(pn, ez), dot(pn, exx), dot(pm, exx), dot(pm, ey), dot(pm, ez)], 1)
    k = 0
    for fo, fi in ((128, 9), (128, 128), (128, 128), (6, 128)):
        f = f @ theta[k:k + fo * fi].reshape(fo, fi).T + theta[k + fo * fi:k + fo * fi + fo]
        k += fo * fi + fo
        if fo == 128:
            f = torch.tanh(f)
    fr = torch.stack([exx, ey, ez], 1)
    lab = torch.cat([torch.einsum("pc,pci->pi", f[:, :3], fr), torch.einsum("pc,pci->pi", f[:, 3:], fr)], 1)
    return torch.zeros(len(R), 6, dtype=R.dtype, device=R.device).index_add(0, tg, lab)


def exact(case, seed):
    dev = torch.device("cuda")
    raw = _raw(case, seed)
    t = {k: torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)
         for k, v in raw.items() if isinstance(v, np.ndarray)}
    kind, R, p = case["kind"], t["R"], t.get("p")
    if kind in ("orbit", "cloud"):
        orbit = kind == "orbit"
        k, vs, s0, d0, dt = ((_k_orbit(), 2 * B1 / 3, -0.6 * B2, 10 * B1 / 3, 0.5) if orbit else
                             (_k_cloud(), VS, S0, 0.0, 0.05))
        z = torch.zeros_like(R)
        for _ in range(case["steps"]):
            R, p = _euler(R, p, *_superpose(R, -k * R, z, _strain(p, s0), d0 * p, vs * p, z), dt)
        return [R, p]
    if kind == "step":
        i = _trap(R, p, case["trunc"], K_TRAP, VS, S0, 0.0)
        V, Om, _ = _galerkin(R, i["Va"], i["Oa"], i["VH"], i["F"], i["T"], case["trunc"])
        return list(_euler(R, p, V, Om, 0.1))
    if kind == "solve":
        i = _trap(R, p, case["trunc"], K_TRAP, VS, S0, 0.0)
        return list(_galerkin(R, i["Va"], i["Oa"], i["VH"], i["F"], i["T"], case["trunc"]))
    if kind == "batch":
        i = _trap(R, p, 2, K_TRAP, VS, S0, 0.0)
        o = raw["offsets"]
        got = [_galerkin(*(v[a:b] for v in (R, i["Va"], i["Oa"], i["VH"], i["F"], i["T"])), 2) for a, b in zip(o, o[1:])]
        return [torch.cat(v) for v in zip(*got)]
    if kind == "labels":
        i = _trap(R, p, 4, 0.0, VS, S0, 0.0)
        return _labels(R, i, raw["offsets"])
    if kind == "gradient":
        th = t["theta"].requires_grad_(True)
        tg, sr = _close_pairs(R, raw["offsets"])
        loss = ((_network(th, R, p, tg, sr) - t["labels"]) ** 2).sum() / (6 * len(R))
        (g,) = torch.autograd.grad(loss, th)
        return [float(loss.detach()), g]
    if kind == "nearfield":
        tg, sr = _close_pairs(R, None)
        s = S0 / 2.0 * _network(t["theta"], R, p, tg, sr)
        return [t["V"] + s[:, :3], t["Om"] + s[:, 3:], len(tg)]
    if kind == "periodic":
        return [_periodic(R, t["F"], t["Va"], raw["L"])]
    if kind == "flow":
        return list(_flow(R, t["Fe"], t["Te"], t["QH"], t["X"], case["trunc"]))
    S = _strain(p, S0)
    V, Om = _superpose(R, -K_TRAP * R, t["Te"], S, 0.02 * p, VS * p, torch.zeros_like(R))
    Vw, Ow = _wall(R, -K_TRAP * R, t["Te"], S)
    return [V + Vw, Om + Ow]


def _labels(R, i, offsets):
    """Dense solves of the two- and three-sphere systems, batched by size."""
    W, K = _weights(4, False)
    g = torch.tensor(_self(4) / A, dtype=torch.float64, device=R.device)
    D = len(g)
    xF, xV, c = _to_x(i["F"], i["T"], i["VH"], 4)
    V, Om, Q = torch.empty_like(R), torch.empty_like(R), torch.empty_like(xV)
    o = np.array(offsets)
    for n in (2, 3):
        first = torch.tensor(o[:-1][np.diff(o) == n], device=R.device)
        for f in first.split(1000):
            ids = f[:, None] + torch.arange(n, device=R.device)                  # [s, n]
            G = torch.zeros(len(f), n, D, n, D, dtype=R.dtype, device=R.device)
            for a in range(n):
                G[:, a, :, a, :] = torch.diag(g)
                for b in range(n):
                    if a != b:
                        d = R[ids[:, a]] - R[ids[:, b]]
                        r, i1 = _derivatives(d, K)
                        G[:, a, :, b, :] = torch.einsum("sa,aqp->spq", torch.stack(r + i1, -1), W)
            H = D - 6
            HH = G[:, :, 6:, :, 6:].reshape(len(f), n * H, n * H)
            HL = G[:, :, 6:, :, :6].reshape(len(f), n * H, n * 6)
            LL = G[:, :, :6, :, :6].reshape(len(f), n * 6, n * 6)
            LH = G[:, :, :6, :, 6:].reshape(len(f), n * 6, n * H)
            F = xF[ids].reshape(len(f), n * 6, 1)
            b = -8 * math.pi * ETA * xV[ids].reshape(len(f), n * H, 1) - HL @ F
            q = torch.linalg.solve(HH, b)
            y = -(LL @ F + LH @ q) / (8 * math.pi * ETA)
            flat = ids.reshape(-1)
            V[flat], Om[flat] = _from_x(y.reshape(-1, 6), i["Va"][flat], i["Oa"][flat], c)
            Q[flat] = q.reshape(-1, H) / c[6:]
    return [V, Om, Q]

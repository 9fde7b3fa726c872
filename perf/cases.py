"""Performance cases: what a user of the sampler has it do, through its public calls.

Sizes are those of the repository's workloads, tests and micro-benchmarks (or
powers of two between them).  A case is a dict of plain values; `op` names the call:

  fields    Hierarchy.sample_fields, loads drawn from the seed
  batched   sample_fields_batched over instances of several surfaces
  grad      WMField forward and backward of the loss sum_s |u_s - g_s|_M^2
  loads     Hierarchy.noise_loads
  sqrt      Hierarchy.noise_loads_sqrt
  mass      Hierarchy.apply_mass (the M-weighted norms and loss gradients)

`exact` is a plain float64 restatement (B-spline bases, the two analytic
surfaces, assembled matrices, dense solves, Philox normals) without the package.
"""
import functools
import math
import random

import numpy as np
import torch

import paper_2605_24882_gb300 as wm

_DEV = "cuda"

# ------------------------------------------------------------------ the cases


def _surface(kind, p, j):
    """Sphere: 6 x 2^j x 2^j elements; torus: 2^(j+1) x 2^j (R = 1, r = 0.4)."""
    if kind == "sphere":
        return dict(kind=kind, p=p, nu=2 ** j, nv=2 ** j, levels=j + 1)
    return dict(kind=kind, p=p, nu=2 ** (j + 1), nv=2 ** j, levels=j - 2)


def _fields(name, surf, ns, kappa, beta, split="standard", precision="mixed", k=0.3, lo=-35, hi=35, rtol=1e-8):
    return dict(name=name, op="fields", **surf, ns=ns, kappa=kappa, beta=beta, split=split, precision=precision,
                k=k, lo=lo, hi=hi, rtol=rtol)


def listed():
    return [
        # the plain method on a coarse sphere (488 DOFs, one sample, float64, 51 nodes): the smallest
        # call, as in interactive use, parameter scans and tests; launches and round trips count
        _fields("sphere8_fp64_s1", _surface("sphere", 2, 3), 1, 2.0, 0.75, precision="fp64", k=0.4, lo=-25, hi=25,
                rtol=1e-11),
        # one realisation of a field on the everyday mesh (25,352 DOFs): 71 systems of different
        # shifts, the latency a user waits for a single picture
        _fields("sphere64_s1", _surface("sphere", 2, 6), 1, 5.0, 1.3),
        # the throughput workload: 256 samples in one call (one integer solve, then 71 nodes)
        _fields("sphere64_s256", _surface("sphere", 2, 6), 256, 5.0, 1.3),
        # a ragged sample count and the improved split (an integer solve and two passes), 6,536 DOFs
        _fields("sphere32_s20_improved", _surface("sphere", 2, 5), 20, 7.5, 1.8, split="improved"),
        # a float64 reference run over a full tile of samples, as accuracy studies make
        _fields("sphere32_fp64_s32", _surface("sphere", 2, 5), 32, 5.0, 1.3, precision="fp64", rtol=1e-10),
        # the large bicubic torus (131,072 DOFs), a Monte Carlo batch of 64 samples
        _fields("torus512_p3_s64", _surface("torus", 3, 8), 64, 10.0, 0.6),
        # a few samples on a fine mesh (393,512 DOFs)
        _fields("sphere256_s3", _surface("sphere", 2, 8), 3, 5.0, 0.8),
        # an uneven batch: 8 instances on 4 surfaces, ragged sample counts, every kappa and beta its own
        dict(name="batched_8", op="batched", n_inst=8, j_lo=3, j_hi=6, draw_seed=11, rtol=1e-8),
        # differentiation: field loss on a bicubic sphere (101,402 DOFs), forward and adjoint
        dict(name="grad_sphere128_p3_s16", op="grad", **_surface("sphere", 3, 7), ns=16, kappa=4.0, beta=0.8,
             split="standard", precision="mixed", k=0.3, lo=-35, hi=35, rtol=1e-8),
        # white-noise loads alone, for a program with its own solver
        dict(name="loads_sphere64_s256", op="loads", **_surface("sphere", 2, 6), ns=256),
        # loads by the matrix square root, 20 nodes on the library's spectrum bounds
        dict(name="sqrt_sphere64_s64", op="sqrt", **_surface("sphere", 2, 6), ns=64, nodes=20, rtol=1e-10),
        # M u of a batch of fields: norms, losses and their gradients
        dict(name="mass_sphere64_s100", op="mass", **_surface("sphere", 2, 6), ns=100),
    ]


def _dofs(c):
    if c["kind"] == "torus":
        return c["nu"] * c["nv"]
    m = c["nu"] + c["p"]
    return 6 * m * m - 12 * m + 8


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: surfaces of both kinds and degrees from a few hundred to
    400,000 DOFs, 1 to 256 samples (odd counts among them), kappa and beta as the uneven
    workload draws them, with the number of unknowns (DOFs x systems) within the listed range."""
    op = rng.choice(["fields"] * 6 + ["grad", "batched", "loads", "sqrt", "mass"])
    if op == "batched":
        return dict(op=op, n_inst=rng.randint(3, 12), j_lo=3, j_hi=rng.randint(4, 6), draw_seed=rng.randint(0, 9999),
                    rtol=1e-8)
    kind, p = rng.choice([("sphere", 2), ("sphere", 3), ("torus", 2), ("torus", 3)])
    c = dict(op=op, **_surface(kind, p, rng.randint(4 if kind == "torus" else 3, 8)))
    n = _dofs(c)
    if op in ("loads", "sqrt", "mass"):
        if op == "sqrt":
            c = dict(op=op, **_surface(kind, p, rng.randint(4, 6)))
            n = _dofs(c)
        most = {"loads": 256 * 25352, "sqrt": 64 * 25352, "mass": 256 * 25352}[op]
        c["ns"] = _log_int(rng, 1, max(1, min(256, most // n)))
        if op == "sqrt":
            c.update(nodes=rng.randint(10, 24), rtol=1e-10)
        return c
    fp64 = op == "fields" and rng.random() < 0.25
    nodes = 71
    most = 2.5e8 if op == "fields" else 1.1e8
    if p == 3:
        most /= 2
    if fp64:
        most /= 12
    while n * nodes > most:  # at least one sample
        j = int(math.log2(c["nv"])) - 1
        c = dict(op=op, **_surface(kind, p, j))
        n = _dofs(c)
    c["ns"] = _log_int(rng, 1, max(1, min(256, int(most / (n * nodes)))))
    c.update(kappa=round(rng.uniform(1.0, 20.0), 4), beta=round(rng.uniform(0.55, 1.95), 4),
             split=rng.choice(["standard", "improved"]), precision="fp64" if fp64 else "mixed", k=0.3, lo=-35, hi=35,
             rtol=1e-10 if fp64 else 1e-8)
    return c


def _instances(c):
    """The uneven batch of a case: surfaces, kappa, beta and sample counts from draw_seed."""
    rng = random.Random(c["draw_seed"])
    out = []
    for i in range(c["n_inst"]):
        kind, p = rng.choice([("sphere", 2), ("torus", 3)])
        j = rng.randint(max(c["j_lo"], 4) if kind == "torus" else c["j_lo"], c["j_hi"])
        out.append(dict(_surface(kind, p, j), ns=rng.randint(1, 64), kappa=round(rng.uniform(1.0, 20.0), 4),
                        beta=round(rng.uniform(0.55, 1.95), 4)))
    return out


# ------------------------------------------------------------------ the calls


def _geometry(c):
    return wm.Geometry(c["kind"], c["p"], c["nu"], c["nv"], 1.0, 0.4)


def _normal(shape, seed):
    g = torch.Generator(device=_DEV).manual_seed(int(seed))
    return torch.randn(shape, dtype=torch.float64, device=_DEV, generator=g)


def _sampler_args(c):
    return dict(beta=c["beta"], sinc_k=c["k"], l_lo=c["lo"], l_hi=c["hi"], n_samples=c["ns"], split=c["split"],
                precision=c["precision"], rtol=c["rtol"])


def prepare(case, seed):
    c = case
    st = {"case": c, "seed": seed}
    if c["op"] == "batched":
        hiers, st["hiers"], st["descs"] = {}, [], []
        for i, e in enumerate(_instances(c)):
            key = (e["kind"], e["p"], e["nu"], e["nv"])
            if key not in hiers:
                hiers[key] = wm.Hierarchy(_geometry(e), e["levels"])
            st["hiers"].append(hiers[key])
            st["descs"].append(wm.Hierarchy.make_desc(kappa=e["kappa"], beta=e["beta"], split="improved",
                                                      n_samples=e["ns"], seed=seed * 1000 + i, rtol=c["rtol"]))
        return st
    geo = _geometry(c)
    st["hier"] = hier = wm.Hierarchy(geo, 1 if c["op"] in ("loads", "sqrt", "mass") else c["levels"])
    if c["op"] == "sqrt":
        st["bounds"] = geo.mass_bounds(0)
    elif c["op"] == "mass":
        st["x"] = _normal((c["ns"], hier.num_dofs(0)), seed)
    elif c["op"] == "grad":
        st["b"] = hier.noise_loads(seed, c["ns"]).requires_grad_(True)
        st["target"] = _normal((c["ns"], hier.num_dofs(0)), seed)
        st["kappa"] = torch.tensor(c["kappa"], dtype=torch.float64, requires_grad=True)
    return st


def run(state):
    c = state["case"]
    if c["op"] == "fields":
        return state["hier"].sample_fields(kappa=c["kappa"], seed=state["seed"], **_sampler_args(c))[0]
    if c["op"] == "batched":
        return wm.sample_fields_batched(state["hiers"], state["descs"])[0]
    if c["op"] == "grad":
        hier = state["hier"]
        u = wm.WMField.apply(state["b"], state["kappa"], hier, _sampler_args(c))
        grad_u = 2.0 * hier.apply_mass(u.detach() - state["target"])
        gb, gk = torch.autograd.grad(u, (state["b"], state["kappa"]), grad_u)
        return {"u": u.detach(), "grad_b": gb, "grad_kappa": gk}
    if c["op"] == "loads":
        return state["hier"].noise_loads(state["seed"], c["ns"])
    if c["op"] == "sqrt":
        lo, hi = state["bounds"]
        return state["hier"].noise_loads_sqrt(state["seed"], c["ns"], lo, hi, c["nodes"], rtol=c["rtol"])[0]
    return state["hier"].apply_mass(state["x"])


def _split(beta, split):
    """(integer solves, fractional exponent, passes) of beta."""
    n = int(math.floor(beta))
    b = beta - n
    if b == 0.0:
        return n, 0.0, 0
    if split == "improved" and b < 1.0 / 3.0 and n >= 1:
        return n - 1, (1.0 + b) / 2.0, 2
    if split == "improved" and b > 2.0 / 3.0:
        return n, b / 2.0, 2
    return n, b, 1


def _systems(c, beta, split, nodes):
    n, _, passes = _split(beta, split)
    return c["ns"] * (n + passes * nodes)


def work(case):
    """Of one pass.  bytes: the inputs read and the outputs written once.  flops: what the result
    cannot be had without; for the solves one product with S + sigma M per system (a direct or
    iterative solve does more)."""
    c = case
    if c["op"] == "batched":
        by = fl = 0.0
        for e in _instances(c):
            w = work(dict(e, op="fields", split="improved", lo=-35, hi=35))
            by, fl = by + w["bytes"], fl + w["flops"]
        return {"bytes": by, "flops": fl}
    n = float(_dofs(c))
    row = (2 * c["p"] + 1) ** 2
    if c["op"] == "fields":
        return {"bytes": 8 * n * c["ns"] + 16 * n * row,
                "flops": 2 * row * n * _systems(c, c["beta"], c["split"], c["hi"] - c["lo"] + 1)}
    if c["op"] == "grad":  # b, target read; u, dL/db written; forward and adjoint systems
        return {"bytes": 32 * n * c["ns"] + 16 * n * row,
                "flops": 4 * row * n * _systems(c, c["beta"], c["split"], c["hi"] - c["lo"] + 1)}
    q = float(c["nu"] * c["nv"] * (6 if c["kind"] == "sphere" else 1) * (c["p"] + 1) ** 2)
    if c["op"] == "loads":  # a Box–Muller pair and the sum-factorised contraction per Gauss point
        return {"bytes": 8 * n * c["ns"] + 8 * q, "flops": q * c["ns"] * (40 + 4 * (c["p"] + 1))}
    if c["op"] == "sqrt":
        return {"bytes": 8 * n * c["ns"] + 8 * n * row, "flops": 2 * row * n * c["ns"] + 2 * c["nodes"] * n * c["ns"]}
    return {"bytes": 16 * n * c["ns"] + 8 * n * row, "flops": 2 * row * n * c["ns"]}


# ------------------------------------------------------------------ float64 values without the package

# cube faces: patch m has coordinate a = 2u - 1, b = 2v - 1 and n = s
_FACES = ((1, 2, 0, 1), (2, 1, 0, -1), (2, 0, 1, 1), (0, 2, 1, -1), (0, 1, 2, 1), (1, 0, 2, -1))


def _bspline(knots, p, x):
    """Values and derivatives [len(x), len(knots) - p - 1] of all B-splines of degree p (Cox–de Boor)."""
    val = ((knots[:-1][None, :] <= x[:, None]) & (x[:, None] < knots[1:][None, :])).astype(np.float64)
    der = np.zeros_like(val)
    for d in range(1, p + 1):
        m = len(knots) - d - 1
        low = val
        val, der = np.zeros((len(x), m)), np.zeros((len(x), m))
        for i in range(m):
            for k, s, w in ((i, 1.0, lambda a, b: x - a), (i + 1, -1.0, lambda a, b: b - x)):
                a, b = knots[k], knots[k + d]
                if b > a:
                    val[:, i] += w(a, b) / (b - a) * low[:, k]
                    der[:, i] += s * d / (b - a) * low[:, k]
    return val, der


def _bases(n, p, gx, periodic):
    """Values and derivatives [n, nq, p + 1] (with respect to the patch parameter) of the p + 1
    functions of every element at its Gauss points."""
    if periodic:
        knots = np.arange(-p, p + 2, dtype=np.float64)
        v, d = _bspline(knots, p, gx)  # the element [0, 1]
        v, d = v[:, :p + 1], d[:, :p + 1] * n
        return np.broadcast_to(v, (n,) + v.shape), np.broadcast_to(d, (n,) + d.shape)
    knots = np.concatenate([np.zeros(p), np.arange(n + 1) / n, np.ones(p)])
    V, D = np.empty((n, len(gx), p + 1)), np.empty((n, len(gx), p + 1))
    for e in range(n):
        v, d = _bspline(knots[e:e + 2 * p + 2], p, (e + gx) / n)
        V[e], D[e] = v, d
    return V, D


def _connectivity(c):
    """Global DOFs [patches, nv, nu, (p+1)^2] of every element and their number; shared DOFs
    (equal points of the cube lattice) keep the index of their first occurrence."""
    p, nu, nv = c["p"], c["nu"], c["nv"]
    k = np.arange(p + 1)
    if c["kind"] == "torus":
        iu, iv = (np.arange(nu)[:, None] - p + k) % nu, (np.arange(nv)[:, None] - p + k) % nv
        conn = iv[:, None, :, None] * nu + iu[None, :, None, :]
        return conn.reshape(1, nv, nu, (p + 1) ** 2), nu * nv
    m = nu + p
    keys = np.empty((6, m, m), dtype=np.int64)
    for f, (a, b, n, s) in enumerate(_FACES):
        pt = [None, None, None]
        pt[a], pt[b] = np.broadcast_to(np.arange(m)[None, :], (m, m)), np.broadcast_to(np.arange(m)[:, None], (m, m))
        pt[n] = np.full((m, m), m - 1 if s > 0 else 0)
        keys[f] = (pt[0] * m + pt[1]) * m + pt[2]
    _, first, inv = np.unique(keys.reshape(-1), return_index=True, return_inverse=True)
    rank = np.empty(len(first), dtype=np.int64)
    rank[np.argsort(first)] = np.arange(len(first))
    l2g = rank[inv.reshape(-1)].reshape(6, m, m)
    iu, iv = np.arange(nu)[:, None] + k, np.arange(nv)[:, None] + k
    conn = l2g[:, iv[:, None, :, None], iu[None, :, None, :]]
    return conn.reshape(6, nv, nu, (p + 1) ** 2), len(first)


def _space(c):
    """Element quadrature of a surface: connectivity, local functions, weights w a and stiffness metric."""
    p, nu, nv = c["p"], c["nu"], c["nv"]
    nq = p + 1
    gx, gw = np.polynomial.legendre.leggauss(nq)
    gx, gw = (gx + 1) / 2, gw / 2
    periodic = c["kind"] == "torus"
    (bu, du), (bv, dv) = _bases(nu, p, gx, periodic), _bases(nv, p, gx, periodic)
    u, v = (np.arange(nu)[:, None] + gx) / nu, (np.arange(nv)[:, None] + gx) / nv
    U, V = u[None, :, None, :], v[:, None, :, None]  # [nv, nu, gv, gu]
    metric = []
    if periodic:
        t = 2 * np.pi
        kuu, kvv, kuv = (t * (1 + 0.4 * np.cos(t * V))) ** 2 + 0 * U, (t * 0.4) ** 2 + 0 * U + 0 * V, 0 * U + 0 * V
        metric.append((kuu, kvv, kuv))
    else:
        A, B = 2 * U - 1 + 0 * V, 2 * V - 1 + 0 * U
        r2 = 1 + A * A + B * B  # the same for the six faces
        metric = [(4 / r2 * (1 - A * A / r2), 4 / r2 * (1 - B * B / r2), -4 / r2 * A * B / r2)] * 6
    out = []
    w = (gw[:, None] * gw[None, :]) / (nu * nv)
    for kuu, kvv, kuv in metric:
        a = np.sqrt(kuu * kvv - kuv * kuv)
        out.append((w * a, w * kvv / a, w * kuu / a, -w * kuv / a))
    conn, n = _connectivity(c)
    return conn, n, (bu, du, bv, dv), out


def _matrices(c):
    """(S, M) as float64 sparse CSR CUDA tensors."""
    conn, n, (bu, du, bv, dv), met = _space(c)
    nk = conn.shape[-1]
    t = lambda x: torch.tensor(np.ascontiguousarray(x), device=_DEV)  # noqa: E731
    rows, cols, vs, vm = [], [], [], []
    for f in range(conn.shape[0]):
        wa, g11, g22, g12 = (t(x) for x in met[f])
        fn = lambda y, x: torch.einsum("ygj,xhi->yxjigh", t(y), t(x)).reshape(  # noqa: E731
            conn.shape[1], conn.shape[2], nk, *wa.shape[2:])
        ph, pu, pv = fn(bv, bu), fn(bv, du), fn(dv, bu)
        vm.append(torch.einsum("yxkgh,yxgh,yxlgh->yxkl", ph, wa, ph).reshape(-1))
        fu, fv = g11[:, :, None] * pu + g12[:, :, None] * pv, g12[:, :, None] * pu + g22[:, :, None] * pv
        vs.append((torch.einsum("yxkgh,yxlgh->yxkl", pu, fu) + torch.einsum("yxkgh,yxlgh->yxkl", pv, fv)).reshape(-1))
        cn = t(conn[f].astype(np.int64))
        rows.append(cn[..., :, None].expand(*cn.shape, nk).reshape(-1))
        cols.append(cn[..., None, :].expand(*cn.shape[:-1], nk, nk).reshape(-1))
    idx = torch.stack([torch.cat(rows), torch.cat(cols)])
    return tuple(torch.sparse_coo_tensor(idx, torch.cat(v), (n, n)).coalesce().to_sparse_csr() for v in (vs, vm))


def _philox(c0, c1, c2, c3, seed):
    mask = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, dtype=np.uint64) for x in (c0, c1, c2, c3)]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for r in range(10):
        if r:
            k0, k1 = np.uint64((int(k0) + 0x9E3779B9) & 0xFFFFFFFF), np.uint64((int(k1) + 0xBB67AE85) & 0xFFFFFFFF)
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ k0, b & mask, (a >> np.uint64(32)) ^ c[3] ^ k1, a & mask]
    return c


def _normals(seed, sample, stream, n):
    """Philox Box–Muller normals 0..n-1 of a sample and stream."""
    q = np.arange((n + 1) // 2, dtype=np.uint64)
    o = _philox(q, np.full_like(q, sample), np.full_like(q, stream), np.zeros_like(q), seed)
    u = [((a >> np.uint64(5)) * np.uint64(1 << 26) + (b >> np.uint64(6)) + np.uint64(1)).astype(np.float64) * 2.0 ** -53
         for a, b in ((o[0], o[1]), (o[2], o[3]))]
    rad, ang = np.sqrt(-2 * np.log(u[0])), 2 * np.pi * u[1]
    return np.stack([rad * np.cos(ang), rad * np.sin(ang)], axis=1).reshape(-1)[:n]


def _loads(c, seed):
    """[ns, N] white-noise loads: sum over the Gauss points of sqrt(w a) xi phi."""
    conn, n, (bu, _, bv, _), met = _space(c)
    shape = (conn.shape[0],) + met[0][0].shape
    b = torch.zeros((c["ns"], n), dtype=torch.float64, device=_DEV)
    t = lambda x: torch.tensor(np.ascontiguousarray(x), device=_DEV)  # noqa: E731
    sw, idx = t(np.stack([np.sqrt(m[0]) for m in met])), t(conn.reshape(-1).astype(np.int64))
    bvt, but = t(bv), t(bu)
    for s in range(c["ns"]):
        xi = t(_normals(seed, s, 0, int(np.prod(shape))).reshape(shape)) * sw
        loc = torch.einsum("ygj,xhi,fyxgh->fyxji", bvt, but, xi)
        b[s].index_add_(0, idx, loc.reshape(-1))
    return b


def _dense_fields(c, seed, S, M):
    """u of the drawn loads by dense Cholesky factors of every shifted matrix."""
    n_int, bf, passes = _split(c["beta"], c["split"])
    factor = lambda s: torch.linalg.cholesky(S + s * M)  # noqa: E731
    b = _loads(c, seed).T
    r = b
    if n_int:
        L = factor(c["kappa"] ** 2)
        for i in range(n_int):
            w = torch.cholesky_solve(r, L)
            r = M @ w
    else:
        w = None
    nodes = range(c["lo"], c["hi"] + 1) if passes else ()
    factors = {}
    for k in range(passes):
        acc = torch.zeros_like(b)
        for l in nodes:
            y = l * c["k"]
            if l not in factors:
                factors[l] = factor(math.exp(y) + c["kappa"] ** 2)
            acc += math.sin(math.pi * bf) / math.pi * c["k"] * math.exp((1 - bf) * y) * torch.cholesky_solve(r, factors[l])
            if k + 1 == passes:
                del factors[l]
        w = acc
        r = M @ w
    return w.T.contiguous()


def _sqrt_loads(c, seed, M):
    """sqrt(M) y by a Chebyshev expansion of sqrt on bounds of M's spectrum."""
    n = M.shape[0]
    y = torch.tensor(np.stack([_normals(seed, s, 2, n) for s in range(c["ns"])]), device=_DEV).T.contiguous()
    x = torch.ones((n, 1), dtype=torch.float64, device=_DEV)
    hi = float((M @ x).max()) * 1.0001  # non-negative entries: the largest row sum
    # the smallest eigenvalue from power iterations on hi I - M, with room
    v = _normal((n, 8), 1)
    for _ in range(400):
        v = hi * v - M @ v
        v /= v.norm(dim=0)
    lo = 0.3 * float((v * (M @ v)).sum(0).min())
    deg = int(min(6000, 18 * math.sqrt(hi / lo)))
    th = (np.arange(deg + 1) + 0.5) * np.pi / (deg + 1)
    f = np.sqrt((hi + lo) / 2 + (hi - lo) / 2 * np.cos(th))
    co = np.array([2.0 / (deg + 1) * np.dot(f, np.cos(k * th)) for k in range(deg + 1)])
    A = lambda z: (2 * (M @ z) - (hi + lo) * z) / (hi - lo)  # noqa: E731
    t0, t1 = y, A(y)
    out = co[0] / 2 * t0 + co[1] * t1
    for k in range(2, deg + 1):
        t0, t1 = t1, 2 * A(t1) - t0
        out += co[k] * t1
    return out.T.contiguous()


@functools.lru_cache(maxsize=2)
def _dense(kind, p, nu, nv):
    S, M = _matrices(dict(kind=kind, p=p, nu=nu, nv=nv))
    return S.to_dense(), M.to_dense()


# largest dense problem worked out (its 70-odd factorisations take some seconds)
_MOST_DENSE = 7000


def exact(case, seed):
    c = case
    if c["op"] == "loads":
        return _loads(c, seed)
    if c["op"] == "mass":
        x = _normal((c["ns"], _dofs(c)), seed)
        return (_matrices(c)[1] @ x.T.contiguous()).T.contiguous()
    if c["op"] == "sqrt":
        return _sqrt_loads(c, seed, _matrices(c)[1])
    if c["op"] == "fields" and _dofs(c) <= _MOST_DENSE:
        return _dense_fields(c, seed, *_dense(c["kind"], c["p"], c["nu"], c["nv"]))
    if c["op"] == "batched":
        out = []
        for i, e in enumerate(_instances(c)):
            e = dict(e, split="improved", k=0.3, lo=-35, hi=35)
            # every instance that a dense factorisation does within a second
            out.append(_dense_fields(e, seed * 1000 + i, *_dense(e["kind"], e["p"], e["nu"], e["nv"]))
                       if _dofs(e) <= 2500 else None)
        return out
    return None

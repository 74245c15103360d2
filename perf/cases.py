"""Performance cases: the work a user of the library has it do, through its public binding.

The cases stand for the workloads the library is written for: the pipeline
from a point cloud to CSR operators (2D and 3D, the scalar, the
divergence-free and the staggered basis, degrees 2 to 4, plain FP64 and FP32 +
refinement, with and without Neumann targets), uneven batches of radius lists,
the request server, and the Stokes collocation system with its solve.

``exact`` restates the same results in 64 bits with torch alone.
"""
import math

import numpy as np
import torch

from paper_2104_14447_gb300 import gmls

EPS_FACTOR = 1.5
#: neighbours of a (dimension, basis, degree)
K = {(2, "scalar", 2): 12, (2, "scalar", 3): 20, (2, "scalar", 4): 36, (2, "divfree", 2): 22, (2, "divfree", 3): 34,
     (2, "divfree", 4): 48, (3, "scalar", 2): 20, (3, "scalar", 3): 40, (3, "scalar", 4): 84, (3, "divfree", 2): 42,
     (3, "divfree", 3): 80, (3, "divfree", 4): 136, (2, "staggered", 2): 24, (2, "staggered", 3): 36,
     (2, "staggered", 4): 48, (3, "staggered", 2): 40}
BASIS = {"scalar": gmls.SCALAR, "divfree": gmls.DIVFREE, "staggered": gmls.STAGGERED}
PRECISION = {"fp64": gmls.FP64, "fp32": gmls.FP32_REFINE}
RADIUS_FACTOR, RADIUS_CAP = 1.8, 160
SHAPES = [s for s in K if s[1] != "staggered"]


def listed():
    return [
        # the smallest call: one 1,024-target cloud, plain FP64 (launches and latency count)
        {"name": "operators_2d_small_fp64", "kind": "operators", "dim": 2, "axis": 32, "degree": 2, "divfree": False,
         "precision": "fp64"},
        # the operators of one 2D Stokes discretisation, FP32 + refinement
        {"name": "operators_2d_512", "kind": "operators", "dim": 2, "axis": 512, "degree": 4, "divfree": True,
         "precision": "fp32"},
        # the same in plain FP64, an odd and smaller grid
        {"name": "operators_2d_fp64", "kind": "operators", "dim": 2, "axis": 181, "degree": 4, "divfree": True,
         "precision": "fp64"},
        # a small 3D porous cloud, half of its points Neumann targets
        {"name": "porous_3d_20", "kind": "porous", "axis": 20, "precision": "fp32"},
        # the largest: the full porous medium, about 1.76 million targets
        {"name": "porous_3d_128", "kind": "porous", "axis": 128, "precision": "fp32"},
        # uneven batches: radius lists, a degree per target, one fifth one-sided
        {"name": "uneven_2d", "kind": "uneven", "dim": 2, "n": 500000, "precision": "fp32"},
        {"name": "uneven_3d", "kind": "uneven", "dim": 3, "n": 500000, "precision": "fp32"},
        # the request server: a burst with one request of every shape, results back to the host
        {"name": "serve_mixed", "kind": "serve", "mix": 1, "nmin": 1000, "nmax": 20000},
        # the stencil stage alone on lists at hand: the largest tile, and the staggered basis at an odd size
        {"name": "stencils_3d_divfree_m4", "kind": "stencils", "dim": 3, "basis": "divfree", "degree": 4, "axis": 31,
         "precision": "fp32"},
        {"name": "stencils_3d_staggered_m2", "kind": "stencils", "dim": 3, "basis": "staggered", "degree": 2,
         "axis": 47, "precision": "fp32"},
        # the Stokes block system from stencils at hand: assembly, right-hand side and one A x
        {"name": "stokes_system_2d", "kind": "system", "axis": 512},
        # cloud to solution: the 3D Stokes problem with quadratic data, GMRES to 1e-12
        {"name": "stokes_solve_3d", "kind": "solve", "axis": 24},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["operators", "operators", "porous", "uneven", "serve", "stencils", "stencils", "system", "solve"])
    if kind == "operators":
        dim, fp64 = rng.choice([2, 3]), rng.random() < 0.35
        degree = rng.choice([2, 3, 4] if dim == 2 else [2, 3])
        n = _log_uniform(rng, 1000, (30000 if dim == 2 else 5000) if fp64 else (260000 if dim == 2 else 60000))
        return {"kind": kind, "dim": dim, "axis": max(10, round(n ** (1.0 / dim))), "degree": degree,
                "divfree": rng.random() < 0.7, "precision": "fp64" if fp64 else "fp32"}
    if kind == "porous":
        return {"kind": kind, "axis": _log_uniform(rng, 16, 96), "precision": "fp32"}
    if kind == "uneven":
        return {"kind": kind, "dim": rng.choice([2, 3]), "n": _log_uniform(rng, 5000, 300000), "precision": "fp32"}
    if kind == "serve":
        nmax = _log_uniform(rng, 4000, 20000)
        return {"kind": kind, "mix": rng.randrange(1, 1 << 20), "nmin": 1000, "nmax": nmax}
    if kind == "stencils":
        dim, basis, degree = rng.choice(sorted(K))
        fp64 = rng.random() < 0.25
        heavy = dim == 3 and basis == "divfree"
        top = (4000 if heavy else 20000) if fp64 else (40000 if heavy else 250000)
        n = _log_uniform(rng, 1000, top)
        return {"kind": kind, "dim": dim, "basis": basis, "degree": degree, "axis": max(10, round(n ** (1.0 / dim))),
                "precision": "fp64" if fp64 else "fp32"}
    if kind == "system":
        return {"kind": kind, "axis": _log_uniform(rng, 64, 512)}
    return {"kind": kind, "axis": rng.randrange(8, 25)}


# ------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _lattice(dim, axis, gen):
    """Jittered lattice in the unit cube, x fastest, jitter U(-h/4, h/4); and the lattice indices."""
    h = 1.0 / axis
    i = torch.arange(axis ** dim, device="cuda")
    ix = torch.stack([(i // axis ** c) % axis for c in range(dim)])
    u = torch.rand(ix.shape, generator=gen, device="cuda", dtype=torch.float64)
    return (ix + 0.5) * h + (2.0 * u - 1.0) * (0.25 * h), ix


def _box_boundary(ix, axis):
    nrm = (ix == axis - 1).double() - (ix == 0).double()
    length = nrm.square().sum(0).sqrt()
    flag = (length > 0).to(torch.uint8)
    return flag, (nrm / length.clamp(min=1.0)).contiguous()


def _porous(axis, gen):
    """A jittered lattice in the unit cube minus 64 non-overlapping spheres (the same for every jitter):
    points near a sphere are projected onto it, boundary points (spheres and cube faces) carry the fluid's
    outward normal."""
    h = 1.0 / axis
    rng = np.random.RandomState(0)
    spheres = []
    while len(spheres) < 64:
        r = 0.05 + 0.07 * rng.rand()
        c = r + (1.0 - 2.0 * r) * rng.rand(3)
        if all(np.sum((c - s[0]) ** 2) > (r + s[1]) ** 2 for s in spheres):
            spheres.append((c, r))
    x, ix = _lattice(3, axis, gen)
    keep = torch.ones(x.shape[1], dtype=torch.bool, device="cuda")
    flag = torch.zeros(x.shape[1], dtype=torch.uint8, device="cuda")
    nrm = torch.zeros_like(x)
    for c, rad in spheres:
        # the lattice site says which points stay and which lie on the sphere, the jittered point where
        ctr = torch.from_numpy(c).cuda()[:, None]
        site = ((ix + 0.5) * h - ctr).square().sum(0).sqrt()
        keep &= site >= rad
        near = (site >= rad) & (site < rad + 0.5 * h)
        d = x - ctr
        u = d / d.square().sum(0).sqrt()
        x = torch.where(near, ctr + rad * u, x)
        nrm = torch.where(near, -u, nrm)
        flag[near] = 1
    for c in range(3):
        for layer, sign in ((0, -1.0), (axis - 1, 1.0)):
            on = (ix[c] == layer) & (flag == 0)
            nrm[c, on] = sign
            flag[on] = 1
    return x[:, keep].contiguous(), flag[keep].contiguous(), nrm[:, keep].contiguous()


def _functionals(basis):
    return [gmls.VEC_LAPLACIAN] if basis == "divfree" else [gmls.GRAD, gmls.LAPLACIAN]


def _basis_size(dim, basis, degree):
    full = math.comb(degree + dim, dim)
    if basis == "scalar":
        return full
    if basis == "staggered":
        return math.comb(degree + 1 + dim, dim) - 1
    return dim * full - math.comb(degree - 1 + dim, dim)


def _requests(case):
    """(shape, points per axis) of each request: one of every shape, sizes log-uniform."""
    rng = np.random.RandomState(case["mix"])
    n = np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]), len(SHAPES)))
    return [(s, max(6, int(round(v ** (1.0 / s[0]))))) for s, v in zip(SHAPES, n)]


def _arena(n, per_target):
    return (3 << 29) + int(1.25 * n * per_target)


def _bytes_per_target(dim, basis, degree):
    k = K[dim, basis, degree]
    rows = dim * dim if basis == "divfree" else dim + 1
    return k * rows * 8 + k * 16 + 256


def _inputs(case, seed):
    """The case's data on the device (the server's on the host)."""
    gen, kind = _generator(seed), case["kind"]
    if kind in ("operators", "stencils"):
        return {"x": _lattice(case["dim"], case["axis"], gen)[0]}
    if kind == "porous":
        x, flag, nrm = _porous(case["axis"], gen)
        return {"x": x, "flag": flag, "normals": nrm}
    if kind == "uneven":
        dim, n = case["dim"], case["n"]
        x = _lattice(dim, math.ceil(n ** (1.0 / dim) - 1e-9), gen)[0][:, :n].contiguous()
        deg = torch.randint(2, 5, (n,), generator=gen, device="cuda").to(torch.int8)
        nrm = torch.randn((n, dim), generator=gen, device="cuda", dtype=torch.float64)
        nrm /= nrm.square().sum(1, keepdim=True).sqrt()
        nrm[(nrm * (x.mean(1) - x.T)).sum(1) > 0] *= -1.0  # the kept side holds the inside of the cloud
        nrm[torch.rand(n, generator=gen, device="cuda") >= 0.2] = 0.0
        q = torch.tensor([0, 0] + [_basis_size(dim, "scalar", m) for m in (2, 3, 4)], dtype=torch.int32, device="cuda")
        return {"x": x, "degree": deg, "halfspace": nrm, "k": q[deg.long()]}
    if kind == "serve":
        return {"clouds": [_lattice(s[0], axis, gen)[0].cpu().numpy() for s, axis in _requests(case)]}
    if kind == "system":
        x, ix = _lattice(2, case["axis"], gen)
        flag, nrm = _box_boundary(ix, case["axis"])
        f, w = (torch.randn(x.shape, generator=gen, device="cuda", dtype=torch.float64) for _ in range(2))
        n = x.shape[1]
        return {"x": x, "flag": flag, "normals": nrm, "f": f, "w": w,
                "div_f": torch.randn(n, generator=gen, device="cuda", dtype=torch.float64),
                "v": torch.randn(3 * n + 1, generator=gen, device="cuda", dtype=torch.float64)}
    x, ix = _lattice(3, case["axis"], gen)
    x = 2.0 * x - 1.0
    flag, nrm = _box_boundary(ix, case["axis"])
    u, p, f, div_f = _quadratic(x)
    return {"x": x, "flag": flag, "normals": nrm, "f": f, "w": u, "div_f": div_f}


def _quadratic(x):
    """A divergence-free quadratic velocity, a quadratic pressure, f = curl curl u + grad p and div f."""
    X, Y, Z = x
    one = torch.ones_like(X)
    u = torch.stack([Y * Y + Y * Z, X * X + Z * Z, X * Y + X * X])
    p = X * X - Y * Z + 2.0 * X * Z + Y - 1.0
    f = torch.stack([2.0 * X + 2.0 * Z - 2.0, -Z + 1.0 - 4.0, -Y + 2.0 * X - 2.0 * one])
    return u, p, f, 2.0 * one


# ----------------------------------------------------------------- the calls
def prepare(case, seed):
    """The inputs and the handle (a context or a server with its memory) that a program keeps; for the
    stencil stage and the Stokes system also the lists or stencils it starts from."""
    d, kind = _inputs(case, seed), case["kind"]
    s = {"case": dict(case), "in": d}
    if kind == "serve":
        s["server"] = gmls.Server(0, arena_bytes=8 << 30, streams=4, max_inflight=8)
        return s
    n = d["x"].shape[1]
    if kind == "operators":
        need = _bytes_per_target(case["dim"], "scalar", case["degree"])
        need += _bytes_per_target(case["dim"], "divfree", case["degree"]) if case["divfree"] else 0
    elif kind == "porous":
        need = _bytes_per_target(3, "scalar", 3) + _bytes_per_target(3, "divfree", 3)
    elif kind == "uneven":
        need = RADIUS_CAP * ((case["dim"] + 1) * 8 + 16) + 256
    elif kind == "stencils":
        need = _bytes_per_target(case["dim"], case["basis"], case["degree"])
    elif kind == "system":
        need = 2 * (_bytes_per_target(2, "scalar", 4) + _bytes_per_target(2, "divfree", 4))
    else:
        need = 2 * (_bytes_per_target(3, "scalar", 2) + _bytes_per_target(3, "divfree", 2)) + 110 * 4 * 8
    ctx = s["ctx"] = gmls.Context(0, arena_bytes=_arena(n, need))
    if kind == "stencils":
        s["lists"] = ctx.neighbors(ctx.cloud(d["x"]), K[case["dim"], case["basis"], case["degree"]], EPS_FACTOR)
    elif kind == "uneven":  # operator buffers for the longest lists, kept from batch to batch
        s["out"] = [(torch.zeros(rows * n + 1, dtype=torch.int64, device="cuda"),
                     torch.zeros(rows * n * RADIUS_CAP, dtype=torch.int32, device="cuda"),
                     torch.zeros(rows * n * RADIUS_CAP, dtype=torch.float64, device="cuda")) for rows in (case["dim"], 1)]
    elif kind == "system":
        s["stencils"] = _stokes_stencils(ctx, d, 2, 4)[-2:]
    return s


def _stokes_stencils(ctx, d, dim, degree):
    cid = ctx.cloud(d["x"], normals=d["normals"], bflags=d["flag"])
    nv = ctx.neighbors(cid, K[dim, "divfree", degree], EPS_FACTOR)
    npr = ctx.neighbors_prefix(nv, K[dim, "scalar", degree], EPS_FACTOR)
    sv = ctx.stencils(nv, gmls.DIVFREE, degree, [gmls.CURLCURL], precision=gmls.FP32_REFINE)
    sp = ctx.stencils(npr, gmls.SCALAR, degree, [gmls.GRAD, gmls.LAPLACIAN], precision=gmls.FP32_REFINE, neumann=True)
    return cid, nv, npr, sv, sp


def run(state):
    return {"operators": _run_operators, "porous": _run_porous, "uneven": _run_uneven, "serve": _run_serve,
            "stencils": _run_stencils, "system": _run_system, "solve": _run_solve}[state["case"]["kind"]](state)


def _operators(ctx, wanted, handles):
    out = {}
    for name, sid, fn in wanted:
        rp, col, val = ctx.assemble_csr(sid, fn)
        out[name] = {"row_ptr": rp, "col": col, "val": val}
    for h in handles:
        ctx.release(h)
    return out


def _run_operators(s):
    """Cloud, lists, stencils and CSR operators."""
    c, ctx = s["case"], s["ctx"]
    dim, degree, prec = c["dim"], c["degree"], PRECISION[c["precision"]]
    cid = ctx.cloud(s["in"]["x"])
    ks = K[dim, "scalar", degree]
    if not c["divfree"]:
        nid = ctx.neighbors(cid, ks, EPS_FACTOR)
        ssc = ctx.stencils(nid, gmls.SCALAR, degree, [gmls.LAPLACIAN, gmls.GRAD], precision=prec)
        return _operators(ctx, [("lap", ssc, gmls.LAPLACIAN), ("grad", ssc, gmls.GRAD)], (ssc, nid, cid))
    nv = ctx.neighbors(cid, K[dim, "divfree", degree], EPS_FACTOR)
    npr = ctx.neighbors_prefix(nv, ks, EPS_FACTOR)
    ssc = ctx.stencils(npr, gmls.SCALAR, degree, [gmls.GRAD, gmls.DIV], precision=prec)
    sdf = ctx.stencils(nv, gmls.DIVFREE, degree, [gmls.VEC_LAPLACIAN], precision=prec)
    return _operators(ctx, [("grad", ssc, gmls.GRAD), ("div", ssc, gmls.DIV), ("vec_lap", sdf, gmls.VEC_LAPLACIAN)],
                      (sdf, ssc, npr, nv, cid))


def _run_porous(s):
    """The porous medium's step: Neumann-constrained scalar and divergence-free operators of degree 3."""
    ctx, d, prec = s["ctx"], s["in"], PRECISION[s["case"]["precision"]]
    cid = ctx.cloud(d["x"], normals=d["normals"], bflags=d["flag"])
    nv = ctx.neighbors(cid, K[3, "divfree", 3], EPS_FACTOR)
    npr = ctx.neighbors_prefix(nv, K[3, "scalar", 3], EPS_FACTOR)
    ssc = ctx.stencils(npr, gmls.SCALAR, 3, [gmls.GRAD, gmls.LAPLACIAN], precision=prec, neumann=True)
    sdf = ctx.stencils(nv, gmls.DIVFREE, 3, [gmls.VEC_LAPLACIAN], precision=prec)
    return _operators(ctx, [("grad", ssc, gmls.GRAD), ("lap", ssc, gmls.LAPLACIAN), ("vec_lap", sdf, gmls.VEC_LAPLACIAN)],
                      (sdf, ssc, npr, nv, cid))


def _run_uneven(s):
    """Radius lists with a neighbour count, a degree and (one fifth) a half-space per target."""
    c, ctx, d = s["case"], s["ctx"], s["in"]
    cid = ctx.cloud(d["x"])
    nid = ctx.neighbors(cid, _basis_size(c["dim"], "scalar", 4), RADIUS_FACTOR, mode=gmls.RADIUS, cap=RADIUS_CAP,
                        halfspace=d["halfspace"], k_per_target=d["k"])
    sid = ctx.stencils(nid, gmls.SCALAR, 0, [gmls.GRAD, gmls.LAPLACIAN], precision=PRECISION[c["precision"]],
                       degree_per_target=d["degree"])
    out = {}
    for name, fn, buf in (("grad", gmls.GRAD, s["out"][0]), ("lap", gmls.LAPLACIAN, s["out"][1])):
        rp, col, val = ctx.assemble_csr(sid, fn, out=buf)
        out[name] = {"row_ptr": rp, "col": col, "val": val}
    for h in (sid, nid, cid):
        ctx.release(h)
    return out


def _run_serve(s):
    """A burst of requests; every result is fetched to the host."""
    srv = s["server"]
    reqs = _requests(s["case"])
    tickets = [srv.submit(x, BASIS[shape[1]], shape[2], K[shape], _functionals(shape[1]), eps_factor=EPS_FACTOR)
               for (shape, _), x in zip(reqs, s["in"]["clouds"])]
    out = []
    for (shape, _), t in zip(reqs, tickets):
        srv.wait(t)
        out.append([srv.result(t, gmls.X_WEIGHTS, torch.float64, fn) for fn in _functionals(shape[1])])
        srv.release(t)
    return out


def _run_stencils(s):
    c, ctx = s["case"], s["ctx"]
    sid = ctx.stencils(s["lists"], BASIS[c["basis"]], c["degree"], _functionals(c["basis"]),
                       precision=PRECISION[c["precision"]])
    out = [ctx.weights(sid, fn) for fn in _functionals(c["basis"])]
    ctx.release(sid)
    return out


def _run_system(s):
    """Block assembly, right-hand side and one matrix-vector product."""
    ctx, d, (sv, sp) = s["ctx"], s["in"], s["stencils"]
    rp, col, val = ctx.stokes_assemble(sv, sp, 1.0)
    b = ctx.stokes_rhs(sv, sp, 1.0, d["f"], d["w"], d["div_f"])
    return {"row_ptr": rp, "col": col, "val": val, "b": b, "y": ctx.spmv(rp, col, val, d["v"])}


def _run_solve(s):
    """Cloud to solution: lists, stencils, block system, GMRES on the equilibrated rows."""
    ctx, d = s["ctx"], s["in"]
    cid, nv, npr, sv, sp = _stokes_stencils(ctx, d, 3, 2)
    rp, col, val = ctx.stokes_assemble(sv, sp, 1.0)
    b = ctx.stokes_rhs(sv, sp, 1.0, d["f"], d["w"], d["div_f"])
    x, _, _ = ctx.gmres(rp, col, val, b, restart=100, max_iter=20000, rtol=1e-12, row_scaling=True)
    for h in (sp, sv, npr, nv, cid):
        ctx.release(h)
    return {"x": x, "row_ptr": rp, "col": col, "val": val, "b": b}


# ----------------------------------------------------- bytes and operations
def _stencil_flops(dim, basis, degree, k):
    """Householder QR of the weighted basis matrix, the apply of each functional row and, for one
    refinement step, its residual."""
    m, n = k * (dim if basis == "divfree" else 1), _basis_size(dim, basis, degree)
    rows = dim if basis == "divfree" else dim + 1
    return 2 * m * n * n - 2 * n ** 3 / 3 + rows * (n * n + 8 * m * n)


def work(case):
    kind = case["kind"]
    if kind in ("operators", "porous"):
        dim, degree = (3, 3) if kind == "porous" else (case["dim"], case["degree"])
        n = case["axis"] ** dim * (0.84 if kind == "porous" else 1.0)
        ks, kv = K[dim, "scalar", degree], K[dim, "divfree", degree]
        divfree = kind == "porous" or case["divfree"]
        nnz = ks * (2 * dim if kind == "operators" and divfree else dim + 1) + (kv * dim * dim if divfree else 0)
        flops = _stencil_flops(dim, "scalar", degree, ks) + (_stencil_flops(dim, "divfree", degree, kv) if divfree else 0)
        return {"bytes": n * (8 * dim + 12 * nnz + 8 * (2 * dim + 1)), "flops": n * flops}
    if kind == "uneven":
        dim, n = case["dim"], case["n"]
        ks = {m: min(RADIUS_CAP, RADIUS_FACTOR ** dim * _basis_size(dim, "scalar", m)) for m in (2, 3, 4)}
        flops = sum(_stencil_flops(dim, "scalar", m, k) for m, k in ks.items()) / 3
        return {"bytes": n * (16 * dim + 5 + 12 * (dim + 1) * sum(ks.values()) / 3 + 8 * (dim + 1)), "flops": n * flops}
    if kind == "serve":
        b = f = 0
        for (dim, basis, degree), axis in _requests(case):
            n, k = axis ** dim, K[dim, basis, degree]
            b += n * (8 * dim + 8 * k * (dim * dim if basis == "divfree" else dim + 1))
            f += n * _stencil_flops(dim, basis, degree, k)
        return {"bytes": b, "flops": f}
    if kind == "stencils":
        dim, basis, degree = case["dim"], case["basis"], case["degree"]
        n, k = case["axis"] ** dim, K[dim, basis, degree]
        rows = dim * dim if basis == "divfree" else dim + 1
        return {"bytes": n * (8 * dim + 8 + 4 * k + 8 * k * rows), "flops": n * _stencil_flops(dim, basis, degree, k)}
    if kind == "system":
        n = case["axis"] ** 2
        nnz = n * (2 * (48 * 2 + 36) + 36 + 2)
        return {"bytes": nnz * 8 + nnz * 12 + nnz * 12 + n * (84 * 4 + 8 * 5 + 3 * 8 * 4), "flops": 2.0 * nnz}
    n = case["axis"] ** 3
    nnz, its, size = n * (3 * (42 * 3 + 20) + 20 + 2), 9.8 * case["axis"], 4 * n
    return {"bytes": n * 8 * 14 + 12 * nnz + 8 * 3 * size,
            "flops": its * (2 * nnz + 8 * size * 50) + n * (_stencil_flops(3, "divfree", 2, 42) + _stencil_flops(3, "scalar", 2, 20))}


# ------------------------------------------------------- the same in 64 bits
EXACT_POINTS = 270000


def _knn(x, k, halfspace=None):
    """The k nearest by (d^2, id), all pairs; entries outside the half-space or the cloud have d^2 = inf."""
    dim, n = x.shape
    idx = torch.empty((n, k), dtype=torch.int64, device="cuda")
    d2 = torch.empty((n, k), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // n)
    for a in range(0, n, step):
        t = x[:, a:a + step]
        d = [x[c][None, :] - t[c][:, None] for c in range(dim)]
        r = d[0] * d[0] + d[1] * d[1]
        r = r + d[2] * d[2] if dim == 3 else r
        if halfspace is not None:
            dot = sum(halfspace[a:a + step, c, None] * d[c] for c in range(dim))
            r = torch.where(dot <= 0, r, math.inf)
        got = torch.topk(r, min(k, n), dim=1, largest=False, sorted=True)
        d2[a:a + step], idx[a:a + step] = got.values, got.indices
    return idx, d2


def _exponents(dim, lo, hi):
    if dim == 2:
        return [(a, s - a) for s in range(lo, hi + 1) for a in range(s, -1, -1)]
    return [(a, b, s - a - b) for s in range(lo, hi + 1) for a in range(s, -1, -1) for b in range(s - a, -1, -1)]


def _divergence_free(dim, degree):
    """Orthonormal coefficients [component][monomial][function] of the divergence-free fields."""
    e, low = _exponents(dim, 0, degree), _exponents(dim, 0, degree - 1)
    div = torch.zeros((len(low), dim, len(e)), dtype=torch.float64, device="cuda")
    for c in range(dim):
        for i, b in enumerate(e):
            if b[c]:
                div[low.index(tuple(v - (j == c) for j, v in enumerate(b))), c, i] = 1.0
    nb = _basis_size(dim, "divfree", degree)
    return torch.linalg.svd(div.reshape(len(low), -1)).Vh[-nb:].T.reshape(dim, len(e), nb).contiguous()


def _solve_rows(B, lam):
    """rows[t] of Q R^-T lam^T for B = Q R: Gram-Schmidt, every column orthogonalised twice."""
    n = B.shape[2]
    Q, R = B.clone(), torch.zeros((B.shape[0], n, n), dtype=B.dtype, device=B.device)
    for j in range(n):
        v = Q[:, :, j:j + 1]
        for _ in range(2 if j else 0):
            h = Q[:, :, :j].transpose(1, 2) @ v
            v = v - Q[:, :, :j] @ h
            R[:, :j, j:j + 1] += h
        R[:, j, j] = v[:, :, 0].square().sum(1).sqrt()
        Q[:, :, j:j + 1] = v / R[:, j, j][:, None, None]
    z = torch.linalg.solve_triangular(R.transpose(1, 2), lam.transpose(1, 2), upper=False)
    return (Q @ z).transpose(1, 2)


def _weights(x, idx, mask, eps, basis, degree, rows, tgt=None, normals=None):
    """Stencil weights [target][row][neighbour][component] and beta [target][row]; rows: "grad", "lap" or
    "vec_lap", one after another; normals (zero for free targets) add the Neumann constraint."""
    dim, (n, k) = x.shape[0], idx.shape
    e = _exponents(dim, 1, degree + 1) if basis == "staggered" else _exponents(dim, 0, degree)
    unit = [tuple(int(i == c) for i in range(dim)) for c in range(dim)]
    C = _divergence_free(dim, degree) if basis == "divfree" else None
    nb = C.shape[2] if C is not None else len(e)
    nc = dim if basis == "divfree" else 1
    nrows = sum({"grad": dim, "lap": 1, "vec_lap": dim}[r] for r in rows)
    out = torch.empty((n, nrows, k, nc), dtype=torch.float64, device="cuda")
    beta = torch.zeros((n, nrows), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // (k * nc * nb))
    for a in range(0, n, step):
        t = torch.arange(a, min(n, a + step), device="cuda") if tgt is None else tgt[a:a + step]
        ep = eps[a:a + step]
        d = (x[:, idx[a:a + step]] - x[:, t][:, :, None]) / ep[None, :, None]
        r = d.square().sum(0).sqrt()
        sw = (1.0 - r).clamp(min=0.0) ** 2 * mask[a:a + step]
        P = torch.stack([math.prod(d[c] ** b[c] for c in range(dim)) / math.prod(math.factorial(v) for v in b) for b in e], 2)
        lam = []
        for name in rows:
            if name == "grad":
                for c in range(dim):
                    v = torch.zeros((len(t), len(e)), dtype=torch.float64, device="cuda")
                    v[:, e.index(unit[c])] = 1.0 / ep
                    lam.append(v)
            elif name == "lap":
                v = torch.zeros((len(t), len(e)), dtype=torch.float64, device="cuda")
                for c in range(dim):
                    v[:, e.index(tuple(2 * u for u in unit[c]))] = 1.0 / ep ** 2
                lam.append(v)
            else:
                for q in range(dim):
                    lam.append(sum(C[q, e.index(tuple(2 * u for u in unit[c]))] for c in range(dim)) / ep[:, None] ** 2)
        lam = torch.stack(lam, 1)
        if C is not None:
            B = torch.einsum("tkq,cqn->tkcn", P * sw[:, :, None], C).reshape(len(t), k * dim, nb)
            out[a:a + step] = _solve_rows(B, lam).reshape(len(t), nrows, k, dim) * sw[:, None, :, None]
            continue
        B = P * sw[:, :, None]
        if normals is None:
            w = _solve_rows(B, lam)
        else:
            # a reflector turns n . grad into a multiple of the first linear coefficient, which the
            # constraint then fixes: the fit takes the remaining columns
            w = torch.empty((len(t), nrows, k), dtype=torch.float64, device="cuda")
            nr = normals[:, t].T
            on = nr.square().sum(1) > 0
            if (~on).any():
                w[~on] = _solve_rows(B[~on], lam[~on])
            if on.any():
                v = nr[on].clone()
                s = torch.where(v[:, 0] >= 0, 1.0, -1.0).double()
                v[:, 0] += s
                H = torch.eye(dim, dtype=torch.float64, device="cuda") - 2.0 * v[:, :, None] * v[:, None, :] / v.square().sum(1)[:, None, None]
                lin = [e.index(u) for u in unit]
                Bn, ln = B[on].clone(), lam[on].clone()
                Bn[:, :, lin] = Bn[:, :, lin] @ H
                ln[:, :, lin] = ln[:, :, lin] @ H
                rest = [i for i in range(nb) if i != lin[0]]
                wn = _solve_rows(Bn[:, :, rest], ln[:, :, rest])
                w[on] = wn
                # n . grad q = -s c_1 / eps, so c_1 = -s eps h
                left = ln[:, :, lin[0]] - (wn @ Bn[:, :, lin[0]][:, :, None])[:, :, 0]
                bt = torch.zeros((len(t), nrows), dtype=torch.float64, device="cuda")
                bt[on] = -s[:, None] * ep[on][:, None] * left
                beta[a:a + step] = bt
        w = w * sw[:, None, :]
        if basis == "staggered":  # the fit is to differences from the target's own value (neighbour 0)
            w[:, :, 0] = 0.0
            w[:, :, 0] = -w.sum(2)
        out[a:a + step] = w[:, :, :, None]
    return out, beta


def _by_id(w, idx, mask=None):
    """Operator values: the rows' entries in the order of the neighbours' ids."""
    key = idx if mask is None else torch.where(mask, idx, 1 << 40)
    order = torch.argsort(key, dim=1)
    w = torch.gather(w, 2, order[:, None, :, None].expand(w.shape))
    if mask is None:
        return w.reshape(-1)
    m = torch.gather(mask, 1, order)
    return w[m[:, None, :, None].expand(w.shape)]


def _values(val):
    return {"row_ptr": None, "col": None, "val": val}


def exact(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    if kind == "solve":
        u, p, _, _ = _quadratic(d["x"])
        return {"x": torch.cat([u.T.reshape(-1), p - p.mean(), p.new_zeros(1)]), "row_ptr": None, "col": None, "val": None,
                "b": None}
    if kind == "serve":
        if case["nmax"] > EXACT_POINTS:
            return None
        out = []
        for (shape, _), x in zip(_requests(case), d["clouds"]):
            out.append([v.reshape(-1).cpu() for v in _stage(torch.from_numpy(x).cuda(), *shape)])
        return out
    x = d["x"]
    n = x.shape[1]
    if n > EXACT_POINTS:
        return None
    if kind == "stencils":
        return [v.reshape(-1) for v in _stage(x, case["dim"], case["basis"], case["degree"])]
    if kind == "uneven":
        return _exact_uneven(case, d)
    dim, degree = (3, 3) if kind == "porous" else (2, 4) if kind == "system" else (case["dim"], case["degree"])
    ks, kv = K[dim, "scalar", degree], K[dim, "divfree", degree]
    idx, d2 = _knn(x, max(ks, kv))
    every = torch.ones_like(idx, dtype=torch.bool)
    eps = {k: EPS_FACTOR * d2[:, k - 1].sqrt() for k in (ks, kv)}
    nrm = d["normals"] * d["flag"] if kind in ("porous", "system") else None
    sc, beta = _weights(x, idx[:, :ks], every[:, :ks], eps[ks], "scalar", degree, ["grad", "lap"], normals=nrm)
    if kind == "operators" and not case["divfree"]:
        return {"lap": _values(_by_id(sc[:, dim:], idx[:, :ks])), "grad": _values(_by_id(sc[:, :dim], idx[:, :ks]))}
    df, _ = _weights(x, idx[:, :kv], every[:, :kv], eps[kv], "divfree", degree, ["vec_lap"])
    if kind == "system":
        return _exact_system(d, idx, ks, kv, sc, beta, df)
    out = {"grad": _values(_by_id(sc[:, :dim], idx[:, :ks])), "vec_lap": _values(_by_id(df, idx[:, :kv]))}
    if kind == "porous":
        out["lap"] = _values(_by_id(sc[:, dim:], idx[:, :ks]))
    else:  # the divergence: d/dx_c applied to component c
        out["div"] = _values(_by_id(sc[:, None, :dim, :, 0].transpose(2, 3), idx[:, :ks]))
    return out


def _stage(x, dim, basis, degree):
    """The weights of each functional of the stencil stage on the fixed lists."""
    k = K[dim, basis, degree]
    idx, d2 = _knn(x, k)
    rows = ["vec_lap"] if basis == "divfree" else ["grad", "lap"]
    w, _ = _weights(x, idx, torch.ones_like(idx, dtype=torch.bool), EPS_FACTOR * d2[:, -1].sqrt(), basis, degree, rows)
    return [w] if basis == "divfree" else [w[:, :dim], w[:, dim:]]


def _exact_uneven(case, d):
    x, dim, kt = d["x"], case["dim"], d["k"].long()
    idx, d2 = _knn(x, RADIUS_CAP, d["halfspace"])
    eps = RADIUS_FACTOR * torch.gather(d2, 1, kt[:, None] - 1)[:, 0].sqrt()
    mask = d2 < (eps * eps)[:, None]
    w = torch.empty((x.shape[1], dim + 1, RADIUS_CAP, 1), dtype=torch.float64, device="cuda")
    for m in (2, 3, 4):
        at = (d["degree"] == m).nonzero()[:, 0]
        w[at], _ = _weights(x, idx[at], mask[at], eps[at], "scalar", m, ["grad", "lap"], tgt=at)

    def buffer(rows):  # filled up to the last entry, then zeros
        v = _by_id(rows, idx, mask)
        return _values(torch.cat([v, v.new_zeros(rows.numel() - v.numel())]))

    return {"grad": buffer(w[:, :dim]), "lap": buffer(w[:, dim:])}


def _exact_system(d, idx, ks, kv, sc, beta, df):
    """The block system (nu = 1), its right-hand side and A v from the stencils: entries as (row, column,
    value), ordered by row and column."""
    x = d["x"]
    n = x.shape[1]
    pt = torch.arange(n, device="cuda")
    on = d["flag"] > 0
    inner, edge = (~on).nonzero()[:, 0], on.nonzero()[:, 0]
    cc, grad, lap, bt = -df, sc[:, :2, :, 0], sc[:, 2, :, 0], beta[:, 2]
    rows, cols, vals = [], [], []

    def put(r, c, v):
        r, c, v = torch.broadcast_tensors(r, c, v)
        rows.append(r.reshape(-1)), cols.append(c.reshape(-1)), vals.append(v.reshape(-1))

    one = torch.ones((), dtype=torch.float64, device="cuda")
    comp = torch.arange(2, device="cuda")
    vcol = idx[:, :kv, None] * 2 + comp
    for c in range(2):
        put((inner * 2 + c)[:, None, None], vcol[inner], cc[inner, c])
        put((inner * 2 + c)[:, None], 2 * n + idx[inner, :ks], grad[inner, c])
        put(edge * 2 + c, edge * 2 + c, one)
    put((2 * n + pt)[:, None], 2 * n + idx[:, :ks], lap)
    put(2 * n + pt, torch.full_like(pt, 3 * n), one)
    na = (d["normals"].T[:, :, None, None] * cc).sum(1)
    put((2 * n + edge)[:, None, None], vcol[edge], -bt[edge, None, None] * na[edge])
    put(torch.full_like(pt, 3 * n), 2 * n + pt, one)
    r, c, v = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    order = torch.argsort(r * (3 * n + 1) + c)
    r, c, v = r[order], c[order], v[order]
    y = torch.zeros(3 * n + 1, dtype=torch.float64, device="cuda").index_add_(0, r, v * d["v"][c])
    nf = (d["normals"] * d["f"]).sum(0)
    mom = torch.where(on, d["w"], d["f"]).T.reshape(-1)
    b = torch.cat([mom, d["div_f"] - torch.where(on, bt * nf, 0.0), mom.new_zeros(1)])
    return {"row_ptr": None, "col": None, "val": v, "b": b, "y": y}

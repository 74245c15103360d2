"""The semi-normal-equation stencil kernel (variant -5) against the FP64 kernel
over the forms it accepts: every basis, dimension and degree it is built for,
fewest and odd and long lists, sets and orders of functionals, weight powers,
target subsets, Neumann rows; and in bucketed launches (radius lists, a degree
per target).  Bars as for the other FP32 + refinement kernels: 1e-9 relative
per target and row, 1e-15 kappa for ill-conditioned ones (the FP64 kernel is
itself held to the oracle at 1e-10)."""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs
from tests.test_gpu_parity import test_neumann_matches_oracle as _neumann_matches_oracle

pytestmark = pytest.mark.gpu

G, L, D, V, C = gmls.GRAD, gmls.LAPLACIAN, gmls.DIV, gmls.VEC_LAPLACIAN, gmls.CURLCURL
S, F, T = gmls.SCALAR, gmls.DIVFREE, gmls.STAGGERED


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    build.build()
    c = gmls.Context(0, arena_bytes=6 << 30)
    c.set_option(gmls.OPT_POISON, 1)  # outputs start as NaN: unwritten entries cannot pass
    yield c
    c.close()


def _compare(ctx, nid, basis, m, fns, k, n, forced=True, **kw):
    """max over targets and rows of |w - w64| / (bar |w64|), and the FP32 run's status."""
    ref = ctx.stencils(nid, basis, m, fns, precision=gmls.FP64, **kw)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5 if forced else 0)
    try:
        sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE, **kw)
    finally:
        ctx.set_option(gmls.OPT_FORCE_VARIANT, 0)
    worst = 0.0
    st = ctx.export(sid, gmls.X_STATUS, torch.uint8)
    redone = (st & gmls.T_FP64_FALLBACK) != 0
    off = ctx.export(nid, gmls.X_NBR_OFFSETS, torch.int64)
    for fn in fns:
        _, rows, nc, _ = ctx.stencil_info(sid, fn)
        a, b = ctx.weights(sid, fn), ctx.weights(ref, fn)
        assert bool(torch.isfinite(a).all())
        # entry -> (target, row): rows of a target are consecutive
        ks = off[1:] - off[:-1]
        seg = torch.repeat_interleave(torch.arange(n * rows, device=a.device), (ks * nc).repeat_interleave(rows))
        err = torch.zeros(n * rows, device=a.device, dtype=torch.float64).scatter_reduce_(0, seg, (a - b).abs(), "amax")
        top = torch.zeros(n * rows, device=a.device, dtype=torch.float64).scatter_reduce_(0, seg, b.abs(), "amax")
        rel = (err / torch.where(top > 0, top, 1.0)).view(n, rows).amax(1)
        rel[redone] = 0.0  # the FP64 kernel's own result
        worst = max(worst, float(rel.max()) / 1e-9)
    ctx.release(sid)
    ctx.release(ref)
    return worst, st


# (dim, basis, degree, functionals, neighbours): fewest (or nearly), odd, long lists
UNIFORM = [(2, S, 2, [L, G], 9), (2, S, 2, [G], 13), (2, S, 3, [G, L], 15), (2, S, 3, [D], 20), (2, S, 4, [D, G], 36),
           (2, S, 4, [G, L], 27), (2, S, 4, [L, G, D], 73), (3, S, 2, [G, L], 17), (3, S, 2, [D], 61),
           (3, S, 3, [G, L], 33), (3, S, 3, [G], 40), (3, S, 3, [L, G], 125), (3, S, 4, [G, L], 57), (3, S, 4, [G], 160),
           (2, F, 2, [V], 12), (2, F, 2, [C], 40), (2, F, 3, [V, C], 19), (2, F, 4, [C, V, D], 48), (2, F, 4, [V], 29),
           (3, F, 2, [V], 23), (3, F, 3, [V], 80), (3, F, 3, [C], 41), (3, F, 4, [V], 136), (3, F, 4, [C], 71),
           (2, T, 2, [G, L], 24), (2, T, 2, [L], 17), (2, T, 3, [L, G], 36), (2, T, 4, [G, L], 48), (3, T, 2, [G, L], 41)]


@pytest.mark.parametrize("dim,basis,m,fns,k", UNIFORM)
def test_uniform_lists_match_fp64(ctx, dim, basis, m, fns, k):
    x = inputs.jittered_grid(dim, 23 if dim == 2 else 9, seed=m + k)
    n = x.shape[1]
    cid = ctx.cloud(x)
    nid = ctx.neighbors(cid, k, 1.5)
    worst, st = _compare(ctx, nid, basis, m, fns, k, n)
    assert worst <= 1.0
    assert int(((st & gmls.T_FP64_FALLBACK) != 0).sum()) <= n // 20
    for h in (nid, cid):
        ctx.release(h)


@pytest.mark.parametrize("power", [2, 6])
@pytest.mark.parametrize("dim,basis,m,fns,k", [(2, S, 4, [G, L], 36), (3, F, 3, [V], 80), (2, T, 3, [G, L], 36)])
def test_weight_powers_and_target_subsets(ctx, dim, basis, m, fns, k, power):
    x = inputs.jittered_grid(dim, 23 if dim == 2 else 9, seed=power) * 3.0 - 7.0
    cid = ctx.cloud(x)
    for n in (1, 5, 131):
        tg = ((np.arange(n) * 37) % x.shape[1]).astype(np.int32)
        nid = ctx.neighbors(cid, k, 1.5, targets=tg)
        worst, _ = _compare(ctx, nid, basis, m, fns, k, n, weight_power=power)
        assert worst <= 1.0, n
        ctx.release(nid)
    ctx.release(cid)


@pytest.mark.parametrize("dim,m,k", [(2, 2, 13), (2, 3, 21), (2, 4, 36), (3, 2, 20), (3, 3, 41), (3, 4, 84)])
def test_neumann_rows_match_fp64(ctx, dim, m, k):
    x = inputs.jittered_grid(dim, 25 if dim == 2 else 10, seed=m)
    n = x.shape[1]
    nrm = inputs.unit_vectors(5, 6, n, dim) * (0.5 + inputs.uniform(5, 7, n))  # any length
    bflag = (inputs.uniform(5, 8, n) < 0.3).astype(np.uint8)
    cid = ctx.cloud(x, normals=nrm, bflags=bflag)
    nid = ctx.neighbors(cid, k, 1.5)
    worst, st = _compare(ctx, nid, S, m, [G, L], k, n, neumann=True)
    assert worst <= 1.0
    assert int(((st & gmls.T_FP64_FALLBACK) != 0).sum()) <= n // 20
    for h in (nid, cid):
        ctx.release(h)


@pytest.mark.parametrize("dim,n_axis,m,k", [(2, 24, 2, 12), (2, 24, 4, 36), (3, 10, 3, 40)])
def test_neumann_weights_and_beta_match_oracle(ctx, dim, n_axis, m, k):
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5)
    try:
        _neumann_matches_oracle(ctx, dim, n_axis, m, k, gmls.FP32_REFINE)
    finally:
        ctx.set_option(gmls.OPT_FORCE_VARIANT, 0)


@pytest.mark.parametrize("dim,basis,fns", [(2, S, [G, L]), (3, S, [G]), (2, F, [V]), (3, F, [C]), (2, T, [G, L])])
def test_bucketed_launches_match_fp64(ctx, dim, basis, fns):
    """Radius lists of every length (some with fewer neighbours than basis
    functions), a degree per target; one target more or less changes no other
    target's weights."""
    x = inputs.jittered_grid(dim, 26 if dim == 2 else 10, seed=3)
    n = x.shape[1]
    deg = (2 + np.arange(n) % (3 if basis != T or dim == 2 else 1)).astype(np.int8)
    if basis == F and dim == 3:
        deg = (2 + np.arange(n) % 2).astype(np.int8)
    kpt = (6 + (np.arange(n) * 7) % (30 if dim == 2 else 45)).astype(np.int32)
    cid = ctx.cloud(x)
    nid = ctx.neighbors(cid, int(kpt.max()), 1.4, mode=gmls.RADIUS, cap=100, k_per_target=kpt)
    ref = ctx.stencils(nid, basis, 0, fns, precision=gmls.FP64, degree_per_target=deg)
    st64 = ctx.export(ref, gmls.X_STATUS, torch.uint8)
    ctx.release(ref)
    sid = ctx.stencils(nid, basis, 0, fns, precision=gmls.FP32_REFINE, degree_per_target=deg)
    st32 = ctx.export(sid, gmls.X_STATUS, torch.uint8)
    w_all = [ctx.weights(sid, fn).cpu().numpy() for fn in fns]
    off = ctx.export(nid, gmls.X_NBR_OFFSETS, torch.int64).cpu().numpy()
    ctx.release(sid)
    bad = gmls.T_RANK_DEFICIENT | gmls.T_UNSUPPORTED | gmls.T_TOO_FEW_NEIGHBOURS
    assert torch.equal(st64 & bad, st32 & bad)
    worst, _ = _compare(ctx, nid, basis, 0, fns, 0, n, forced=False, degree_per_target=deg)
    assert worst <= 1.0
    sub = np.arange(0, n - 1, 2, dtype=np.int32)
    nsub = ctx.neighbors(cid, int(kpt.max()), 1.4, mode=gmls.RADIUS, cap=100, targets=sub, k_per_target=kpt[sub])
    sid = ctx.stencils(nsub, basis, 0, fns, precision=gmls.FP32_REFINE, degree_per_target=deg[sub])
    osub = ctx.export(nsub, gmls.X_NBR_OFFSETS, torch.int64).cpu().numpy()
    for fn, wa in zip(fns, w_all):
        _, rows, nc, _ = ctx.stencil_info(sid, fn)
        ws, r = ctx.weights(sid, fn).cpu().numpy(), rows * nc
        for q, t in enumerate(sub):
            assert np.array_equal(ws[osub[q] * r:osub[q + 1] * r], wa[off[t] * r:off[t + 1] * r])
    for h in (sid, nsub, nid, cid):
        ctx.release(h)


def test_small_arena_runs_a_smaller_grid(ctx):
    """The kernel's slots come from the arena; where it cannot hold those of a
    full grid, a smaller grid gives the same weights bit for bit."""
    x = inputs.jittered_grid(3, 14, seed=4)
    small = gmls.Context(0, arena_bytes=35 << 20)
    out = []
    for c in (ctx, small):
        cid = c.cloud(x)
        nid = c.neighbors(cid, 80, 1.5)
        c.set_option(gmls.OPT_FORCE_VARIANT, -5)
        sid = c.stencils(nid, F, 3, [V], precision=gmls.FP32_REFINE)
        c.set_option(gmls.OPT_FORCE_VARIANT, 0)
        out.append(c.weights(sid, V).cpu().numpy())
        c.sync()
        for h in (sid, nid, cid):
            c.release(h)
    assert np.all(np.isfinite(out[0])) and np.array_equal(out[0], out[1])

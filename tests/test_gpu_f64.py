"""The FP64 stencil kernel of column-owning lanes (variant -6) against the
shared-memory FP64 kernel over the forms it accepts: every basis, dimension and
degree it is built for, fewest and odd and long lists, sets and orders of functionals, weight
powers, target subsets; and the targets it hands off.  Bar: both solve the same
systems with a forward error of a few kappa u_64; clouds here have kappa below
1e5, so 1e-10 relative per target and row (the bar the FP64 kernel is held to
against the oracle)."""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs

pytestmark = pytest.mark.gpu

G, L, D, V, C = gmls.GRAD, gmls.LAPLACIAN, gmls.DIV, gmls.VEC_LAPLACIAN, gmls.CURLCURL
S, F = gmls.SCALAR, gmls.DIVFREE


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


def _both(ctx, nid, basis, m, fns, **kw):
    """(weights per functional, status, beta-free info) of the forced kernel and of the shared-memory kernel."""
    out = []
    for variant in (-6, 0):
        ctx.set_option(gmls.OPT_FORCE_VARIANT, variant)
        ctx.set_option(gmls.OPT_FORCE_GENERIC, int(variant == 0))
        try:
            sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP64, **kw)
        finally:
            ctx.set_option(gmls.OPT_FORCE_VARIANT, 0)
            ctx.set_option(gmls.OPT_FORCE_GENERIC, 0)
        shapes = [ctx.stencil_info(sid, fn)[1:3] for fn in fns]
        w = [ctx.weights(sid, fn).cpu().numpy() for fn in fns]
        out.append((w, ctx.export(sid, gmls.X_STATUS, torch.uint8).cpu().numpy(), shapes))
        ctx.release(sid)
    return out


def _check(pair, n, k):
    (wa, sa, shapes), (wb, sb, _) = pair
    assert np.array_equal(sa, sb)
    for a, b, (rows, nc) in zip(wa, wb, shapes):
        a, b = a.reshape(n, rows, k, nc), b.reshape(n, rows, k, nc)
        assert np.isfinite(a).all()
        top = np.abs(b).max(axis=(2, 3))
        err = np.abs(a - b).max(axis=(2, 3)) / np.where(top > 0, top, 1.0)
        assert err.max() <= 1e-10


UNIFORM = [(2, S, 2, [L, G], 9), (2, S, 2, [G], 13), (2, S, 3, [G, L], 15), (2, S, 3, [D], 20), (2, S, 4, [D, G], 36),
           (2, S, 4, [G, L], 27), (2, S, 4, [L, G, D], 73), (2, S, 4, [G, L], 160), (2, S, 2, [L], 64),
           (2, F, 2, [V], 12), (2, F, 2, [C], 40), (2, F, 3, [V, C], 19), (2, F, 4, [C, V, D], 48), (2, F, 4, [V], 29),
           (3, F, 2, [V], 23), (3, F, 2, [C, D], 42), (3, F, 4, [V], 136), (3, F, 4, [C, D], 71)]


@pytest.mark.parametrize("dim,basis,m,fns,k", UNIFORM)
def test_uniform_lists_match_shared_memory_kernel(ctx, dim, basis, m, fns, k):
    x = inputs.jittered_grid(dim, 23 if dim == 2 else 8, seed=m + k)
    cid = ctx.cloud(x)
    nid = ctx.neighbors(cid, k, 1.5)
    _check(_both(ctx, nid, basis, m, fns), x.shape[1], k)
    for h in (nid, cid):
        ctx.release(h)


@pytest.mark.parametrize("power", [2, 6])
@pytest.mark.parametrize("dim,basis,m,fns,k", [(2, S, 4, [G, L], 36), (2, F, 3, [V], 34), (3, F, 2, [V], 42)])
def test_weight_powers_and_target_subsets(ctx, dim, basis, m, fns, k, power):
    x = inputs.jittered_grid(dim, 23 if dim == 2 else 9, seed=power) * 3.0 - 7.0
    cid = ctx.cloud(x)
    whole = None
    for n in (131, 5, 1):
        tg = ((np.arange(n) * 37) % x.shape[1]).astype(np.int32)
        nid = ctx.neighbors(cid, k, 1.5, targets=tg)
        pair = _both(ctx, nid, basis, m, fns, weight_power=power)
        _check(pair, n, k)
        first = [w.reshape(n, -1)[0] for w in pair[0][0]]
        whole = whole or first
        assert all(np.array_equal(a, b) for a, b in zip(first, whole))  # whatever the other targets
        ctx.release(nid)
    ctx.release(cid)


@pytest.mark.parametrize("basis,m,fns,k", [(S, 3, [G, L], 20), (F, 2, [V], 22)])
def test_degenerate_targets_are_handed_off(ctx, basis, m, fns, k):
    """A column of collinear points beside a regular part: the targets whose
    neighbours lie on the line are rank deficient and keep the shared-memory
    kernel's zeros and status."""
    x = inputs.jittered_grid(2, 16, seed=3)
    line = np.stack([np.full(60, 9.0), np.arange(60) / 60.0])
    x = np.ascontiguousarray(np.concatenate([x, line], axis=1))
    cid = ctx.cloud(x)
    nid = ctx.neighbors(cid, k, 1.5)
    pair = _both(ctx, nid, basis, m, fns)
    (wa, sa, shapes), (wb, sb, _) = pair
    bad = (sb & gmls.T_RANK_DEFICIENT) != 0
    assert bad[-60:].all() and not bad[:-60].any()
    assert np.array_equal(sa, sb)
    n = x.shape[1]
    for a, b, (rows, nc) in zip(wa, wb, shapes):
        assert np.array_equal(a.reshape(n, -1)[bad], b.reshape(n, -1)[bad])
    for h in (nid, cid):
        ctx.release(h)

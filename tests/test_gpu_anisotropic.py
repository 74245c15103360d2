"""Clouds flattened along one or two axes (boundary layers, thin sheets): the
FP32 + refinement stencils against the FP64 shared-memory kernel.  Bar as for any
cloud: 1e-9 relative per target and row."""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs

pytestmark = pytest.mark.gpu

G, L, V, C = gmls.GRAD, gmls.LAPLACIAN, gmls.VEC_LAPLACIAN, gmls.CURLCURL
S, F, T = gmls.SCALAR, gmls.DIVFREE, gmls.STAGGERED


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    build.build()
    c = gmls.Context(0, arena_bytes=4 << 30)
    c.set_option(gmls.OPT_POISON, 1)  # outputs start as NaN: unwritten entries cannot pass
    yield c
    c.close()


@pytest.mark.parametrize("stretch", [(1, 0.01, 1), (0.01, 1, 1), (1, 1, 0.03), (0.02, 1, 0.1)])
@pytest.mark.parametrize("dim,basis,m,fns,k,neu", [
    (2, S, 4, [G, L], 36, False), (2, F, 3, [V], 34, False), (2, F, 4, [C], 48, False), (2, T, 3, [G, L], 36, False),
    (3, S, 2, [L, G], 20, False), (3, S, 3, [G, L], 40, False), (3, F, 2, [V], 42, False), (3, F, 3, [C], 80, False),
    (3, T, 2, [G, L], 40, False), (3, S, 3, [G, L], 40, True)])
def test_flattened_clouds_match_fp64(ctx, dim, basis, m, fns, k, neu, stretch):
    x = inputs.jittered_grid(dim, 50 if dim == 2 else 14, seed=m) * np.array(stretch[:dim])[:, None]
    n = x.shape[1]
    kw = {}
    if neu:
        kw = dict(normals=inputs.unit_vectors(5, 6, n, dim), bflags=(inputs.uniform(5, 8, n) < 0.3).astype(np.uint8))
    cid = ctx.cloud(x, **kw)
    nid = ctx.neighbors(cid, k, 1.5)
    ctx.set_option(gmls.OPT_FORCE_GENERIC, 1)
    ref = ctx.stencils(nid, basis, m, fns, precision=gmls.FP64, neumann=neu)
    ctx.set_option(gmls.OPT_FORCE_GENERIC, 0)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5)
    sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE, neumann=neu)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, 0)
    bad = (ctx.export(ref, gmls.X_STATUS, torch.uint8) & gmls.T_RANK_DEFICIENT) != 0
    assert torch.equal(bad, (ctx.export(sid, gmls.X_STATUS, torch.uint8) & gmls.T_RANK_DEFICIENT) != 0)
    for fn in fns:
        _, rows, nc, _ = ctx.stencil_info(sid, fn)
        a, b = (ctx.weights(h, fn).view(n, rows, k * nc) for h in (sid, ref))
        err = ((a - b).abs().amax(2) / b.abs().amax(2).clamp(min=1e-300)).amax(1)
        assert float(err[~bad].max()) <= 1e-9
    for h in (sid, ref, nid, cid):
        ctx.release(h)


@pytest.mark.parametrize("power", [12, 20])
@pytest.mark.parametrize("dim,basis,m,fns,k", [(2, S, 2, [G, L], 12), (2, S, 3, [G, L], 20), (3, S, 2, [L, G], 20), (3, S, 3, [G, L], 40),
                                               (3, F, 3, [V], 80)])
def test_high_weight_powers_match_fp64(ctx, dim, basis, m, fns, k, power):
    x = inputs.jittered_grid(dim, 60 if dim == 2 else 16, seed=m)
    n = x.shape[1]
    cid = ctx.cloud(x)
    nid = ctx.neighbors(cid, k, 1.5)
    ctx.set_option(gmls.OPT_FORCE_GENERIC, 1)
    ref = ctx.stencils(nid, basis, m, fns, precision=gmls.FP64, weight_power=power)
    ctx.set_option(gmls.OPT_FORCE_GENERIC, 0)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5)
    sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE, weight_power=power)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, 0)
    for fn in fns:
        _, rows, nc, _ = ctx.stencil_info(sid, fn)
        a, b = (ctx.weights(h, fn).view(n, rows, k * nc) for h in (sid, ref))
        assert float(((a - b).abs().amax(2) / b.abs().amax(2)).max()) <= 1e-9
    for h in (sid, ref, nid, cid):
        ctx.release(h)


@pytest.mark.parametrize("dim,m,k,axis", [(2, 2, 12, 70), (3, 2, 20, 17), (2, 3, 20, 70), (2, 4, 36, 70), (3, 3, 40, 17),
                                          (3, 4, 84, 14)])
def test_neumann_rows_are_as_accurate_as_by_elimination(ctx, dim, m, k, axis):
    """On the one-sided targets of a box the constraint's share of the Laplacian
    row is the larger part of it.  Degree 2, whose systems are well conditioned: four
    units of the kernel's sums (2^-43), or the shared-memory FP32 kernel's error,
    which eliminates the constraint; degrees 3 and 4: the larger error of the two
    functionals is no more than that kernel's (a quarter for the clouds' spread)."""
    x = inputs.jittered_grid(dim, axis, seed=3)
    n = x.shape[1]
    i = np.arange(n)
    ix = np.stack([(i // axis ** c) % axis for c in range(dim)])
    nrm = (ix == axis - 1).astype(float) - (ix == 0)
    length = np.sqrt((nrm ** 2).sum(0))
    cid = ctx.cloud(x, normals=nrm / np.maximum(length, 1.0), bflags=(length > 0).astype(np.uint8))
    nid = ctx.neighbors(cid, k, 1.5)
    bnd = torch.from_numpy(length > 0).cuda()
    handles = []
    for precision, option, value in ((gmls.FP64, gmls.OPT_FORCE_GENERIC, 1), (gmls.FP32_REFINE, gmls.OPT_FORCE_GENERIC, 1),
                                     (gmls.FP32_REFINE, gmls.OPT_FORCE_VARIANT, -5)):
        ctx.set_option(option, value)
        handles.append(ctx.stencils(nid, S, m, [G, L], precision=precision, neumann=True))
        ctx.set_option(option, 0)
    err = []
    for h in handles[1:]:
        pairs = [(ctx.weights(h, fn).view(n, -1)[bnd], ctx.weights(handles[0], fn).view(n, -1)[bnd]) for fn in (G, L)]
        err.append(max(float((a - b).norm() / b.norm()) for a, b in pairs))
    assert err[1] <= (max(4 * 2.0 ** -43, err[0]) if m == 2 else 1.25 * err[0]), err
    for h in handles + [nid, cid]:
        ctx.release(h)

"""Clouds of any length unit (nanometres to light years): FP32 + refinement
stencils on scaled copies of a cloud.  Scaled by a power of two every operation
of the semi-normal-equation and the FP64 kernel scales exactly, so the weights are
those of the unscaled cloud times 2^(-order e), bit for bit (one refinement step:
nothing goes to the shared-memory FP32 kernel, whose smallest products
underflow); scaled by other factors they meet the bar against the FP64 kernel
(1e-9 relative per target and row).  (The exact comparison takes rows of one order
for the staggered basis: the stopping rule weighs all rows of a target together,
so with rows of both orders the number of targets redone in FP64 depends on the
length unit.)"""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs
from tests.test_gpu_seminormal import _compare

pytestmark = pytest.mark.gpu

G, L, D, V, C = gmls.GRAD, gmls.LAPLACIAN, gmls.DIV, gmls.VEC_LAPLACIAN, gmls.CURLCURL
S, F, T = gmls.SCALAR, gmls.DIVFREE, gmls.STAGGERED
SHAPES = [(2, S, 4, [G, L], 36, False), (2, S, 3, [G], 20, False), (3, S, 3, [L, G], 40, False), (2, F, 3, [V], 34, False),
          (3, F, 3, [C], 80, False), (3, F, 4, [V], 136, False), (2, T, 3, [G, L], 36, False), (2, S, 4, [G, L], 36, True),
          (3, S, 3, [G, L], 40, True)]


@pytest.fixture
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    build.build()
    c = gmls.Context(0, arena_bytes=2 << 30)
    c.set_option(gmls.OPT_POISON, 1)  # outputs start as NaN: unwritten entries cannot pass
    yield c
    c.close()


def _lists(ctx, dim, k, neu, scale):
    x = inputs.jittered_grid(dim, 40 if dim == 2 else 11, seed=k) * scale
    n = x.shape[1]
    kw = {}
    if neu:
        kw = dict(normals=inputs.unit_vectors(5, 6, n, dim) * (0.5 + inputs.uniform(5, 7, n)),
                  bflags=(inputs.uniform(5, 8, n) < 0.3).astype(np.uint8))
    return ctx.neighbors(ctx.cloud(x, **kw), k, 1.5), n


@pytest.mark.parametrize("e", [-43, -30, 30])
@pytest.mark.parametrize("dim,basis,m,fns,k,neu", [s for s in SHAPES if s[1] != T] + [(2, T, 3, [L], 36, False)])
def test_powers_of_two_scale_exactly(ctx, dim, basis, m, fns, k, neu, e):
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5)
    out = []
    for scale in (1.0, 2.0 ** e):
        nid, _ = _lists(ctx, dim, k, neu, scale)
        sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE, neumann=neu, max_refine=1)
        out.append([ctx.weights(sid, fn).cpu().numpy() for fn in fns] +
                   [ctx.export(nid, gmls.X_NBR_INDEX, torch.int32).cpu().numpy(),
                    ctx.export(sid, gmls.X_STATUS, torch.uint8).cpu().numpy()])
    for a, b, fn in zip(out[0], out[1], fns + [None, None]):
        order = 0 if fn is None else 1 if fn in (G, D) else 2
        assert np.isfinite(a).all()
        assert np.array_equal(np.ldexp(a, -order * e) if order else a, b)


@pytest.mark.parametrize("scale", [1e-13, 1e-9, 1e12])
@pytest.mark.parametrize("dim,basis,m,fns,k,neu", SHAPES)
def test_scaled_clouds_match_fp64(ctx, dim, basis, m, fns, k, neu, scale):
    nid, n = _lists(ctx, dim, k, neu, scale)
    worst, st = _compare(ctx, nid, basis, m, fns, k, n, neumann=neu)
    assert worst <= 1.0
    assert int(((st & gmls.T_FP64_FALLBACK) != 0).sum()) <= n // 20


@pytest.mark.parametrize("dim,m,k", [(2, 4, 36), (3, 3, 40)])
def test_beta_of_scaled_clouds(ctx, dim, m, k):
    """beta of the gradient rows does not depend on the length unit, that of the
    Laplacian scales with its inverse: exactly so for a power of two."""
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5)
    out = []
    for e in (0, -43, 30):
        nid, n = _lists(ctx, dim, k, True, 2.0 ** e)
        sid = ctx.stencils(nid, S, m, [G, L], precision=gmls.FP32_REFINE, neumann=True)
        beta = ctx.export(sid, gmls.X_BETA, torch.float64).cpu().numpy().reshape(n, dim + 1)
        beta[:, dim] = np.ldexp(beta[:, dim], e)
        out.append(beta)
    assert np.isfinite(out[0]).all() and (out[0] != 0).any()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


@pytest.mark.parametrize("basis,m,fns,k", [(S, 3, [G, L], 40), (S, 2, [L, G], 20), (F, 2, [V], 42)])
def test_weights_beyond_the_fp32_range_go_to_other_kernels(ctx, basis, m, fns, k):
    """At 1e14 the neighbour search of a 3D cloud stops short of the nearest
    points (flagged), and targets far outside their lists have rows of 1e6 and more
    times the usual size: a correction that is not finite does not count as
    converged."""
    nid, _ = _lists(ctx, 3, k, False, 1e14)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, -5)
    sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE)
    ctx.set_option(gmls.OPT_FORCE_VARIANT, 0)
    for fn in fns:
        assert bool(torch.isfinite(ctx.weights(sid, fn)).all())

"""The kernel a stencil call takes: a choice cached for one call must not serve
another that the kernel does not take (weight powers in turn on one context).
Bars as for the FP32 + refinement kernels: 1e-9 relative per target and row
against the FP64 kernel."""
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs
from tests.test_gpu_seminormal import _compare

pytestmark = pytest.mark.gpu

G, L, V = gmls.GRAD, gmls.LAPLACIAN, gmls.VEC_LAPLACIAN
S, F, T = gmls.SCALAR, gmls.DIVFREE, gmls.STAGGERED


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


@pytest.mark.parametrize("autotune", [1, 0])
@pytest.mark.parametrize("dim,basis,m,fns,k,axis", [(2, S, 4, [G, L], 36, 72), (2, F, 3, [V], 34, 72), (2, T, 3, [G, L], 36, 72),
                                                    (3, S, 3, [G, L], 40, 17), (3, F, 3, [V], 80, 13)])
def test_weight_powers_in_turn(ctx, dim, basis, m, fns, k, axis, autotune):
    ctx.set_option(gmls.OPT_AUTOTUNE, autotune)
    x = inputs.jittered_grid(dim, axis, seed=m)
    nid = ctx.neighbors(ctx.cloud(x), k, 1.5)
    for power in (4, 3, 1, 4, 5, 2):
        worst, _ = _compare(ctx, nid, basis, m, fns, k, x.shape[1], forced=False, weight_power=power)
        assert worst <= 1.0, power


@pytest.mark.parametrize("basis,fns", [(S, [G, L]), (F, [V])])
def test_weight_powers_in_turn_on_uneven_lists(ctx, basis, fns):
    x = inputs.jittered_grid(2, 72, seed=5)
    nid = ctx.neighbors(ctx.cloud(x), 24, 1.3, mode=gmls.RADIUS, cap=100)
    for power in (4, 3, 4):
        worst, _ = _compare(ctx, nid, basis, 3, fns, 0, x.shape[1], forced=False, weight_power=power)
        assert worst <= 1.0, power


@pytest.mark.parametrize("autotune", [1, 0])
@pytest.mark.parametrize("dim,basis,m,fns,k,axis,large", [(2, S, 3, [G, L], 20, 31, 80), (2, F, 2, [V], 22, 31, 80),
                                                          (3, S, 2, [G, L], 20, 10, 17)])
def test_small_cloud_does_not_depend_on_earlier_calls(ctx, dim, basis, m, fns, k, axis, large, autotune):
    """A large cloud of the same shape on the same context changes nothing."""
    ctx.set_option(gmls.OPT_AUTOTUNE, autotune)
    nid = ctx.neighbors(ctx.cloud(inputs.jittered_grid(dim, axis, seed=1)), k, 1.5)
    nlarge = ctx.neighbors(ctx.cloud(inputs.jittered_grid(dim, large, seed=2)), k, 1.5)
    out = []
    for _ in range(2):
        sid = ctx.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE)
        out.append([ctx.weights(sid, fn) for fn in fns])
        ctx.release(sid)
        ctx.release(ctx.stencils(nlarge, basis, m, fns, precision=gmls.FP32_REFINE))
    assert all(torch.equal(a, b) for a, b in zip(*out))


def _cloud_list(ctx, dim, k, n):
    axis = int(round(n ** (1.0 / dim)))
    assert axis ** dim == n
    return ctx.neighbors(ctx.cloud(inputs.jittered_grid(dim, axis, seed=k)), k, 1.5)


def _same_bits(ctx, nid, basis, m, fns, precision, option, value, **kw):
    """Whether the call's own choice (no timing) gives the bits of the forced kernel."""
    out = []
    ctx.set_option(gmls.OPT_AUTOTUNE, 0)
    for v in (0, value):
        ctx.set_option(option, v)
        sid = ctx.stencils(nid, basis, m, fns, precision=precision, **kw)
        out.append([ctx.weights(sid, fn) for fn in fns])
        ctx.set_option(option, 0)
    return all(torch.equal(a.view(torch.int64), b.view(torch.int64)) for a, b in zip(*out))


@pytest.mark.parametrize("dim,basis,m,fns,k,n,sne", [
    (2, S, 3, [G, L], 20, 2500, False), (2, S, 3, [G, L], 20, 3600, True), (2, S, 4, [G, L], 18, 3600, False),
    (2, S, 4, [G, L], 18, 8281, True), (2, S, 4, [G, L], 144, 2116, True), (2, S, 4, [G, L], 144, 1936, False),
    (2, T, 3, [G, L], 36, 3600, False), (2, T, 3, [G, L], 36, 4900, True), (2, T, 4, [G, L], 48, 4900, False),
    (3, T, 2, [G, L], 22, 4913, False), (3, F, 3, [V], 80, 343, True), (3, S, 4, [G, L], 84, 125, True),
    (3, S, 4, [G, L], 140, 216, False), (3, S, 4, [G, L], 38, 2744, False), (2, F, 2, [V], 22, 2500, False)])
def test_fp32_choice_by_targets_and_list_length(ctx, dim, basis, m, fns, k, n, sne):
    nid = _cloud_list(ctx, dim, k, n)
    assert _same_bits(ctx, nid, basis, m, fns, gmls.FP32_REFINE, gmls.OPT_FORCE_VARIANT, -5) == sne


@pytest.mark.parametrize("dim,basis,m,fns,k,n,cols", [
    (2, S, 2, [L, G], 12, 256, False), (2, S, 2, [L, G], 12, 1024, True), (2, S, 2, [L, G], 36, 900, False),
    (2, S, 4, [G, L], 36, 900, False), (2, S, 4, [G, L], 36, 1296, True), (2, S, 4, [G, L], 17, 2025, False),
    (2, S, 4, [G, L], 160, 4096, False), (2, F, 3, [V], 34, 900, False), (2, F, 3, [V], 34, 1296, True),
    (3, F, 2, [V], 42, 343, False), (3, F, 2, [V], 42, 512, True), (3, F, 4, [V], 136, 216, True)])
def test_fp64_choice_by_targets_and_list_length(ctx, dim, basis, m, fns, k, n, cols):
    nid = _cloud_list(ctx, dim, k, n)
    assert _same_bits(ctx, nid, basis, m, fns, gmls.FP64, gmls.OPT_FORCE_VARIANT, -6) == cols
    assert _same_bits(ctx, nid, basis, m, fns, gmls.FP64, gmls.OPT_FORCE_GENERIC, 1) != cols

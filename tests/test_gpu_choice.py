"""The kernel a stencil call takes: a choice cached for one call must not serve
another that the kernel does not take (weight powers in turn on one context).
Bars as for the FP32 + refinement kernels: 1e-9 relative per target and row
against the FP64 kernel."""
import math

import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs
from tests.test_gpu_seminormal import _compare

pytestmark = pytest.mark.gpu

G, L, V, C = gmls.GRAD, gmls.LAPLACIAN, gmls.VEC_LAPLACIAN, gmls.CURLCURL
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


def _size(dim, basis, degree):
    full = math.comb(degree + dim, dim)
    return {S: full, F: dim * full - math.comb(degree - 1 + dim, dim), T: math.comb(degree + 1 + dim, dim) - 1}[basis]


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
    (2, S, 3, [G, L], 20, 1936, False), (2, S, 3, [G, L], 20, 2116, True), (2, S, 4, [G, L], 18, 3600, False),
    (2, S, 4, [G, L], 18, 8281, True), (2, S, 4, [G, L], 144, 2116, True), (2, S, 4, [G, L], 144, 1936, False),
    (2, T, 3, [G, L], 36, 3600, False), (2, T, 3, [G, L], 36, 4900, True), (2, T, 4, [G, L], 48, 4900, False),
    (3, T, 2, [G, L], 22, 4913, False), (3, F, 3, [V], 80, 343, True), (3, S, 4, [G, L], 84, 125, True),
    (3, S, 4, [G, L], 140, 216, False), (3, S, 4, [G, L], 38, 2744, False), (2, F, 2, [V], 22, 1936, False)])
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


@pytest.mark.parametrize("dim,basis,fns,n,per_target,buckets", [
    (2, S, [G, L], 900, True, False), (2, S, [G, L], 4900, True, True), (3, S, [G, L], 2197, True, False),
    (3, S, [G, L], 4913, True, True), (2, S, [G], 900, False, False), (2, S, [G], 1600, False, True),
    (2, F, [V], 1600, True, False), (2, F, [V], 2025, True, True), (3, F, [V], 343, True, False), (3, F, [V], 729, True, True),
    (2, T, [G, L], 3600, True, False), (2, T, [G, L], 4900, True, True)])
def test_uneven_choice_by_targets(ctx, dim, basis, fns, n, per_target, buckets):
    """One persistent launch for few targets (the bits of the shared-memory
    kernel), a launch a bucket for many."""
    axis = int(round(n ** (1.0 / dim)))
    x = inputs.jittered_grid(dim, axis, seed=4)
    assert x.shape[1] == n
    nid = ctx.neighbors(ctx.cloud(x), 24 if dim == 2 else 45, 1.4, mode=gmls.RADIUS, cap=128)
    kw = dict(degree_per_target=(2 + np.arange(n) % 2).astype(np.int8)) if per_target else {}
    assert _same_bits(ctx, nid, basis, 0 if per_target else 3, fns, gmls.FP32_REFINE, gmls.OPT_FORCE_GENERIC, 1, **kw) != buckets


@pytest.mark.parametrize("dim,basis,fns", [(2, S, [G, L]), (3, S, [G]), (2, F, [V]), (3, F, [C]), (2, T, [G, L])])
def test_launches_per_bucket_match_fp64(ctx, dim, basis, fns):
    """Radius lists of every length (some with fewer neighbours than basis
    functions) and a degree per target, on enough targets for a launch a bucket.
    Weights of lists of 3/2 of the basis size and more (shorter ones are
    ill-conditioned: the kernels used before, too, were off by up to 4e-9 there)."""
    x = inputs.jittered_grid(dim, 70 if dim == 2 else 17, seed=3)
    n = x.shape[1]
    deg = (2 + np.arange(n) % (2 if dim == 3 and basis == F else 3)).astype(np.int8)
    kpt = (6 + (np.arange(n) * 7) % (30 if dim == 2 else 45)).astype(np.int32)
    nid = ctx.neighbors(ctx.cloud(x), int(kpt.max()), 1.4, mode=gmls.RADIUS, cap=100, k_per_target=kpt)
    ref = ctx.stencils(nid, basis, 0, fns, precision=gmls.FP64, degree_per_target=deg)
    sid = ctx.stencils(nid, basis, 0, fns, precision=gmls.FP32_REFINE, degree_per_target=deg)
    st64, st32 = (ctx.export(h, gmls.X_STATUS, torch.uint8) for h in (ref, sid))
    bad = gmls.T_RANK_DEFICIENT | gmls.T_UNSUPPORTED | gmls.T_TOO_FEW_NEIGHBOURS
    assert torch.equal(st64 & bad, st32 & bad)
    off = ctx.export(nid, gmls.X_NBR_OFFSETS, torch.int64).cpu().numpy()
    size = {d: _size(dim, basis, d) for d in (2, 3, 4)}
    long = [t for t in range(n) if 2 * (off[t + 1] - off[t]) * (dim if basis == F else 1) >= 3 * size[int(deg[t])]]
    assert len(long) > n // 3
    for fn in fns:
        _, rows, nc, _ = ctx.stencil_info(sid, fn)
        a, b = (ctx.weights(h, fn).cpu().numpy() for h in (sid, ref))
        for t in long:
            wa, wb = (w[off[t] * rows * nc:off[t + 1] * rows * nc].reshape(rows, -1) for w in (a, b))
            assert (np.abs(wa - wb).max(1) <= 1e-9 * np.abs(wb).max(1)).all(), t


@pytest.mark.parametrize("dim,m,k,n", [(2, 4, 48, 4900), (3, 3, 80, 2744), (3, 4, 136, 1000), (2, 3, None, 4900)])
def test_tight_tolerance_on_divergence_free_systems(ctx, dim, m, k, n):
    """refine_tol 1e-13 ends at the roundings of the float-float residuals, 2^-48
    times conditions of up to a thousand: 4e-12."""
    axis = int(round(n ** (1.0 / dim)))
    x = inputs.jittered_grid(dim, axis, seed=9)
    cid = ctx.cloud(x)
    nid = ctx.neighbors(cid, k, 1.5) if k else ctx.neighbors(cid, 34, 1.4, mode=gmls.RADIUS, cap=100)
    ref = ctx.stencils(nid, F, m, [V], precision=gmls.FP64)
    sid = ctx.stencils(nid, F, m, [V], precision=gmls.FP32_REFINE, refine_tol=1e-13)
    off = ctx.export(nid, gmls.X_NBR_OFFSETS, torch.int64)
    seg = torch.repeat_interleave(torch.arange(dim * n, device="cuda"), ((off[1:] - off[:-1]) * dim).repeat_interleave(dim))
    total = seg.shape[0]
    a, b = (ctx.weights(h, V)[:total] for h in (sid, ref))
    err, top = (torch.zeros(dim * n, device="cuda", dtype=torch.float64).scatter_reduce_(0, seg, v, "amax")
                for v in ((a - b).abs(), b.abs()))
    assert float((err / top).max()) <= 4e-12


@pytest.mark.parametrize("power,cols", [(4, True), (8, True), (10, False), (20, False)])
def test_fp64_choice_by_weight_power(ctx, power, cols):
    nid = _cloud_list(ctx, 2, 12, 1600)
    assert _same_bits(ctx, nid, S, 2, [L, G], gmls.FP64, gmls.OPT_FORCE_VARIANT, -6, weight_power=power) == cols
    assert _same_bits(ctx, nid, S, 2, [L, G], gmls.FP64, gmls.OPT_FORCE_GENERIC, 1, weight_power=power) != cols

"""Arena limits: what a call needs beside its results."""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs

pytestmark = pytest.mark.gpu

G, L, V, C = gmls.GRAD, gmls.LAPLACIAN, gmls.VEC_LAPLACIAN, gmls.CURLCURL
S, F, T = gmls.SCALAR, gmls.DIVFREE, gmls.STAGGERED


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    build.build()


def test_uneven_batch_does_not_reserve_tiles_for_the_list_capacity():
    """Short lists under a capacity of 1,024: 122 MB of results and lists, a
    persistent launch with tiles of the row classes; no more for the hand-off."""
    ctx = gmls.Context(0, arena_bytes=400 << 20)
    x = inputs.jittered_grid(3, 10, seed=1)
    n = x.shape[1]
    nid = ctx.neighbors(ctx.cloud(x), 45, 1.4, mode=gmls.RADIUS, cap=1024)
    sid = ctx.stencils(nid, F, 0, [V], precision=gmls.FP32_REFINE, degree_per_target=(2 + np.arange(n) % 3).astype(np.int8))
    total = int(ctx.export(nid, gmls.X_NBR_OFFSETS, torch.int64)[-1])
    assert bool(torch.isfinite(ctx.weights(sid, V)[:total * 9]).all())
    ctx.close()


def _lists(ctx, dim, k, n_axis, neu):
    x = inputs.jittered_grid(dim, n_axis, seed=2)
    n = x.shape[1]
    kw = dict(normals=inputs.unit_vectors(5, 6, n, dim), bflags=(inputs.uniform(5, 8, n) < 0.3).astype(np.uint8)) if neu else {}
    return ctx.neighbors(ctx.cloud(x, **kw), k, 1.5)


@pytest.mark.parametrize("dim,basis,m,fns,k,n_axis,variant,neu", [
    (2, S, 4, [G, L], 36, 64, -2, False), (3, S, 3, [G, L], 40, 16, -1, False), (2, T, 3, [G, L], 36, 72, -1, False),
    (2, S, 4, [G, L], 36, 64, -2, True)])
def test_call_fits_where_the_register_kernels_do(dim, basis, m, fns, k, n_axis, variant, neu):
    """A call runs in an arena with no room for the slots of the
    semi-normal-equation kernel."""
    big = gmls.Context(0, arena_bytes=1 << 30)
    nid = _lists(big, dim, k, n_axis, neu)
    big.set_option(gmls.OPT_FORCE_VARIANT, variant)
    big.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE, neumann=neu)
    peak = big.arena_usage()[1]
    small = gmls.Context(0, arena_bytes=peak + 512)  # (the buffer's start is rounded up to 256 bytes)
    small.set_option(gmls.OPT_AUTOTUNE, 0)
    nid = _lists(small, dim, k, n_axis, neu)
    sid = small.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE, neumann=neu)
    assert all(bool(torch.isfinite(small.weights(sid, fn)).all()) for fn in fns)
    for c in (big, small):
        c.close()


@pytest.mark.parametrize("part", [0.9, 0.5, 0.3, 0.1, 0.02])
@pytest.mark.parametrize("dim,basis,m,fns,k,n_axis", [(3, F, 3, [V], 80, 14), (2, S, 4, [G, L], 36, 64)])
def test_grid_shrinks_to_the_slots_the_arena_holds(dim, basis, m, fns, k, n_axis, part):
    """The forced kernel with a part of a full grid's slots: the same bits."""
    big = gmls.Context(0, arena_bytes=1 << 30)
    nid = _lists(big, dim, k, n_axis, False)
    lists = big.arena_usage()[1]
    big.set_option(gmls.OPT_FORCE_VARIANT, -5)
    sid = big.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE)
    used, peak, _ = big.arena_usage()
    slots = peak - used
    assert slots > 1 << 20 and peak > lists
    room = used + int(part * slots)
    assert room >= lists
    small = gmls.Context(0, arena_bytes=room)
    nid = _lists(small, dim, k, n_axis, False)
    small.set_option(gmls.OPT_FORCE_VARIANT, -5)
    sid2 = small.stencils(nid, basis, m, fns, precision=gmls.FP32_REFINE)
    assert small.arena_usage()[2] - small.arena_usage()[0] < slots  # a full grid's slots cannot fit
    for fn in fns:
        assert torch.equal(big.weights(sid, fn), small.weights(sid2, fn))
    for c in (big, small):
        c.close()


@pytest.mark.parametrize("row_scaling", [False, True])
@pytest.mark.parametrize("restart", [1, 2, 7, 30, 100, 256])
def test_gmres_needs_its_basis_and_a_few_vectors(restart, row_scaling):
    """The arena of a solve: the basis, up to four vectors and reductions of 304
    partial sums a column."""
    n, m = 60000, restart

    def up(count, size):
        return (count * size + 255) // 256 * 256

    need = (up((m + 1) * n, 8) + (3 if row_scaling else 2) * up(n, 8) + up(n, 4) + up(304 * (m + 2), 8) + up(2 * (m + 2), 8) +
            up(1, 4) + up(64 * 128, 8))
    ctx = gmls.Context(0, arena_bytes=need + 512)  # (the buffer's start is rounded up to 256 bytes)
    i = torch.arange(n, device="cuda")
    col = torch.stack([(i - 1).clamp(min=0), i, (i + 1).clamp(max=n - 1)], 1).reshape(-1).to(torch.int32)
    val = torch.tensor([-1.0, 4.0, -1.0], device="cuda", dtype=torch.float64).repeat(n)
    row = torch.arange(n + 1, device="cuda") * 3
    x, its, rel = ctx.gmres(row, col, val, torch.ones(n, dtype=torch.float64, device="cuda"), restart=m, max_iter=4 * m + 20,
                            rtol=1e-9, row_scaling=row_scaling)
    assert its > 0 and rel < 1e-2 and bool(torch.isfinite(x).all())
    ctx.close()


def test_server_admits_what_its_arena_holds():
    """31,684 points in 64 MiB: results, lists and cloud take 42 MB, the slots come
    out of the margin; the same bits as in a context with room to spare."""
    x = inputs.jittered_grid(2, 178, seed=6)
    srv = gmls.Server(0, arena_bytes=64 << 20, streams=1, max_inflight=1)
    t = srv.submit(x, S, 4, 36, [G, L])
    assert srv.wait(t, 60000)
    ctx = gmls.Context(0, arena_bytes=1 << 30)
    ctx.set_option(gmls.OPT_AUTOTUNE, 0)
    sid = ctx.stencils(ctx.neighbors(ctx.cloud(x), 36, 1.5), S, 4, [G, L], precision=gmls.FP32_REFINE)
    for fn in (G, L):
        assert torch.equal(srv.result(t, gmls.X_WEIGHTS, torch.float64, fn), ctx.weights(sid, fn).cpu())
    srv.release(t)
    srv.close()
    ctx.close()

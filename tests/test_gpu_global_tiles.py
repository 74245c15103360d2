"""Buckets whose tiles live in global memory, of different warps per target, in
one persistent launch: the autotuner's choice gives the weights of the choice
without timing (every such bucket with four warps per target).  Bar: both solve
the same systems in FP64, 1e-10 relative per target and row."""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fn", [gmls.VEC_LAPLACIAN, gmls.CURLCURL])
def test_autotuned_buckets_match_untimed_ones(fn):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    build.build()
    ctx = gmls.Context(0, arena_bytes=4 << 30)
    ctx.set_option(gmls.OPT_POISON, 1)
    x = inputs.jittered_grid(3, 17, seed=3)
    n = x.shape[1]
    deg = (2 + np.arange(n) % 2).astype(np.int8)
    kpt = (24 + (np.arange(n) * 7) % 45).astype(np.int32)
    nid = ctx.neighbors(ctx.cloud(x), int(kpt.max()), 1.4, mode=gmls.RADIUS, cap=110, k_per_target=kpt)
    off = ctx.export(nid, gmls.X_NBR_OFFSETS, torch.int64)
    out = []
    for generic in (0, 1):
        ctx.set_option(gmls.OPT_FORCE_GENERIC, generic)
        sid = ctx.stencils(nid, gmls.DIVFREE, 0, [fn], precision=gmls.FP64, degree_per_target=deg)
        out.append((ctx.weights(sid, fn), ctx.export(sid, gmls.X_STATUS, torch.uint8)))
    (wa, sa), (wb, sb) = out
    assert torch.equal(sa, sb)
    seg = torch.repeat_interleave(torch.arange(3 * n, device="cuda"), ((off[1:] - off[:-1]) * 3).repeat_interleave(3))
    err, top = (torch.zeros(3 * n, device="cuda", dtype=torch.float64).scatter_reduce_(0, seg, v, "amax")
                for v in ((wa - wb).abs(), wb.abs()))
    assert float((err / torch.where(top > 0, top, 1.0)).max()) <= 1e-10
    ctx.close()

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

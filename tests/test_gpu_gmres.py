"""gmls_gmres where its device-side cycle can go wrong: restarts shorter and
longer than the chunk of iterations the host queues, a stop inside a chunk (by
tolerance and by max_iter), no, a few and more than 64 long rows in A x, one
unknown, an exact start."""
import numpy as np
import pytest
import torch

from paper_2104_14447_gb300 import gmls

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    build.build()
    c = gmls.Context(0, arena_bytes=1 << 30)
    yield c
    c.close()


def _system(n, band, dense_rows, seed):
    """A diagonally dominant sparse matrix with a few full rows (scipy CSR)."""
    sp = pytest.importorskip("scipy.sparse")
    rng = np.random.RandomState(seed)
    offs = rng.permutation(np.arange(1, max(2, min(n, 40))))[:band] if n > 1 else []
    A = sp.diags([np.full(n, 4.0 + 0.1 * band)], [0], format="lil")
    A = A.tocsr()
    for o in offs:
        A = A + sp.diags([rng.uniform(-0.4, 0.4, n - o)], [int(o)], shape=(n, n)) if o < n else A
    if dense_rows:
        D = sp.lil_matrix((n, n))
        for r in rng.permutation(n)[:dense_rows]:
            D[r, :] = rng.uniform(-1.0, 1.0, n) / n
        A = A + D.tocsr()
    A = A.tocsr()
    A.sort_indices()
    return A


@pytest.mark.parametrize("row_scaling", [False, True])
@pytest.mark.parametrize("n,band,dense_rows,restart", [(1, 0, 0, 5), (37, 3, 0, 3), (1000, 9, 0, 8), (3001, 12, 2, 30),
                                                       (9001, 7, 3, 100), (8300, 5, 70, 20)])
def test_gmres_matches_direct_solve(ctx, n, band, dense_rows, restart, row_scaling):
    A = _system(n, band, dense_rows, n)
    rng = np.random.RandomState(7)
    xe = rng.randn(n)
    b = A @ xe
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (A.indptr.astype(np.int64), A.indices.astype(np.int32),
                                                                       A.data.astype(np.float64), b)]
    x, its, rel = ctx.gmres(*dev, restart=restart, max_iter=2000, rtol=1e-11, row_scaling=row_scaling)
    assert rel <= 1e-11 and 1 <= its < 2000
    # |x - xe| <= |A^-1| |r|: the diagonal exceeds the sum of its row's other entries by at least 1
    assert np.abs(x.cpu().numpy() - xe).max() <= 1e-11 * np.linalg.norm(b) * 4
    x2, its2, _ = ctx.gmres(*dev, restart=restart, max_iter=2000, rtol=1e-11, row_scaling=row_scaling)
    assert its2 == its and torch.equal(x, x2)  # reproducible bit for bit
    # stopped inside a chunk by max_iter: that many iterations, a residual that went down
    if its > 5:
        _, it5, rel5 = ctx.gmres(*dev, restart=restart, max_iter=5, rtol=1e-11, row_scaling=row_scaling)
        assert it5 == 5 and rel < rel5 < 1.0
    # started from the solution: nothing to do
    x0 = torch.from_numpy(xe).cuda()
    _, it0, rel0 = ctx.gmres(*dev, x0=x0, restart=restart, max_iter=50, rtol=1e-9, row_scaling=row_scaling)
    assert it0 == 0 and rel0 <= 1e-9

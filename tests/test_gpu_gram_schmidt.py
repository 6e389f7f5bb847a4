"""CGS2 at the edges of its launch shapes: lengths around a warp, a block and
the switch between eight threads and one thread a row; column counts around
the groups of eight; a leading dimension beyond n; partial sums added by the
update itself and by a reduction; the allocation-free form alike.  Bars as in
test_gpu_krylov.py: 1e-12 ||w|| against numpy in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_03859_gb300 import nsstab  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,j,pad", [(1, 1, 0), (31, 7, 3), (33, 8, 0), (1024, 9, 1), (1025, 17, 0), (4097, 64, 5),
                                     (16385, 3, 0), (155392, 15, 0), (155393, 16, 1), (200003, 33, 0), (5000, 300, 0),
                                     (16, 0, 0), (300001, 0, 0)])
def test_cgs2_at_launch_edges(n, j, pad):
    rng = np.random.default_rng(7 * n + j)
    q = min(j, n)
    V = np.zeros((max(j, 1), n + pad))
    if q:
        V[:q, :n] = np.linalg.qr(rng.standard_normal((n, q)))[0].T     # beyond n columns: zeros
    V[:, n:] = np.nan                                                    # never read
    w = rng.standard_normal(n)
    Vn = V[:j, :n]
    h1 = Vn @ w
    w1 = w - h1 @ Vn
    h2 = Vn @ w1
    w2 = w1 - h2 @ Vn
    tol = 1e-12 * np.linalg.norm(w)
    for call in (nsstab.cgs2_orthogonalize, nsstab.cgs2_orthogonalize_noalloc):
        if call is nsstab.cgs2_orthogonalize_noalloc and j > nsstab.NOALLOC_MAX_COLS:
            continue
        wd = torch.from_numpy(w).cuda()
        h, beta = call(torch.from_numpy(V).cuda(), n, j, wd, ldv=n + pad)
        torch.cuda.synchronize()
        assert np.abs(h - (h1 + h2)).max(initial=0.0) <= tol
        assert abs(beta - np.linalg.norm(w2)) <= tol
        assert np.abs(wd.cpu().numpy() - w2).max() <= tol
        again = torch.from_numpy(w).cuda()
        hb, bb = call(torch.from_numpy(V).cuda(), n, j, again, ldv=n + pad)
        assert np.array_equal(h, hb) and beta == bb and torch.equal(wd, again)   # fixed order of every sum

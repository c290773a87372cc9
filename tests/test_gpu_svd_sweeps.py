"""The Jacobi sweeps of the block SVD at the sizes where their kernels take another path: one
and few columns, an odd number of them, more than one block of 16, columns longer than the 512 rows
that stay in registers, columns too long for shared memory (r + k above about 1450 rows), and more
pairs than a grid of resident warps.

M = U diag(s) V^T with orthonormal U, V and known s.  One-sided Jacobi returns the singular values
of M to a small multiple of eps s_max per rotation that a column goes through (k - 1 a sweep), and
forming M rounds by at most sqrt(k) eps s_max: 4 (r + k) eps s_max bounds both.  The rotations are
shears of determinant one, so the factors' columns stay unit vectors far closer than that: their
mean square is 1 to the rounding of single elements, not of k rotations.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2007_05540_gb300 import heff              # noqa: E402

EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("rows,cols", [(1, 1), (5, 2), (31, 3), (17, 40), (70, 33), (513, 64), (700, 130), (64, 1600),
                                       (1600, 96), (2500, 2450)])
def test_sweeps_at_edge_sizes(rows, cols):
    rng = np.random.default_rng(rows * 7 + cols)
    k = min(rows, cols)
    U = np.linalg.qr(rng.standard_normal((rows, k)))[0]
    V = np.linalg.qr(rng.standard_normal((cols, k)))[0]
    s = np.logspace(0, -4, k)
    M = (U * s) @ V.T
    q0 = np.zeros((1, 1), dtype=np.int32)

    def index(n, sign):
        return (q0, np.array([n], dtype=np.int32), sign)

    x_l = heff.Layout([index(rows, 1), index(1, 1), index(1, -1), index(cols, -1)])
    h = heff.heff_svd_create(x_l.handle)
    try:
        ws = torch.empty(heff.heff_svd_workspace_size(h), dtype=torch.uint8, device="cuda")
        x = torch.from_numpy(M.reshape(-1)).to("cuda")
        heff.heff_svd_compute(h, x, ws)
        q, d, disc, norm = heff.heff_svd_truncate(h, 10 ** 6, 0.0, 1, 16)
        assert d.tolist() == [k] and disc < 1e-12
        got = np.sort(heff.heff_svd_singular_values(h, k))[::-1]
        tol = 4 * (rows + cols) * EPS
        assert np.abs(got - s).max() < tol
        A_l = heff.Layout([index(rows, 1), index(1, 1), index(k, -1)])
        B_l = heff.Layout([index(k, 1), index(1, -1), index(cols, -1)])
        A = torch.empty(A_l.nelem, dtype=torch.float64, device="cuda")
        B = torch.empty(B_l.nelem, dtype=torch.float64, device="cuda")
        heff.heff_svd_write(h, A_l.handle, B_l.handle, A, B, True, ws)
        a, b = A.cpu().numpy().reshape(rows, k), B.cpu().numpy().reshape(k, cols)
        assert np.abs(a @ b - M).max() < tol
        assert abs((a.astype(np.longdouble) ** 2).sum() / k - 1) < 16 * EPS
        assert np.abs(a.T @ a - np.eye(k)).max() < 1e-12
    finally:
        heff.heff_svd_destroy(h)

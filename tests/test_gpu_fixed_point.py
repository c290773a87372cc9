"""FP64 block products as fixed-point digits on the tensor cores (csrc/fx_gemm.cu).

One charge sector and one local state turn the two-site product x[a, b] = sum_c A[a, c] B[c, b]
into a plain matrix product, so tile edges, contraction remainders and special values can be
set directly.  Bound per element: the operands keep 61 bits below their row's (column's) largest
element, the dropped digit products and the FP32 roundings of the low accumulators stay below
2^-50 K of the two largest elements' product, and the sum is rounded to FP64 once.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _product(a, b):
    import torch
    from paper_2007_05540_gb300 import heff
    m, k = a.shape
    n = b.shape[1]
    q = np.zeros((1, 1), dtype=np.int32)
    one = np.ones(1, dtype=np.int32)
    bond = lambda d: (q, np.array([d], dtype=np.int32))
    A = heff.Layout([(*bond(m), 1), (q, one, 1), (*bond(k), -1)])
    B = heff.Layout([(*bond(k), 1), (q, one, 1), (*bond(n), -1)])
    X = heff.Layout([(*bond(m), 1), (q, one, 1), (q, one, 1), (*bond(n), -1)])
    h = heff.heff_two_site_create(A.handle, B.handle, X.handle)
    ta = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()
    tb = torch.from_numpy(np.ascontiguousarray(b).reshape(-1)).cuda()
    # guard elements around the output: nothing outside it may be written
    x = torch.full((m * n + 64,), 7.0, dtype=torch.float64, device="cuda")
    heff.heff_two_site_apply(h, ta, tb, x[32:32 + m * n])
    out = x.cpu().numpy()
    heff.heff_two_site_destroy(h)
    assert (out[:32] == 7.0).all() and (out[32 + m * n:] == 7.0).all()
    return out[32:32 + m * n].reshape(m, n)


def _bound(a, b, c):
    k = a.shape[1]
    return 2.0 ** -50 * k * np.outer(np.abs(a).max(1), np.abs(b).max(0)) + 2.0 ** -52 * np.abs(c)


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (127, 15, 63), (128, 16, 64), (129, 17, 65), (5, 255, 16), (64, 256, 17),
                                   (130, 257, 33), (33, 513, 48), (300, 1100, 140)])
@pytest.mark.parametrize("fill", ["normal", "graded", "ones", "ragged_scales"])
def test_product_within_the_fixed_point_bound(m, k, n, fill):
    rng = np.random.default_rng([m, k, n])
    a, b = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    if fill == "graded":                      # both fall off along the contraction index
        w = np.exp(-20.0 * np.arange(k) / k)
        a, b = a * w, b * w[:, None]
    elif fill == "ones":                      # every digit of every element alike: the largest sums
        a, b = np.full((m, k), 0.5 + 127.0 / 510), np.full((k, n), -(0.5 + 127.0 / 510))
    elif fill == "ragged_scales":             # a scale per row and per column
        a = a * 10.0 ** rng.integers(-60, 60, (m, 1))
        b = b * 10.0 ** rng.integers(-60, 60, (1, n))
        a[rng.integers(m)] = 0.0
    ref = np.asarray(a.astype(np.longdouble) @ b.astype(np.longdouble))
    got = _product(a, b)
    assert (np.abs(got - ref) <= _bound(a, b, ref.astype(np.float64))).all()


def test_integers_are_exact():
    rng = np.random.default_rng(3)
    a = rng.integers(-2 ** 20, 2 ** 20, (150, 300)).astype(np.float64)
    b = rng.integers(-2 ** 20, 2 ** 20, (300, 90)).astype(np.float64)
    assert (_product(a, b) == (a.astype(np.int64) @ b.astype(np.int64)).astype(np.float64)).all()


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e300, 1e-300, 5e-324])
@pytest.mark.parametrize("where", ["a", "b"])
def test_values_outside_the_fixed_point_range(value, where):
    """Rows that no scale of the fixed-point range holds run in FP64 arithmetic: infinities and
    NaNs land where IEEE arithmetic puts them, tiny and huge magnitudes keep their result."""
    rng = np.random.default_rng(5)
    a, b = rng.standard_normal((140, 40)), rng.standard_normal((40, 70))
    t = a if where == "a" else b.T
    t[3] = 0.0
    t[3, 7] = value
    t[9] = 0.0                                # an all-zero row beside it
    with np.errstate(all="ignore"):
        ref = np.stack([[np.sum(a[i] * b[:, j]) for j in range(70)] for i in range(140)])
    got = _product(a, b)
    fin = np.isfinite(ref)
    assert (np.isnan(got) == np.isnan(ref)).all() and (got[np.isinf(ref)] == ref[np.isinf(ref)]).all()
    # 40 terms: the FP64 sum's bound 40 * 2^-53 sum |a||b|, on either path
    tol = 40 * 2.0 ** -52 * (np.abs(a) @ np.abs(b))
    assert (np.abs(got[fin] - ref[fin]) <= np.maximum(tol[fin], 5e-324)).all()


@pytest.mark.parametrize("power", [-700, -350, 0, 350])
def test_matvec_is_homogeneous_over_the_exponent_range(power):
    """y = K x for x times a power of two: inside and outside the fixed-point range."""
    import torch
    import workloads as wl
    from paper_2007_05540_gb300 import heff
    from tests.helpers import library_problem
    w = wl.workload_by_name("electron_m40")
    lays, bufs = library_problem(w)
    plan = heff.Plan(*lays, bufs["W1"], bufs["W2"], "fp64", "f64")
    d = {k: torch.from_numpy(np.asarray(bufs[k])).cuda() for k in ("L", "W1", "W2", "R")}
    x = torch.from_numpy(bufs["x"][0]).cuda()
    ws = plan.workspace()
    y, ys = torch.empty_like(x), torch.empty_like(x)
    heff.heff_apply(plan.handle, d["L"], d["W1"], d["W2"], d["R"], x, y, ws)
    heff.heff_apply(plan.handle, d["L"], d["W1"], d["W2"], d["R"], x * 2.0 ** power, ys, ws)
    assert heff.heff_workspace_status(plan.handle, ws) == 0
    assert float((ys * 2.0 ** -power - y).norm() / y.norm()) < 1e-14

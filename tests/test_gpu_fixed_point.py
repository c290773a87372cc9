"""FP64 products as fixed-point digits on the tensor cores (csrc/fx_gemm.cu, csrc/fx_planes.cu).

One charge sector and one local state turn the two-site product x[a, b] = sum_c A[a, c] B[c, b]
into a plain matrix product, and the matvec into y = L x R^T, so tile edges, contraction remainders
and special values can be set directly.  The bound is that of a running FP64 sum, element by element:
K 2^-53 sum |a||b|, whose factor is 1.2 where digits are used (csrc/fx_check.cuh), and one rounding.
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


def _bound(a, b):
    return (1.2 * a.shape[1] + 2) * 2.0 ** -53 * (np.abs(a) @ np.abs(b))


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
    assert (np.abs(got - ref) <= _bound(a, b)).all()


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (127, 15, 63), (130, 96, 70), (33, 513, 48), (300, 1100, 140)])
@pytest.mark.parametrize("fill", ["opposite", "gauge", "spike", "sparse", "mixed", "coherent"])
def test_product_of_operands_whose_large_elements_do_not_meet(m, k, n, fill):
    a, b = _operands(fill, m, k, n, np.random.default_rng([m, k, n]))
    for u, v in ((a, b), (b.T, a.T)):
        ref = u.astype(np.longdouble) @ v.astype(np.longdouble)
        assert (np.abs(_product(u, v) - ref) <= _bound(u, v)).all()


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


# ------------------------------------------------------------------ the matvec
def _matvec(L, x, R):
    """y = L x R^T by a plan with one sector, one local state and one MPO channel."""
    import torch
    from paper_2007_05540_gb300 import heff
    m, n = x.shape
    q, one = np.zeros((1, 1), dtype=np.int32), np.zeros((1, 1), dtype=np.int32)
    lays = heff.heff_layouts((q, np.array([m], dtype=np.int32)), (q, np.array([n], dtype=np.int32)), one, q, q, q)
    w = np.ones(1)
    plan = heff.Plan(*lays, w, w, "fp64", "f64")
    t = [torch.from_numpy(np.ascontiguousarray(v).reshape(-1)).cuda() for v in (L, w, w, R, x)]
    y, ws = torch.full((m * n,), float("nan"), dtype=torch.float64, device="cuda"), plan.workspace()
    heff.heff_apply(plan.handle, *t, y, ws)
    assert heff.heff_workspace_status(plan.handle, ws) == 0
    return y.cpu().numpy().reshape(m, n)


def _operands(fill, m, k, n, rng):
    """(m x k, k x n) whose large elements do not meet."""
    a, b = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    if fill == "opposite":                    # a falls off along the contraction index, b rises
        w = np.exp(-40.0 * np.arange(k) / k)
        a, b = a * w, b / w[:, None]
    elif fill == "gauge":                     # D and its inverse between the operands
        d = 2.0 ** rng.integers(-40, 41, k)
        a, b = a * d, b / d[:, None]
    elif fill == "spike":                     # the row's largest element meets a zero
        a[:, :-1] *= 1e-20
        b[-1] = 0.0
    elif fill == "sparse":                    # one element a row, graded columns
        a = np.eye(m, k) * 2.0 ** rng.integers(-3, 4, (m, 1))
        b = b * np.exp(-60.0 * rng.random((k, 1)))
    elif fill == "mixed":                     # a few such rows and columns among others
        a[::7] *= np.exp(-40.0 * np.arange(k) / k)
        b[:, ::5] *= np.exp(40.0 * np.arange(k) / k)[:, None]
    elif fill == "coherent":                  # low digits all alike below a single large element: the
        v = (0x007f7f7f7f7f7f7f + 0.0) / 2.0 ** 62   # low accumulators pass 2^24
        a, b = np.full((m, k), v), np.full((k, n), v)
        a[:, 0], b[-1] = 0.9, 0.9
    return a, b


@pytest.mark.parametrize("m,n", [(1, 1), (17, 5), (33, 70), (64, 31), (130, 96), (300, 70), (520, 33)])
@pytest.mark.parametrize("fill", ["opposite", "gauge", "spike", "sparse", "mixed", "coherent"])
def test_matvec_within_the_bound_of_an_fp64_sum(m, n, fill):
    rng = np.random.default_rng([m, n])
    # both contractions: L x with R = 1, and x R^T with L = 1
    L, x = _operands(fill, m, m, n, rng)
    one = np.eye(n)
    ld = lambda v: v.astype(np.longdouble)
    err = np.abs(_matvec(L, x, one) - ld(L) @ ld(x))
    assert (err <= _bound(L, x)).all()
    x, rt = _operands(fill, n, m, m, rng)     # n x m by m x m
    err = np.abs(_matvec(np.eye(n), x, np.ascontiguousarray(rt.T)) - ld(x) @ ld(rt))
    assert (err <= _bound(x, rt)).all()


def test_matvec_with_identities_is_exact():
    rng = np.random.default_rng(8)
    x = rng.standard_normal((210, 150)) * np.exp(-50.0 * rng.random((210, 150)))
    x[rng.random(x.shape) < 0.2] = 0.0
    assert (_matvec(np.eye(210), x, np.eye(150)) == x).all()

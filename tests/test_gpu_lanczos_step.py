"""The cooperative Lanczos step: one block and many, the basis piece in shared memory and in
place, few and many vectors per block, and capture into a CUDA graph."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(name, precision):
    import torch
    import workloads as wl
    from paper_2007_05540_gb300 import heff
    from tests.helpers import library_problem
    w = wl.workload_by_name(name)
    lays, bufs = library_problem(w)
    plan = heff.Plan(*lays, bufs["W1"], bufs["W2"], precision, "f64")
    d = [torch.from_numpy(np.asarray(bufs[k])).cuda() for k in ("L", "W1", "W2", "R")]
    x = torch.from_numpy(bufs["x"][0]).cuda()
    return plan, d, x, plan.workspace()


def _lanczos(plan, d, x, ws, n):
    import torch
    from paper_2007_05540_gb300 import heff
    lz = torch.empty(heff.heff_lanczos_workspace_size(plan.handle, n), dtype=torch.uint8, device="cuda")
    res = torch.zeros(3 + 2 * (n + 1), dtype=torch.float64, device="cuda")
    xo = torch.empty_like(x)
    run = lambda: heff.heff_lanczos(plan.handle, *d, x, n, xo, res, ws, lz)
    return run, res, xo, lz


# spin_m24: one block; spin_m4096: the vectors' pieces (n / 152 SMs) exceed shared memory
@pytest.mark.parametrize("name,n", [("spin_m24", 1), ("spin_m24", 40), ("spin_m200", 17), ("spin_m1024", 60),
                                    ("spin_m4096", 9)])
def test_ritz_pair_is_consistent(name, n):
    """theta is the Rayleigh quotient of the returned vector, and the residual estimate its
    residual: both hold exactly for a Krylov basis that is orthonormal."""
    import torch
    from paper_2007_05540_gb300 import heff
    prec = "fp64" if name in ("spin_m24", "spin_m200") else "bf16x3"
    plan, d, x, ws = _problem(name, prec)
    run, res, xo, _ = _lanczos(plan, d, x, ws, n)
    run()
    y = torch.empty_like(xo)
    heff.heff_apply(plan.handle, *d, xo, y, ws)
    assert heff.heff_workspace_status(plan.handle, ws) == 0
    theta, est, dim = (float(v) for v in res[:3])
    # the matvec's own accuracy: FP64, or about 1e-5 of ||H x|| in BF16x3
    tol = 1e-12 if prec == "fp64" else 5e-5
    scale = float(y.norm())
    assert dim == n
    assert abs(float(torch.dot(xo, xo)) - 1) < 1e-12
    assert abs(float(torch.dot(xo, y)) - theta) < tol * scale
    assert abs(float((y - theta * xo).norm()) - est) < tol * scale + 1e-9 * est


def test_lanczos_in_a_graph():
    import torch
    plan, d, x, ws = _problem("spin_m200", "bf16x3")
    run, res, xo, _ = _lanczos(plan, d, x, ws, 12)
    run()
    ref, rx = res.clone(), xo.clone()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        run()
    for _ in range(2):
        res.zero_()
        xo.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(res[:3], ref[:3]) and torch.equal(xo, rx)

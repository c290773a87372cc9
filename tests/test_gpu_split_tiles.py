"""GEMM 2 tiles whose contraction is split over several CTAs (few long tiles, m of about 1000): the
parts are added in a fixed order, so repeated calls, every tile variant, batched applies and a
graph replay give the same bits; an FP64 plan's parts also when some of them run in FP64 arithmetic."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(name, prec, io, nb=1):
    import torch
    import workloads as wl
    from paper_2007_05540_gb300 import heff
    from tests.helpers import library_problem
    w = wl.workload_by_name(name)
    lays, bufs = library_problem(w)
    dt = torch.float64 if io == "f64" else torch.float32
    d = [torch.from_numpy(np.asarray(bufs[k])).to("cuda", dt) for k in ("L", "W1", "W2", "R")]
    x = torch.from_numpy(bufs["x"][0]).to("cuda", dt)
    plan = heff.Plan(*lays, bufs["W1"], bufs["W2"], prec, io, max_batch=nb)
    return heff, plan, d, x, plan.workspace()


@pytest.mark.parametrize("prec,io", [("bf16x3", "f32"), ("bf16x3", "f64"), ("tf32x3", "f32"), ("fp64", "f64")])
@pytest.mark.parametrize("name", ["spin_m1024", "spin_m384"])
@pytest.mark.parametrize("nb", [1, 2])                # plans for batches are not cut (but TF32x3's)
def test_same_bits_on_every_route(name, prec, io, nb):
    import torch
    heff, plan, d, x, ws = _problem(name, prec, io, nb)
    y, z = torch.empty_like(x), torch.full_like(x, float("nan"))
    heff.heff_apply(plan.handle, *d, x, y, ws)
    assert heff.heff_workspace_status(plan.handle, ws) == 0
    assert bool(torch.isfinite(y).all())
    heff.heff_apply(plan.handle, *d, x, z, ws)
    assert torch.equal(y, z)
    for tiles in (128, 512, 256) if prec != "fp64" else ():
        heff.heff_plan_select_tiles(plan.handle, tiles, tiles)
        z.fill_(float("nan"))
        heff.heff_apply(plan.handle, *d, x, z, ws)
        assert torch.equal(y, z), tiles
    zs = [torch.full_like(x, float("nan")) for _ in range(nb)]
    heff.heff_apply_batched(plan.handle, *d, [x] * nb, zs, ws)
    assert all(torch.equal(y, z) for z in zs)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        heff.heff_apply(plan.handle, *d, x, z, ws)
    for _ in range(2):
        z.fill_(float("nan"))
        g.replay()
        assert torch.equal(y, z)


def test_parts_in_fp64_arithmetic():
    """One block of x beyond the fixed-point range: K x is linear in that block's scale."""
    import torch
    heff, plan, d, x, ws = _problem("spin_m1024", "fp64", "f64")
    xl = plan.layouts[4]
    _, off, size = sorted(xl.blocks(), key=lambda b: -b[2])[0]
    lone, rest = torch.zeros_like(x), x.clone()
    lone[off:off + size] = x[off:off + size]
    rest[off:off + size] = 0.0
    ya, yb, y = (torch.empty_like(x) for _ in range(3))
    heff.heff_apply(plan.handle, *d, lone, ya, ws)
    heff.heff_apply(plan.handle, *d, rest, yb, ws)
    heff.heff_apply(plan.handle, *d, rest + lone * 2.0 ** 450, y, ws)
    assert heff.heff_workspace_status(plan.handle, ws) == 0
    ref = ya * 2.0 ** 450 + yb
    assert float(((y - ref) * 2.0 ** -450).norm() / ya.norm()) < 1e-13
    far = ya == 0.0                            # rows that the block does not reach keep their digits
    assert float((y - yb)[far].norm()) <= 1e-13 * float(yb.norm())

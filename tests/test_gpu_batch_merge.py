"""Batched applies whose vectors share tensor-core tiles: every vector equals its single apply
bitwise, for batch sizes around the slot counts (2, 4, 8 to a tile) and all tile variants."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,prec,io,nb,tiles", [
    ("spin_m64", "bf16x3", "f32", 40, 0), ("spin_m384", "bf16x3", "f32", 2, 0), ("spin_m384", "tf32x3", "f64", 9, 128),
    ("electron_m96", "bf16x3", "f64", 7, 512), ("electron_m96", "tf32x3", "f32", 65, 0),
    ("electron_m256", "bf16x3", "f32", 3, 0), ("electron_m256", "bf16x3", "f32", 8, 128)])
def test_merged_batch_equals_single_applies(name, prec, io, nb, tiles):
    import torch
    import workloads as wl
    from paper_2007_05540_gb300 import heff
    from tests.helpers import library_problem
    w = wl.workload_by_name(name)
    lays, bufs = library_problem(w)
    plan = heff.Plan(*lays, bufs["W1"], bufs["W2"], prec, io, max_batch=nb)
    dt = torch.float64 if io == "f64" else torch.float32
    d = [torch.from_numpy(np.asarray(bufs[k])).to("cuda", dt) for k in ("L", "W1", "W2", "R")]
    g = torch.Generator(device="cuda").manual_seed(3)
    xs = [torch.randn(lays[4].nelem, dtype=dt, device="cuda", generator=g) for _ in range(nb)]
    ws = plan.workspace()
    ws.fill_(0xff)                            # NaNs wherever nothing is written
    ys = [torch.full_like(x, float("nan")) for x in xs]
    if tiles:
        heff.heff_plan_select_tiles(plan.handle, tiles, tiles)
    heff.heff_apply_batched(plan.handle, *d, xs, ys, ws)
    assert heff.heff_workspace_status(plan.handle, ws) == 0
    y = torch.empty_like(xs[0])
    for b in range(nb):
        heff.heff_apply(plan.handle, *d, xs[b], y, ws)
        assert torch.equal(y, ys[b]), b

"""Device-side bounded waits give up instead of hanging, and the host learns of it.

A single-block kernel waits, with the GEMM kernels' own mbarrier wait (kind 0) or at the
SVD sweeps' grid barrier (kind 1), on something nothing completes.  The wait must expire
after its cycle limit (about 1.5 s / 1 s), set the workspace's sticky error flag, which
heff_workspace_status reports as HEFF_ERR_TIMEOUT and clears, and leave the context
usable: an apply afterwards still matches the oracle.  No kernel faults or traps.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected only with -m gpu on CPU
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2007_05540_gb300 import heff                       # noqa: E402
from tests.helpers import oracle_flat                           # noqa: E402
from tests.test_gpu_parity import Lib, _compare, _oracle, TOL  # noqa: E402

import workloads as wl                                          # noqa: E402

HEFF_ERR_TIMEOUT = -6


@pytest.mark.parametrize("kind", [0, 1])
def test_bounded_wait_expires_and_context_stays_usable(kind):
    w = wl.workload_by_name("spin_m64")
    lib = Lib(w, "bf16x3")
    y_ref = oracle_flat(lib.lays[4], _oracle(w))
    _compare(lib.apply(), y_ref, TOL["bf16x3"])
    assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == 0

    ms = heff.heff_wait_selftest(lib.plan.handle, lib.ws, kind)
    print(f"kind {kind}: wait expired after {ms:.1f} ms")
    # the limits are 3 * 2^30 (kind 0) and 2^31 (kind 1) SM cycles: ~0.5-2.5 s at the
    # clocks a GB300 runs (2.07 GHz at most)
    assert 300.0 < ms < 5000.0, ms
    assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == HEFF_ERR_TIMEOUT
    assert "expired" in heff.heff_last_error()
    assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == 0   # read clears it

    _compare(lib.apply(), y_ref, TOL["bf16x3"])
    assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == 0


def test_workspace_status_fp64_plan_has_no_waits():
    w = wl.workload_by_name("spin_m64")
    lib = Lib(w, "fp64")
    _compare(lib.apply(), oracle_flat(lib.lays[4], _oracle(w)), TOL["fp64"])
    assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == 0
    with pytest.raises(heff.HeffError):
        heff.heff_wait_selftest(lib.plan.handle, lib.ws, 0)


def _raise_flag(ws):
    """What an expired wait leaves: 1 in the flag, an int before 28 more bytes of its pattern."""
    head = ws[:ws.numel() // 256 * 256].view(-1, 256)[:, :32]
    at = (head == 0x5A).all(1).nonzero().flatten()
    assert len(at) == 1
    head[int(at[0]), :4] = torch.tensor([1, 0, 0, 0], dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
def test_status_belongs_to_the_workspace(prec):
    """Three workspaces of one plan in turn: an expired wait in the first is reported there, after the plan has
    been used elsewhere; a workspace in which nothing has run has no flag."""
    w = wl.workload_by_name("spin_m64")
    lib = Lib(w, prec)
    lib.apply()
    _raise_flag(lib.ws)
    first = lib.ws
    for _ in range(2):
        lib.ws = lib.plan.workspace().fill_(0xFF)
        assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == 0
        lib.apply()
        assert heff.heff_workspace_status(lib.plan.handle, lib.ws) == 0
    assert heff.heff_workspace_status(lib.plan.handle, first) == HEFF_ERR_TIMEOUT
    assert heff.heff_workspace_status(lib.plan.handle, first) == 0


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
def test_environment_status_belongs_to_the_workspace(prec):
    from tests.test_gpu_env import _dev, _env_case
    old_l, site_l, W_l, new_l, bufs, _ = _env_case("spin_m64", "left", 70, 9)
    t = [_dev(bufs[k]) for k in ("old", "site", "W")]
    plan = heff.heff_env_plan_create(old_l.handle, site_l.handle, W_l.handle, new_l.handle, bufs["W"], "left")
    try:
        size = heff.heff_env_workspace_size(plan)
        a, b = (torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda") for _ in range(2))
        out = torch.empty(new_l.nelem, dtype=torch.float64, device="cuda")
        assert heff.heff_env_status(plan, a) == 0                # nothing has run there
        heff.heff_env_plan_set_precision(plan, prec)
        heff.heff_env_update(plan, *t, out, a)
        _raise_flag(a)
        heff.heff_env_update(plan, *t, out, b)
        assert heff.heff_env_status(plan, b) == 0
        heff.heff_env_plan_set_precision(plan, "bf16x3" if prec == "fp64" else "fp64")
        assert heff.heff_env_status(plan, a) == HEFF_ERR_TIMEOUT
        assert heff.heff_env_status(plan, a) == 0
    finally:
        heff.heff_env_plan_destroy(plan)

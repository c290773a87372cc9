"""GPU environment extension (heff_env_update) against the oracle (Section II-C).

Inputs come from the shared seeded generators: the workload's environment and MPO
tensors and Gaussian site tensors on a new bond with even 2Sz charges (the bond after
one more spin-1/2 site).  Both sides enumerate blocks on their own; the GPU result must
match the oracle's block-by-block extension to 1e-12 relative (FP64).
"""
import numpy as np
import pytest

import workloads as wl
from workloads.fill import site_block
from oracle import env as oenv
from oracle.blocks import BlockTensor, Index
from oracle.heff import mpo_index

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2007_05540_gb300 import heff              # noqa: E402


def _dev(a):
    return torch.from_numpy(np.asarray(a, dtype=np.float64)).to("cuda")


def _env_case(name, side, new_m, new_nsec, seed=31):
    w = wl.workload_by_name(name)
    ph = w.phys
    ones = lambda n: np.ones(n, dtype=np.int32)
    gq, gd = wl.binomial_sectors(new_m, new_nsec, seed, parity=0)      # even charges
    if side == "left":
        bq, bd = w.alpha_q, w.alpha_d            # env_old bond (site's left bond)
        site_idx = [(bq, bd, 1), (ph, ones(len(ph)), 1), (gq, gd, -1)]
        env_old_fill, ch_old, ch_new, W = w.L_block, w.ql, w.qm, w.W1
        new_q, new_d = gq, gd
    else:
        bq, bd = w.beta_q, w.beta_d              # env_old bond (site's right bond)
        site_idx = [(gq, gd, 1), (ph, ones(len(ph)), 1), (bq, bd, -1)]
        env_old_fill, ch_old, ch_new, W = w.R_block, w.qr, w.qm, w.W2
        new_q, new_d = gq, gd
    # library layouts and buffers
    site_l = heff.Layout(site_idx)
    W_l = heff.Layout([(w.ql if side == "left" else w.qm, ones(W.shape[0]), 1), (ph, ones(len(ph)), 1),
                       (ph, ones(len(ph)), -1), (w.qm if side == "left" else w.qr, ones(W.shape[3]), -1)])
    old_l = heff.Layout([(bq, bd, -1), (ch_old, ones(len(ch_old)), 1), (bq, bd, 1)])
    new_l = heff.Layout([(new_q, new_d, -1), (ch_new, ones(len(ch_new)), 1), (new_q, new_d, 1)])
    site_fill = lambda k: site_block(seed + 5, k, (int(site_idx[0][1][k[0]]), int(site_idx[2][1][k[2]])))
    bufs = {"site": site_l.assemble(site_fill), "W": W_l.assemble(lambda k: W[k]),
            "old": old_l.assemble(lambda k: env_old_fill(k))}
    # oracle tensors built from the same generators
    phys_ix = Index(ph, ones(len(ph)))
    site_o = BlockTensor.from_fill([Index(site_idx[0][0], site_idx[0][1]), phys_ix,
                                    Index(site_idx[2][0], site_idx[2][1])], (1, 1, -1), np.zeros(w.nq),
                                   lambda k: site_fill(k))
    old_o = BlockTensor.from_fill([Index(bq, bd), mpo_index(ch_old), Index(bq, bd)], (-1, 1, 1),
                                  np.zeros(w.nq), env_old_fill)
    if side == "left":
        ref = oenv.extend_left(old_o, site_o, W, ch_new)
    else:
        ref = oenv.extend_right(old_o, site_o, W, ch_new)
    ref_flat = new_l.assemble(lambda k: ref.blocks[k])
    return old_l, site_l, W_l, new_l, bufs, ref_flat


# FP64 block products: 1e-12; tensor-core BF16x3 products (two chained contractions, FP32
# accumulation): the BF16 path's 1e-3 bound of the matvec, norm-wise, and every element
# within 20x of it relative to the largest
TOL = {"fp64": 1e-12, "bf16x3": 1e-3}


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
@pytest.mark.parametrize("side", ["left", "right"])
@pytest.mark.parametrize("name,new_m,new_nsec", [("spin_m64", 70, 9), ("spin_m1024", 1100, 31)])
def test_env_update_matches_oracle(name, new_m, new_nsec, side, prec):
    old_l, site_l, W_l, new_l, bufs, ref = _env_case(name, side, new_m, new_nsec)
    plan = heff.heff_env_plan_create(old_l.handle, site_l.handle, W_l.handle, new_l.handle, bufs["W"], side)
    try:
        heff.heff_env_plan_set_precision(plan, prec)
        ws = torch.empty(heff.heff_env_workspace_size(plan), dtype=torch.uint8, device="cuda")
        out = torch.full((new_l.nelem,), float("nan"), dtype=torch.float64, device="cuda")
        heff.heff_env_update(plan, _dev(bufs["old"]), _dev(bufs["site"]), _dev(bufs["W"]), out, ws)
        torch.cuda.synchronize()
        assert heff.heff_env_status(plan, ws) == 0
        y = out.cpu().numpy()
        assert not np.isnan(y).any()
        err = np.linalg.norm(y - ref) / np.linalg.norm(ref)
        merr = np.abs(y - ref).max() / np.abs(ref).max()
        print(f"env {side} {name} {prec}: rel err {err:.2e} (max element {merr:.2e}), "
              f"flops {heff.heff_env_flops(plan):.3e}")
        assert err < TOL[prec] and merr < 20 * TOL[prec]
    finally:
        heff.heff_env_plan_destroy(plan)


def test_env_update_precision_switch_back_to_fp64_is_exact():
    # retiling for the tensor cores and back leaves the FP64 result bitwise unchanged
    old_l, site_l, W_l, new_l, bufs, ref = _env_case("spin_m64", "left", 70, 9)
    plan = heff.heff_env_plan_create(old_l.handle, site_l.handle, W_l.handle, new_l.handle, bufs["W"], "left")
    try:
        ws = torch.empty(heff.heff_env_workspace_size(plan), dtype=torch.uint8, device="cuda")
        outs = []
        for prec in ("fp64", "bf16x3", "fp64"):
            heff.heff_env_plan_set_precision(plan, prec)
            out = torch.empty((new_l.nelem,), dtype=torch.float64, device="cuda")
            heff.heff_env_update(plan, _dev(bufs["old"]), _dev(bufs["site"]), _dev(bufs["W"]), out, ws)
            torch.cuda.synchronize()
            outs.append(out.cpu().numpy())
        assert np.array_equal(outs[0], outs[2])
        assert not np.array_equal(outs[0], outs[1])
        with pytest.raises(heff.HeffError):
            heff.heff_env_plan_set_precision(plan, "tf32x3")
    finally:
        heff.heff_env_plan_destroy(plan)


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
def test_env_update_captured_right_after_the_precision_is_set(prec):
    """create, workspace size, set_precision, update: the update allocates and synchronises nothing, so it can
    be the first thing that a graph captures."""
    old_l, site_l, W_l, new_l, bufs, ref = _env_case("spin_m64", "left", 70, 9)
    t = [_dev(bufs[k]) for k in ("old", "site", "W")]
    make = lambda: heff.heff_env_plan_create(old_l.handle, site_l.handle, W_l.handle, new_l.handle, bufs["W"], "left")
    new = lambda: torch.full((new_l.nelem,), float("nan"), dtype=torch.float64, device="cuda")
    first, plan = make(), make()
    try:
        ws = torch.empty(heff.heff_env_workspace_size(plan), dtype=torch.uint8, device="cuda")
        want, got = new(), new()
        heff.heff_env_plan_set_precision(first, prec)
        heff.heff_env_update(first, *t, want, ws)                   # (the kernels are loaded)
        heff.heff_env_plan_set_precision(plan, "bf16x3" if prec == "fp64" else "fp64")
        torch.cuda.synchronize()
        heff.heff_env_plan_set_precision(plan, prec)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            heff.heff_env_update(plan, *t, got, ws)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want)
    finally:
        heff.heff_env_plan_destroy(first)
        heff.heff_env_plan_destroy(plan)


@pytest.mark.parametrize("side", ["left", "right"])
@pytest.mark.parametrize("name,new_m,new_nsec", [("spin_m64", 70, 9), ("spin_m1024", 1100, 31)])
def test_env_update_in_the_workspace_of_bf16x3(name, new_m, new_nsec, side):
    """The size reported with BF16x3 serves an FP64 update too (on the FP64 units: no digit planes fit); with a
    byte less both precisions refuse it."""
    old_l, site_l, W_l, new_l, bufs, ref = _env_case(name, side, new_m, new_nsec)
    t = [_dev(bufs[k]) for k in ("old", "site", "W")]
    plan = heff.heff_env_plan_create(old_l.handle, site_l.handle, W_l.handle, new_l.handle, bufs["W"], side)
    try:
        full = heff.heff_env_workspace_size(plan)
        heff.heff_env_plan_set_precision(plan, "bf16x3")
        size = heff.heff_env_workspace_size(plan)
        assert size < 0.4 * full
        ws = torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda")
        for prec in ("bf16x3", "fp64"):
            heff.heff_env_plan_set_precision(plan, prec)
            out = torch.full((new_l.nelem,), float("nan"), dtype=torch.float64, device="cuda")
            heff.heff_env_update(plan, *t, out, ws)
            torch.cuda.synchronize()
            assert heff.heff_env_status(plan, ws) == 0
            y = out.cpu().numpy()
            assert np.linalg.norm(y - ref) < TOL[prec] * np.linalg.norm(ref)
            assert np.abs(y - ref).max() < 20 * TOL[prec] * np.abs(ref).max()
            with pytest.raises(heff.HeffError) as e:
                heff.heff_env_update(plan, *t, out, ws[:size - 1])
            assert e.value.code == -7
    finally:
        heff.heff_env_plan_destroy(plan)


@pytest.mark.parametrize("side", ["left", "right"])
def test_env_update_past_the_dense_limit(side):
    """An update whose dense operands would pass 64 GiB (264 new channels, each with a copy of the environment's
    4097 rows) while its tensors are small: the block-product lists, in a few MB beside the FP32 copies."""
    rng = np.random.default_rng(5)
    ones = lambda n: np.ones(n, dtype=np.int32)
    ph = np.array([[1], [-1]], dtype=np.int32)
    old = np.array([[0], [2]], dtype=np.int32), np.array([4097, 35], dtype=np.int32)
    new = np.array([[-1], [1], [3]], dtype=np.int32), np.array([5, 70, 9], dtype=np.int32)
    one = np.zeros((1, 1), dtype=np.int32)
    many = np.repeat(np.array([[0], [2], [-2]], dtype=np.int32), [260, 2, 2], axis=0)
    (la, ra), (lc, rc) = ((old, new), (one, many)) if side == "left" else ((new, old), (many, one))
    site_l = heff.Layout([(*la, 1), (ph, ones(2), 1), (*ra, -1)])
    W_l = heff.Layout([(lc, ones(len(lc)), 1), (ph, ones(2), 1), (ph, ones(2), -1), (rc, ones(len(rc)), -1)])
    old_l = heff.Layout([(*old, -1), (one, ones(1), 1), (*old, 1)])
    new_l = heff.Layout([(*new, -1), (many, ones(len(many)), 1), (*new, 1)])
    bufs = {k: rng.standard_normal(lay.nelem) for k, lay in (("site", site_l), ("W", W_l), ("old", old_l))}

    ix = lambda b: Index(b[0], b[1])
    views = lambda lay, k: lay.split(bufs[k])
    W = np.zeros((len(lc), 2, 2, len(rc)))
    for key, v in views(W_l, "W").items():
        W[key] = v[0]
    so, oo = views(site_l, "site"), views(old_l, "old")
    site_o = BlockTensor.from_fill([ix(la), Index(ph, ones(2)), ix(ra)], (1, 1, -1), np.zeros(1), lambda k: so[k])
    old_o = BlockTensor.from_fill([ix(old), mpo_index(one), ix(old)], (-1, 1, 1), np.zeros(1), lambda k: oo[k])
    ref = (oenv.extend_left if side == "left" else oenv.extend_right)(old_o, site_o, W, many)
    ref = new_l.assemble(lambda k: ref.blocks[k])

    plan = heff.heff_env_plan_create(old_l.handle, site_l.handle, W_l.handle, new_l.handle, bufs["W"], side)
    try:
        t = [_dev(bufs[k]) for k in ("old", "site", "W")]
        size = heff.heff_env_workspace_size(plan)
        assert size < 1 << 28
        ws = torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda")
        for prec in ("fp64", "bf16x3", "fp64"):
            heff.heff_env_plan_set_precision(plan, prec)
            assert heff.heff_env_workspace_size(plan) == size
            out = torch.full((new_l.nelem,), float("nan"), dtype=torch.float64, device="cuda")
            heff.heff_env_update(plan, *t, out, ws)
            torch.cuda.synchronize()
            assert heff.heff_env_status(plan, ws) == 0
            y = out.cpu().numpy()
            assert np.linalg.norm(y - ref) < TOL[prec] * np.linalg.norm(ref)
            assert np.abs(y - ref).max() < 20 * TOL[prec] * np.abs(ref).max()
    finally:
        heff.heff_env_plan_destroy(plan)

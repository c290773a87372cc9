"""A host allocation that fails inside a C entry comes back as HEFF_ERR_OOM: no exception crosses the C call.

A child process has `operator new` replaced by one that fails once, at a chosen allocation of at least a chosen
size.  Without a device this covers the planning and the tables of another precision; with one, also the staging
copies of the uploads (buffers of a few KB and more; smaller allocations may be the CUDA runtime's).
"""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOOK = r"""
#include <cstdlib>
#include <new>
static thread_local long left_ = -1;
static thread_local std::size_t least_ = 0;
extern "C" void arm(long n, std::size_t least) { left_ = n; least_ = least; }
extern "C" long disarm() { const long n = left_; left_ = -1; return n; }
void* operator new(std::size_t n) {
    if (left_ >= 0 && n >= least_ && left_-- == 0) throw std::bad_alloc();
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""
CHILD = r"""
import ctypes, sys
import numpy as np
import workloads as wl
from paper_2007_05540_gb300 import heff
least = int(sys.argv[2])
hook = ctypes.CDLL(sys.argv[1])
hook.arm.argtypes, hook.disarm.restype = [ctypes.c_long, ctypes.c_size_t], ctypes.c_long
w = wl.workload_by_name("spin_m64")
ones = lambda n: np.ones(n, dtype=np.int32)
Ll, W1l, W2l, Rl, xl = heff.heff_layouts((w.alpha_q, w.alpha_d), (w.beta_q, w.beta_d), w.phys, w.ql, w.qm, w.qr)
W1, W2 = W1l.assemble(lambda k: w.W1[k]), W2l.assemble(lambda k: w.W2[k])
gq, gd = wl.binomial_sectors(70, 9, 31, parity=0)
site = heff.Layout([(w.alpha_q, w.alpha_d, 1), (w.phys, ones(2), 1), (gq, gd, -1)])
right = heff.Layout([(gq, gd, 1), (w.phys, ones(2), 1), (w.beta_q, w.beta_d, -1)])
env = heff.Layout([(gq, gd, -1), (w.qm, ones(len(w.qm)), 1), (gq, gd, 1)])

def plan(prec):
    return (lambda: heff.Plan(Ll, W1l, W2l, Rl, xl, W1, W2, prec, "f64"), lambda p: None)

def env_plan():
    return heff.heff_env_plan_create(Ll.handle, site.handle, W1l.handle, env.handle, W1, "left")

def grad_plan():
    return heff.heff_grad_plan_create(Ll.handle, W1l.handle, W2l.handle, Rl.handle, xl.handle, W1, W2, 0)

def other(create, set_precision, destroy):
    state = {}
    def before():
        state["p"] = create()
    return before, lambda: set_precision(state["p"], "bf16x3"), lambda _: destroy(state["p"])

nothing = lambda: None
CASES = {
    "plan fp64": (nothing, *plan("fp64")),
    "plan bf16x3": (nothing, *plan("bf16x3")),
    "env": (nothing, env_plan, heff.heff_env_plan_destroy),
    "env precision": other(env_plan, heff.heff_env_plan_set_precision, heff.heff_env_plan_destroy),
    "grad": (nothing, grad_plan, heff.heff_grad_plan_destroy),
    "grad precision": other(grad_plan, heff.heff_grad_plan_set_precision, heff.heff_grad_plan_destroy),
    "two-site": (nothing, lambda: heff.heff_two_site_create(site.handle, right.handle, xl.handle),
                 heff.heff_two_site_destroy),
}
for name, (before, call, after) in CASES.items():
    before()
    call_result = call()                       # (the CUDA runtime, if there is one, is up)
    after(call_result)
    before()
    hook.arm(1 << 40, least)
    r = call()
    n = (1 << 40) - hook.disarm()
    after(r)
    picks = sorted(set(range(min(n, 12))) | set(int(v) for v in np.linspace(0, n - 1, 40)) |
                   set(range(max(0, n - 25), n))) if n else []
    failed = 0
    for k in picks:
        before()
        hook.arm(k, least)
        r, code = None, 0
        try:
            r = call()
        except heff.HeffError as e:
            code = e.code
        hook.disarm()
        assert code in (0, -4), (name, k, n, code)
        failed += code == -4
        if code == 0 or name.endswith("precision"):
            after(r)
    print(name, n, len(picks), failed, flush=True)
    assert failed > 0 or n == 0, name
print("done")
"""


def _run(tmp_path, least):
    src, lib = tmp_path / "hook.cpp", tmp_path / "hook.so"
    src.write_text(HOOK)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    p = subprocess.run([sys.executable, "-c", CHILD, str(lib), str(least)], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT), timeout=300)
    print(p.stdout, p.stderr)
    assert p.returncode == 0 and p.stdout.endswith("done\n"), p.stderr[-2000:]


def test_failed_host_allocations_are_reported(tmp_path):
    _run(tmp_path, 0)


@pytest.mark.gpu
def test_failed_host_allocations_around_uploads_are_reported(tmp_path):
    _run(tmp_path, 2048)

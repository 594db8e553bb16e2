"""Nothing throws through the C interface: with every C++ allocation failing, calls still return a status.

`operator new` is replaced for a child process (a preloaded library with a switch), since an exception that leaves an
extern "C" function ends the process."""
import os
import subprocess
import sys

import pytest

from paper_1908_05460_b200 import build as build_mod

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NEW = r"""
#include <cstdlib>
#include <new>
static thread_local int failing = 0;
extern "C" void fail_new(int on) { failing = on; }
static void* get(std::size_t n) { return failing ? nullptr : std::malloc(n ? n : 1); }
void* operator new(std::size_t n) { void* p = get(n); if (!p) throw std::bad_alloc(); return p; }
void* operator new[](std::size_t n) { void* p = get(n); if (!p) throw std::bad_alloc(); return p; }
void* operator new(std::size_t n, const std::nothrow_t&) noexcept { return get(n); }
void* operator new[](std::size_t n, const std::nothrow_t&) noexcept { return get(n); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
void operator delete[](void* p, std::size_t) noexcept { std::free(p); }
"""
HEAD = r"""
import ctypes, os, sys
fail = ctypes.CDLL(os.environ["LD_PRELOAD"]).fail_new
import torch
from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200.layers import ConvLayer
lib = B.load()
def starved(call):
    fail(1)
    r = call()
    fail(0)
    return r
"""
PLANS = HEAD + r"""
for n in range(1, 40):
    d = B.make_desc(ConvLayer("l", n, 64, 8, 8, 64, 3, 3, 1, 1), torch.bfloat16)
    out = ctypes.c_size_t(0)
    for m in (B.METHOD_EXACT, B.METHOD_TOP1):
        assert starved(lambda: lib.gaconv_workspace_size(ctypes.byref(d), m, ctypes.byref(out))) == 0
        assert out.value == B.gaconv_workspace_size(d, m)
h = ctypes.c_void_p()
assert starved(lambda: lib.gaconv_schedule_create(ctypes.byref(h), 4, 0, B.METHOD_TOP1, ctypes.c_double(0.0), ctypes.c_uint64(1))) != 0
print("done")
"""
STEPS = HEAD + r"""
sys.path.insert(0, "tests")
from helpers import GpuLayer
from paper_1908_05460_b200 import inputs as I
layers = [ConvLayer("l", 4 + i, 16, 16, 16, 16, 3, 3, 1, 1) for i in range(7)]
gs = [GpuLayer(l, torch.float32, *I.make_layer_inputs(l, torch.float32, 23, i)) for i, l in enumerate(layers)]
s = B.Schedule(7, B.SCHED_EVERY_4TH_LAYER, B.METHOD_RANDOM, 0.0, 3)
want = []
for i, g in enumerate(gs):
    s.run_layer(i, 1, g.x, g.dy, g.dw, g.desc)
    want.append(g.logical_dw())
n, xs, dys, dws, ds = s.pack_step([g.x for g in gs], [g.dy for g in gs], [g.dw for g in gs], [g.desc for g in gs])
stream = torch.cuda.current_stream().cuda_stream
for starve in (True, True, False, True, False, True, True):        # before the first, the second (recorded) and later times
    for g in gs: g.dw.fill_(float("nan"))
    call = lambda: lib.gaconv_schedule_run_step(s._h, 1, n, xs, dys, dws, ds, 3, stream)
    assert (starved(call) if starve else call()) == 0
    for g, w in zip(gs, want): assert (g.logical_dw() == w).all()
print("done")
"""


def _run(tmp_path, program):
    build_mod.build()
    src, so = tmp_path / "new.cpp", tmp_path / "libnew.so"
    src.write_text(NEW)
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-o", str(so), str(src)])
    out = subprocess.run([sys.executable, "-c", program], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT),
                         capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip().endswith("done"), (out.returncode, out.stdout[-500:], out.stderr[-1500:])


def test_plans_without_host_memory(tmp_path):
    _run(tmp_path, PLANS)


@pytest.mark.gpu
def test_steps_without_host_memory(tmp_path):
    _run(tmp_path, STEPS)

"""A handle's first compute call builds and uploads its layout: out of host memory anywhere in there is a status, nothing has
been launched, and the same call works once there is memory.  A child process runs with an operator new that fails on demand,
for allocations made from the library's own code."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAILING_NEW = r"""
#include <atomic>
#include <cstdlib>
#include <new>
static std::atomic<long> left_{-1};
static std::atomic<unsigned long> lo_{0}, hi_{0};
static void* get(size_t n, unsigned long from) {
  if (from >= lo_ && from < hi_) {
    long left = left_.load();
    while (left >= 0 && !left_.compare_exchange_weak(left, left - 1)) {}
    if (left == 0) return nullptr;
  }
  return std::malloc(n ? n : 1);
}
void* operator new(size_t n) {
  void* p = get(n, (unsigned long)__builtin_return_address(0));
  if (!p) throw std::bad_alloc();
  return p;
}
void* operator new(size_t n, const std::nothrow_t&) noexcept { return get(n, (unsigned long)__builtin_return_address(0)); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
extern "C" void fail_at(long k, unsigned long lo, unsigned long hi) { lo_ = lo; hi_ = hi; left_ = k; }
extern "C" int failed() { const bool f = left_ < 0; left_ = -1; return f; }
"""

CHILD = r"""
import ctypes, sys
import torch
import rt3d_synth as synth
from paper_2007_09835_b200 import binding as B, nets

new = ctypes.CDLL(sys.argv[1])
new.fail_at.argtypes = [ctypes.c_long, ctypes.c_ulong, ctypes.c_ulong]
lines = [l.split() for l in open("/proc/self/maps") if l.rstrip().endswith("/librt3d.so")]
spans = [tuple(int(v, 16) for v in l[0].split("-")) for l in lines if "x" in l[1]]
lo, hi = min(a for a, _ in spans), max(b for _, b in spans)
seen = 0
for dtype in (torch.float32, torch.bfloat16):
    spec = synth.ConvSpec("l", 160, 160, (3, 3, 3), (1, 1, 1), (1, 1, 1), True)
    L = synth.make_layer(spec, 3, 0, 4, 4, "bernoulli", 0.4)
    make = lambda: nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, dtype)
    x = nets.to_device(synth.make_input(1, (1, 4, 12, 12, 160)), dtype)
    want = make()(x)
    for k in range(10000):
        lay, y = make(), torch.zeros_like(want)
        a = (ctypes.byref(B.tensor_desc(x, 160)), lay.packed.handle, B._bias_ptr(lay.bias),
             ctypes.byref(B._params(spec.stride, spec.pad, True, 0)), ctypes.byref(B.tensor_desc(y, 160)), B._stream_ptr(None))
        launches = B.rt3d_launch_count()
        new.fail_at(k, lo, hi)
        s = B.lib().rt3d_conv3d_sparse(*a)
        hit = new.failed()
        assert s in (B.OK, B.ERR_ALLOC) and (hit or s == B.OK), (k, s)
        if s == B.ERR_ALLOC:
            seen += 1
            assert B.rt3d_launch_count() == launches and not y.any()
            assert B.lib().rt3d_conv3d_sparse(*a) == B.OK, k
        assert torch.equal(y, want), k
        if not hit:
            break
assert B.rt3d_last_device_status() == B.OK
print("ok", seen)
"""


@pytest.mark.gpu
def test_first_call_without_memory_is_a_status(tmp_path):
    (tmp_path / "new.cpp").write_text(FAILING_NEW)
    so = str(tmp_path / "libnew.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-o", so, str(tmp_path / "new.cpp")])
    env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, so], capture_output=True, text=True, timeout=300, env=env, cwd=ROOT)
    assert r.returncode == 0, (r.returncode, r.stdout[-1000:], r.stderr[-2000:])
    assert r.stdout.startswith("ok ") and int(r.stdout.split()[1]) >= 20, r.stdout

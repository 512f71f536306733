"""Host side of the library against a stand-in for the CUDA runtime
(fake_cudart.c): each test runs a child process with it preloaded, which calls
the C entry points on made-up device addresses and reports what the runtime
was asked for.  No GPU, no kernel runs."""
import json
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

# Helpers of the children: plans and calls over made-up addresses, 16-byte
# aligned and far from each other.
CHILD = """
import ctypes, json, sys
import numpy as np
sys.path.insert(0, %r)
from paper_1601_07378_gb300 import synth, vloc
lib, rt = vloc.load(), ctypes.CDLL(None)
rt.fake_set_free.argtypes = [ctypes.c_size_t]
rt.fake_allocated.restype = ctypes.c_size_t
rt.fake_launch_stream.restype = ctypes.c_size_t
def plan(n, r, flags, chunk=0):
    g = synth.sphere_glist(*n, r)
    if flags & vloc.VLOC_GAMMA:
        g = synth.half_sphere(g)
    g = np.ascontiguousarray(g, dtype=np.int32)
    h = ctypes.c_void_p()
    rc = lib.vloc_plan_create(ctypes.byref(h), *n, g.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), len(g), flags, chunk, None)
    assert rc == 0, rc
    return h
def info(h):
    i = vloc.VlocInfo()
    assert lib.vloc_get_info(h, ctypes.byref(i)) == 0
    return i
addr = lambda k: (1 << 44) + (k << 38)
def done(x):
    print("RESULT " + json.dumps(x))
""" % ROOT

# operator new of the child: allocation number fake_new_at (counted from the
# call of that function) throws, with no memory to spare.
NEW = """
#include <cstdlib>
#include <new>
static long g_left = -1;
extern "C" void fake_new_at(long k) { g_left = k; }
void* operator new(std::size_t n) {
    if (g_left == 0) throw std::bad_alloc();
    if (g_left > 0) --g_left;
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1601_07378_gb300 import build
    if not sys.platform.startswith("linux") or shutil.which("gcc") is None:
        pytest.skip("needs gcc and LD_PRELOAD")
    build.build()
    tmp = tmp_path_factory.mktemp("fake")
    so, new = str(tmp / "libfake_cudart.so"), str(tmp / "libfake_new.so")
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-O1", "-Wno-builtin-declaration-mismatch",
                           "-I" + os.path.join(build._cuda_home(), "include"), "-o", so, os.path.join(HERE, "fake_cudart.c")])
    (tmp / "new.cpp").write_text(NEW)
    subprocess.check_call(["g++", "-shared", "-fPIC", "-O1", "-o", new, str(tmp / "new.cpp")])

    def child(code):
        env = dict(os.environ, LD_PRELOAD=so + ":" + new)
        p = subprocess.run([sys.executable, "-c", CHILD + code], env=env, capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, p.stdout + p.stderr
        return json.loads([ln for ln in p.stdout.splitlines() if ln.startswith("RESULT ")][-1][7:])
    return child


# The kernels with more than 48 KB of dynamic shared memory: the fused y/x
# passes, the FP64 and double-float passes, the dL/dV pass.
@pytest.mark.parametrize("n,r,flags", [((96, 96, 96), 24, "VLOC_F32"), ((144, 144, 144), 36, "VLOC_F32"),
                                       ((96, 96, 96), 24, "VLOC_F64"), ((120, 120, 120), 30, "VLOC_F64"),
                                       ((96, 96, 96), 24, "VLOC_F64 | vloc.VLOC_DOUBLE_FLOAT"),
                                       ((96, 96, 100), 30, "VLOC_F64"), ((54, 54, 54), 13, "VLOC_F64")])
def test_every_device_gets_the_shared_memory_limits(run, n, r, flags):
    """Plans on two devices in one process: the limit is the kernel's on one
    device, so the second device's launches need it raised again; a device's
    second call does not."""
    out = run(f"""
res = []
for dev in (0, 1, 0):
    rt.fake_set_device(dev)
    h = plan({n!r}, {r}, vloc.{flags}, 16)
    before = rt.fake_limits()
    rcs = [lib.vloc_apply(h, addr(0), addr(1), 16, addr(2), None), lib.vloc_density(h, addr(0), None, 16, addr(3), None),
           lib.vloc_backward(h, addr(0), addr(4), addr(1), 16, addr(2), addr(3), None)]
    mid = rt.fake_limits()
    rcs.append(lib.vloc_apply(h, addr(0), addr(1), 16, addr(2), None))
    res.append([rcs, mid - before, rt.fake_limits() - mid])
done(res)
""")
    assert [r[0] for r in out] == [[0] * 4] * 3
    assert out[0][1] == out[1][1]      # the second device as the first
    assert out[2][1] == 0 and [r[2] for r in out] == [0] * 3


@pytest.mark.parametrize("flags", ["VLOC_F32", "VLOC_F64", "VLOC_F32 | vloc.VLOC_GAMMA"])
@pytest.mark.parametrize("n,r", [((144, 144, 144), 3), ((144, 144, 144), 9), ((96, 96, 96), 5), ((128, 100, 96), 6.5),
                                 ((96, 96, 96), 24), ((144, 144, 144), 36), ((54, 54, 54), 13), ((48, 48, 48), 2)])
def test_automatic_chunk_keeps_the_documented_workspace(run, n, r, flags):
    """max_bands_per_chunk <= 0: the per-band workspace of a chunk (cylinder,
    and slab or dense rows) stays within 6 GiB and a sixteenth of the free
    memory, whatever the sphere; the V / density accumulators and the Gamma
    buffers are apart."""
    out = run(f"""
res = []
for free in (270 << 30, 24 << 30):
    rt.fake_set_free(free)
    h = plan({n!r}, {r}, vloc.{flags})
    i = info(h)
    res.append([free, i.chunk_bands, i.workspace_bytes, i.npw])
done(res)
""")
    N = n[0] * n[1] * n[2]
    elem = 16 if "F64" in flags else 8
    for free, chunk, ws, npw in out:
        groups = (max(1, max(chunk, 2) // 2) + 15) // 16
        ws -= N * 8 * (1 + groups)
        if "GAMMA" in flags:
            ws -= 2 * chunk * (2 * npw - 1) * elem    # G = 0 is its own mirror
        assert 1 <= chunk <= 2048
        assert ws <= min(6 << 30, free // 16)
        assert ws * (chunk + 1) > min(6 << 30, free // 16) * chunk or chunk == 2048    # and uses it


def test_given_chunk_that_does_not_fit_with_the_dense_rows(run):
    """A small sphere on a large grid with a chunk sized by the caller: where
    the dense rows of the three-launch form do not fit, the plan is made for
    five launches; where not even the slab does, the call fails."""
    out = run("""
def create(free):
    rt.fake_set_free(free)
    g = np.ascontiguousarray(synth.sphere_glist(96, 96, 96, 4), dtype=np.int32)
    h = ctypes.c_void_p()
    rc = lib.vloc_plan_create(ctypes.byref(h), 96, 96, 96, g.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), len(g),
                              vloc.VLOC_F32, 1024, None)
    if rc:
        return [rc, None, None]
    n0 = rt.fake_launches()
    rcs = [lib.vloc_apply(h, addr(0), addr(1), 64, addr(2), None), lib.vloc_density(h, addr(0), None, 64, addr(3), None)]
    ws = info(h).workspace_bytes
    return [rc, rcs, ws, lib.vloc_plan_destroy(h)]
done([create(8 << 30), create(2 << 30), create(256 << 20), [rt.cudaGetLastError(), rt.fake_allocated()]])
""")
    assert out[0][:2] == [0, [0, 0]] and out[1][:2] == [0, [0, 0]]
    assert out[1][2] <= 2 << 30 and out[1][2] <= out[0][2]
    assert out[2][0] == -4    # VLOC_ERR_ALLOC
    assert out[3] == [0, 0]    # nothing leaks, and the failures leave no error behind


# Two large instances of different lengths: in turn on one branch if both run
# the fused y/x pass on enough bands, else on two branches.
@pytest.mark.parametrize("bands,flags,chunk,branches", [
    (60, "VLOC_F32", 0, 1), (30, "VLOC_F32", 0, 2), (200, "VLOC_F32", 2, 2),    # chunk 2: five launches
    (60, "VLOC_F32 | vloc.VLOC_GAMMA", 0, 1), (30, "VLOC_F32 | vloc.VLOC_GAMMA", 0, 2),
    (120, "VLOC_F32 | vloc.VLOC_GAMMA", 2, 2),
    (60, "VLOC_F64", 0, 2)])
def test_batch_instances_in_turn_or_on_branches(run, bands, flags, chunk, branches):
    out = run(f"""
hs = [plan((n,) * 3, n / 4, vloc.{flags} | vloc.VLOC_GRAPH, {chunk}) for n in (96, 100)]
n0 = rt.fake_launches()
vp = ctypes.c_void_p * 2
rc = lib.vloc_apply_batched(2, vp(*hs), vp(addr(0), addr(1)), vp(addr(2), addr(3)), (ctypes.c_int64 * 2)({bands}, {bands}),
                            vp(addr(4), addr(5)), None)
done([rc, [rt.fake_launch_stream(i) for i in range(n0, rt.fake_launches())]])
""")
    assert out[0] == 0
    assert len(set(out[1])) == branches and 0 not in out[1]


@pytest.mark.parametrize("flags", ["VLOC_F32", "VLOC_F32 | vloc.VLOC_GAMMA", "VLOC_F64", "VLOC_F32 | vloc.VLOC_HOST_ONLY"])
def test_host_memory_that_runs_out_in_plan_creation_is_an_error_code(run, flags):
    """Every host allocation of vloc_plan_create fails in turn (from that one
    on): the call returns VLOC_ERR_ALLOC, frees what it had, and no exception
    reaches the caller."""
    out = run(f"""
n, flags = (24, 24, 24), vloc.{flags}
g = synth.sphere_glist(*n, 6)
g = np.ascontiguousarray(synth.half_sphere(g) if flags & vloc.VLOC_GAMMA else g, dtype=np.int32)
gp = g.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
codes, k = [], 0
while True:
    h = ctypes.c_void_p()
    rt.fake_new_at(k)
    rc = lib.vloc_plan_create(ctypes.byref(h), *n, gp, len(g), flags, 0, None)
    rt.fake_new_at(-1)
    codes.append(rc)
    if rc == 0:
        break
    assert not h.value and rt.fake_allocated() == 0
    k = k + 1 if k < 60 else k + 1 + k // 8
done([codes[:-1], lib.vloc_plan_destroy(h), rt.fake_allocated()])
""")
    assert len(out[0]) > 20 and set(out[0]) == {-4}
    assert out[1:] == [0, 0]


def test_host_memory_that_runs_out_in_a_captured_batch_is_an_error_code(run):
    out = run("""
hs = [plan((n,) * 3, n / 4, vloc.VLOC_F32 | vloc.VLOC_GRAPH) for n in (48, 60, 48)]
vp = ctypes.c_void_p * 3
args = (3, vp(*hs), vp(addr(0), addr(1), addr(2)), vp(addr(3), addr(4), addr(5)), (ctypes.c_int64 * 3)(20, 20, 20),
        vp(addr(6), addr(7), addr(8)), None)
codes, k = [], 0
while not codes or codes[-1]:
    rt.fake_new_at(k)
    codes.append(lib.vloc_apply_batched(*args))
    rt.fake_new_at(-1)
    k += 1
done([codes, rt.fake_captures()])
""")
    assert len(out[0]) > 5 and set(out[0][:-1]) == {-4} and out[0][-1] == 0
    assert out[1] == 0    # every capture that was begun was ended


# Launches of an FP32 apply and a density of 64 bands (the line path: V's
# transpose and three, and three; else five, and K1, K2, x-pass, reduction):
# spheres well inside the quarter band of large grids, cells with one length
# that suits the five launches, Gamma pairs, and what keeps the line path.
@pytest.mark.parametrize("n,r,gamma,apply_line,density_line", [
    ((144, 144, 144), 36, False, True, True), ((144, 144, 144), 12, False, False, True),
    ((128, 128, 128), 32, False, True, True), ((128, 128, 128), 32, True, False, True),
    ((128, 128, 128), 8, False, False, False), ((128, 96, 96), 24, False, False, False),
    ((96, 96, 96), 24, False, True, True), ((96, 96, 96), 4, False, False, False),
    ((100, 100, 100), 25, True, True, True), ((100, 100, 100), 6, False, False, True),
    ((80, 80, 80), 10, False, True, True), ((64, 64, 64), 16, True, True, True), ((64, 64, 64), 4, False, False, False),
    ((90, 96, 100), 3, False, True, None),        # a length without compile-time kernels
    ((128, 128, 40), 10, False, True, True)])     # axes that are no cell's
def test_line_path_where_it_pays(run, n, r, gamma, apply_line, density_line):
    out = run(f"""
h = plan({n!r}, {r}, vloc.VLOC_F32 | {"vloc.VLOC_GAMMA" if gamma else 0})
l = [rt.fake_launches()]
assert lib.vloc_apply(h, addr(0), addr(1), 128, addr(2), None) == 0
l.append(rt.fake_launches())
assert lib.vloc_density(h, addr(0), None, 128, addr(3), None) == 0
l.append(rt.fake_launches())
done([l[1] - l[0], l[2] - l[1]])
""")
    assert out[0] == (4 if apply_line else 5)
    assert density_line is None or out[1] == (3 if density_line else 4)


@pytest.mark.parametrize("call", ["lib.vloc_apply(h, addr(0), addr(1), 20, addr(2), None)",    # profiled
                                  "lib.vloc_apply_host(h, addr(0), addr(1), 4000, addr(2), None)"])
def test_memory_that_runs_out_in_a_call_is_an_error_code(run, call):
    """Host allocations of the profiling records and of the staging schedule,
    and the device allocation of the staging buffers: VLOC_ERR_ALLOC, the call
    works afterwards, and no CUDA error is left for a later launch check."""
    out = run(f"""
h = plan((48, 48, 48), 12, vloc.VLOC_F32)
assert lib.vloc_profile(h, 1) == 0
call = lambda: {call}
codes, k = [], 0
if "host" in {call!r}:
    rt.fake_set_free(1 << 20)
    codes.append(call())
    rt.fake_set_free(64 << 30)
while not codes or codes[-1]:
    rt.fake_new_at(k)
    codes.append(call())
    rt.fake_new_at(-1)
    k += 1
n = ctypes.c_int64()
stats = (vloc.VlocKernelStat * 12)()
assert lib.vloc_get_profile(h, stats) == 0
done([codes, call(), rt.cudaGetLastError(), sum(x.launches for x in stats)])
""")
    assert len(out[0]) >= 3 and set(out[0][:-1]) == {-4} and out[0][-1] == 0
    assert out[1:3] == [0, 0] and out[3] >= 4

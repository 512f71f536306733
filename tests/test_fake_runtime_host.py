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


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1601_07378_gb300 import build
    if not sys.platform.startswith("linux") or shutil.which("gcc") is None:
        pytest.skip("needs gcc and LD_PRELOAD")
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-O1", "-Wno-builtin-declaration-mismatch",
                           "-I" + os.path.join(build._cuda_home(), "include"), "-o", so, os.path.join(HERE, "fake_cudart.c")])

    def child(code):
        env = dict(os.environ, LD_PRELOAD=so)
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
# the fused y/x pass on enough complex bands, else on two branches.
@pytest.mark.parametrize("bands,flags,chunk,branches", [
    (60, "VLOC_F32", 0, 1), (30, "VLOC_F32", 0, 2), (200, "VLOC_F32", 2, 2),    # chunk 2: five launches
    (60, "VLOC_F32 | vloc.VLOC_GAMMA", 0, 2), (120, "VLOC_F32 | vloc.VLOC_GAMMA", 0, 1),    # 30 and 60 pairs
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

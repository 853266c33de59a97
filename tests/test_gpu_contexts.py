"""A second CUDA context on the device: it has its own copy of everything the library keeps in
device variables.  The same calls there give the bits of the first context's.  (In a child
process, which makes the context with the driver's own calls and takes it down again.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_CHILD = r"""
import ctypes, sys
import numpy as np
import paper_2308_00763_gb300 as pf
from paper_2308_00763_gb300 import synth

cu = ctypes.CDLL("libcuda.so.1")


def check(rc, what):
    if rc != 0:
        raise RuntimeError("%s: %d" % (what, rc))


check(cu.cuInit(0), "cuInit")
pf.lib(build_if_missing=True)
v = synth.make_video(96, 80, 3, 4, noise=5.0, seed=51)


def engine(prec):
    f = pf.Filter(v.W, v.H, 3001, 4, prec, stream=0, init=tuple(v.centres[0]), seed=52)
    for frame in v.frames:
        f.step(frame)
    st = f.get_state()
    est = f.estimates(0, v.T)
    f.close()
    return [st["x"], st["y"], st["L"], np.asarray(est)]


def in_second_context(call):
    ctx = ctypes.c_void_p()
    dev = ctypes.c_int()
    check(cu.cuDeviceGet(ctypes.byref(dev), 0), "cuDeviceGet")
    check(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev), "cuCtxCreate")   # (made current)
    try:
        return call()
    finally:
        check(cu.cuCtxDestroy_v2(ctx), "cuCtxDestroy")


def same(a, b):
    for p, q in zip(a, b):
        assert np.array_equal(np.asarray(p).view(np.uint8), np.asarray(q).view(np.uint8))


def run_engine(prec):
    first = engine(prec)
    same(first, in_second_context(lambda: engine(prec)))
    same(first, engine(prec))     # (and the first context is as it was)


def noalloc(prec):   # two frames through the allocation-free entry point, in the current context
    n, size = 5001, {"ref64": 8, "f32": 4, "f16": 2}[prec]

    def alloc(nbytes):
        p = ctypes.c_uint64()
        check(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(nbytes)), "cuMemAlloc")
        return p.value

    frames = alloc(v.frames[:2].nbytes)
    host = np.ascontiguousarray(v.frames[:2])
    check(cu.cuMemcpyHtoD_v2(ctypes.c_uint64(frames), host.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(host.nbytes)),
          "cuMemcpyHtoD")
    slots = [[alloc(n * size) for _ in range(3)] for _ in range(2)]
    cfg = pf.make_config(v.W, v.H, n, 4, prec, init=tuple(v.centres[0]), seed=53)
    hdr = pf.PfStateHeader(magic=0x31534650, precision=cfg.precision, num_particles=n, t=0)
    step = host.strides[0]
    hdr = pf.pf_step_frame_noalloc(cfg, hdr, 0, 0, 0, frames, v.W, *slots[0], stream=0)
    hdr = pf.pf_step_frame_noalloc(cfg, hdr, *slots[0], frames + step, v.W, *slots[1], stream=0)
    out = [np.frombuffer(bytes(hdr), np.uint8)]
    for p in slots[1]:
        a = np.empty(n * size, np.uint8)
        check(cu.cuMemcpyDtoH_v2(a.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint64(p), ctypes.c_size_t(a.nbytes)),
              "cuMemcpyDtoH")
        out.append(a)
    for p in [frames] + slots[0] + slots[1]:
        check(cu.cuMemFree_v2(ctypes.c_uint64(p)), "cuMemFree")
    return out


def run_noalloc(prec):
    engine(prec)                  # (the first context is the library's own choice)
    first = noalloc(prec)
    same(first, in_second_context(lambda: noalloc(prec)))
    same(first, noalloc(prec))


globals()["run_" + sys.argv[1]](sys.argv[2])
print("same bits")
"""


def _child(kind, prec):
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    p = subprocess.run([sys.executable, "-c", _CHILD, kind, prec], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0 and "same bits" in p.stdout, p.stdout + p.stderr


@pytest.mark.parametrize("prec", ["ref64", "f32"])
def test_filter_in_a_second_context(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _child("engine", prec)


@pytest.mark.parametrize("prec", ["ref64", "f32", "f16"])
def test_allocation_free_step_in_a_second_context(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _child("noalloc", prec)

"""Steps on a stream that has a part of the SMs (a green context), so that a launch's CTAs are not all
resident: every tile still finds its predecessors running or done, whatever the number of waves,
and the bits are those of the whole device.
"""
import ctypes

import numpy as np
import pytest

from paper_2308_00763_gb300 import synth

pytestmark = pytest.mark.gpu

SMS = 16


class _Resource(ctypes.Structure):   # CUdevResource: type, padding, union (smCount first)
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sm_count", ctypes.c_uint),
                ("rest", ctypes.c_ubyte * 44)]


@pytest.fixture(scope="module")
def pf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_00763_gb300 as m
    m.lib(build_if_missing=True)
    return m


@pytest.fixture(scope="module")
def part_stream(pf):
    """A stream of a green context of SMS SMs of the current device."""
    import torch
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    dev = ctypes.c_int()
    every, part, rest = _Resource(), _Resource(), _Resource()
    groups, desc = ctypes.c_uint(1), ctypes.c_void_p()
    ctx, stream = ctypes.c_void_p(), ctypes.c_void_p()
    calls = [lambda: cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()),
             lambda: cu.cuDeviceGetDevResource(dev, ctypes.byref(every), 1),
             lambda: cu.cuDevSmResourceSplitByCount(ctypes.byref(part), ctypes.byref(groups), ctypes.byref(every),
                                                    ctypes.byref(rest), 0, SMS),
             lambda: cu.cuDevResourceGenerateDesc(ctypes.byref(desc), ctypes.byref(part), 1),
             lambda: cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, dev, 1),
             lambda: cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0)]
    for call in calls:
        if call() != 0:
            pytest.skip("no green contexts here")
    assert 0 < part.sm_count < every.sm_count
    yield stream.value
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("prec,n,resampler", [
    ("f32", 300001, "systematic"),           # one wave on the whole device
    ("f16", 1 << 20, "systematic"),          # one wave that fills it
    ("f16", 3 * (1 << 20) + 7, "systematic"),   # several waves, tables by tile
    ("f16", (1 << 22) + 9, "systematic"),    # several waves, the tracker's table
    ("ref64", 200003, "stratified"),
    ("f32", (1 << 21) + 5, "multinomial"),   # several waves of the CDF and pull kernels
    ("f32", 70001, "rejection"),
])
def test_tracker_on_a_part_of_the_device(pf, part_stream, prec, n, resampler):
    v = synth.make_video(128, 96, 3, 4, noise=8.0, seed=61)
    got = []
    for stream in (0, part_stream):
        f = pf.Filter(v.W, v.H, n, 4, prec, stream=stream, init=tuple(v.centres[0]), seed=62, resampler=resampler)
        f.run(v.frames)
        e, ms = f.estimates(0, v.T, with_stats=True)
        got.append((np.asarray(e), np.asarray(ms)))
        f.close()
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


def test_batch_on_a_part_of_the_device(pf, part_stream):
    """A batch of several waves whose trackers begin in one wave and end in the next."""
    import torch
    v = synth.make_video(128, 96, 3, 4, noise=8.0, seed=63)
    frames = torch.from_numpy(v.frames).cuda()
    sizes = [200003 if i % 3 == 0 else 5000 + 1000 * i for i in range(48)]
    got = []
    for stream in (0, part_stream):
        cfgs = [pf.make_config(v.W, v.H, n, 4, "f16", init=tuple(v.centres[0]), seed=64 + i) for i, n in enumerate(sizes)]
        b = pf.Batch(cfgs, stream=stream)
        b.set_videos([frames] * len(cfgs))
        b.run(v.T)
        got.append(np.stack([np.asarray(b.estimates(t)) for t in range(v.T)]))
        b.close()
    assert np.array_equal(got[0], got[1])

"""Scenes on a stream that has only some of the GPU's SMs (a green context),
where the ordering's grid barriers cannot be had, and two scenes' points
replaced at the same time on two streams: the transients of an ordinary
stream."""
import ctypes

import numpy as np
import pytest
import torch

import scenes
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

SM_RESOURCE, DEFAULT_STREAM, NON_BLOCKING = 1, 1, 1


def _driver():
    try:
        d = ctypes.CDLL("libcuda.so.1")
        d.cuGreenCtxCreate, d.cuDevSmResourceSplitByCount
    except (OSError, AttributeError):
        pytest.skip("no driver with green contexts")
    return d


def _ok(status):
    if status == 801:
        pytest.skip("green contexts are not supported here")
    assert status == 0, status


@pytest.fixture
def part_stream():
    """A stream of a green context with the smallest set of SMs the GPU grants from 8 up."""
    torch.zeros(1, device="cuda")
    d = _driver()
    whole, part = (ctypes.create_string_buffer(1024) for _ in range(2))  # CUdevResource, with room
    groups, dev = ctypes.c_uint(1), torch.cuda.current_device()
    desc, ctx, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    _ok(d.cuDeviceGetDevResource(dev, whole, SM_RESOURCE))
    _ok(d.cuDevSmResourceSplitByCount(part, ctypes.byref(groups), whole, None, 0, 8))
    sms = int.from_bytes(part.raw[96:100], "little")  # sm.smCount
    assert 8 <= sms < int.from_bytes(whole.raw[96:100], "little")
    _ok(d.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1))
    _ok(d.cuGreenCtxCreate(ctypes.byref(ctx), desc, dev, DEFAULT_STREAM))
    _ok(d.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, NON_BLOCKING, 0))
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    d.cuStreamDestroy_v2(stream)
    d.cuGreenCtxDestroy(ctx)


def _params():
    return scenes.default_params(scan_nx=9, scan_ny=7, wall_half_x=0.5, wall_half_y=0.5, bin_width_s=16e-12,
                                 num_bins=203, window_start_m=0.3, scan_mode="nonconfocal",
                                 laser_xy=(0.2, -0.1), jitter_fwhm_s=60e-12)


def _close(a, b):
    # the same FP32 terms in another order
    assert ((a - b).abs() <= 1e-5 * b.amax(dim=1, keepdim=True)).all()


@pytest.mark.parametrize("n", [1, 513, 20001, 300001])
def test_partition_gives_the_same(part_stream, n):
    from paper_2506_03747_gb300 import nlos
    H.lib()
    prm = nlos.params(_params())
    pts = scenes.random_points(np.random.default_rng(n), n)
    pts[::3, 6] = 0.0  # some without weight
    moved = torch.from_numpy(scenes.random_points(np.random.default_rng(n + 1), n)).cuda()
    back = torch.from_numpy(pts).cuda()
    out = []
    for stream in (torch.cuda.current_stream(), part_stream):
        sc = nlos.scene_create(prm, pts, stream=stream)
        taus = [torch.zeros(sc.num_scan, sc.num_bins, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        nlos.forward(sc, taus[0], stream=stream)
        nlos.scene_set_points(sc, moved, stream=stream)
        nlos.forward(sc, taus[1], stream=stream)
        nlos.scene_set_points(sc, back, stream=stream)
        nlos.forward(sc, taus[2], stream=stream)
        nlos.scene_check(sc, stream=stream)
        torch.cuda.synchronize()
        out.append(taus)
        sc.destroy()
    for a, b in zip(*out):
        assert n < 3 or b.max() > 0
        _close(b, a)


def test_two_streams_at_once():
    from paper_2506_03747_gb300 import nlos
    H.lib()
    n = 300001
    prm = nlos.params(_params())
    pts = [torch.from_numpy(scenes.random_points(np.random.default_rng(k), n)).cuda() for k in range(2)]
    scs = [nlos.scene_create(prm, p) for p in pts]
    ref = [torch.empty(63, 203, device="cuda") for _ in pts]
    for sc, t in zip(scs, ref):
        nlos.forward(sc, t)
    tau = [torch.empty_like(t) for t in ref]
    streams = [torch.cuda.Stream() for _ in pts]
    torch.cuda.synchronize()
    for _ in range(50):
        for sc, p, t, st in zip(scs, pts, tau, streams):
            nlos.scene_set_points(sc, p, stream=st)
            nlos.forward(sc, t, stream=st)
    for sc, st in zip(scs, streams):
        nlos.scene_check(sc, stream=st)
    torch.cuda.synchronize()
    for a, b in zip(tau, ref):
        _close(a, b)

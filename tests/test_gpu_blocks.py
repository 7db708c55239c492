"""Device memory of the weight handles: a freed handle's blocks may serve the next one.  Contents never leak from one handle into the
next, threads and streams do not disturb each other, and what is kept is bounded."""
import ctypes
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2509_21302_b200 as q
import workload
from _util import dev_bf16

pytestmark = pytest.mark.gpu


def _layer(K, N, seed):
    spec = workload.LinearSpec("b", K, N, workload.DIST_NORMAL, seed, 0)
    W, b = spec.weight(), spec.bias()
    c = oracle.smooth_factors(spec.x_calib(16), W)
    return dev_bf16(W), dev_bf16(b), torch.from_numpy(c).cuda(), oracle.prepare_weights(W, c), b


def _check(h, ref, bias, flags):
    v = h.view()
    assert np.array_equal(v["w_scale"].cpu().numpy(), ref["w_scale"]) and np.array_equal(v["amul"].cpu().numpy(), ref["amul"])
    assert (v["bias"] is None) == (bias is None)
    if bias is not None:
        assert np.array_equal(v["bias"].view(torch.int16).cpu().numpy().view(np.uint16), bias)
    if flags in (False, True):
        assert np.array_equal(v["wq"].cpu().numpy(), ref["wq_packed"])
    if flags:
        assert np.array_equal(h.view_c8().cpu().numpy(), ref["wq"])
    assert h.device_status() == 0


@pytest.mark.parametrize("flags", [False, True, "only"])
def test_handles_of_changing_size_one_after_the_other(flags):
    layers = [_layer(K, N, 40 + i) for i, (K, N) in enumerate([(1024, 384), (4096, 128), (1024, 384), (1024, 512), (4096, 128)])]
    for i in range(3):
        for W, b, c, ref, bias in layers:
            with_bias = i != 1
            h = q.prepare_weights(W, b if with_bias else None, c, None, c8=flags)
            _check(h, ref, bias if with_bias else None, flags)
            h.free()


def test_threads_and_streams_prepare_and_free_at_the_same_time():
    layers = [_layer(K, N, 60 + i) for i, (K, N) in enumerate([(1024, 384), (1024, 384), (4096, 128), (1024, 256)])]
    torch.cuda.synchronize()
    failed = []

    def work(i):
        try:
            W, b, c, ref, bias = layers[i]
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(12):
                    h = q.prepare_weights(W, b, c, None, c8=True)
                    _check(h, ref, bias, True)
                    h.free()
        except BaseException as e:      # reported by the main thread
            failed.append(e)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(layers))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed


def test_what_is_kept_is_bounded():
    W, b, c, _, _ = _layer(4096, 1024, 80)
    q.prepare_weights(W, b, c, None, c8="only").free()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    hs = [q.prepare_weights(W, b, c, None, c8="only") for _ in range(48)]       # 200 MB of codes
    for h in hs:
        h.free()
    # at most 64 MB of freed blocks stay with the library (and the allocator's own granules)
    assert free0 - torch.cuda.mem_get_info()[0] <= (64 << 20) + (4 << 20)


class _Capture:
    """A capture of a stream of its own, begun and ended through the runtime API (torch keeps no state about it)."""

    def __init__(self, mode):
        self.rt, self.mode, self.stream = ctypes.CDLL("libcudart.so.12"), mode, ctypes.c_void_p()

    def __enter__(self):
        assert self.rt.cudaStreamCreate(ctypes.byref(self.stream)) == 0
        assert self.rt.cudaStreamBeginCapture(self.stream, self.mode) == 0
        return self

    def __exit__(self, *exc):
        graph = ctypes.c_void_p()
        self.ended = self.rt.cudaStreamEndCapture(self.stream, ctypes.byref(graph))
        if graph.value:
            self.rt.cudaGraphDestroy(graph)
        self.rt.cudaStreamDestroy(self.stream)
        self.rt.cudaGetLastError()


def _addresses(h):
    p, s = ctypes.c_void_p(), ctypes.c_void_p()
    assert q.lib().qvggt_weights_view_c8(h.handle, ctypes.byref(p), None) == 0
    assert q.lib().qvggt_weights_view(h.handle, None, ctypes.byref(s), None, None, None, None) == 0
    return p.value, s.value


def test_memory_freed_without_a_synchronisation_is_not_handed_on():
    """While a stream is captured the device cannot be synchronised, so work that was queued before may still read a handle that is
    freed then: its memory must not become the next handle's.  (Global capture mode refuses cudaFree as well: the address cannot
    come back from the driver either.)"""
    W, b, c, ref, bias = _layer(1024, 640, 90)
    q.prepare_weights(W, b, c, None, c8="only").free()           # what is kept, freed in the ordinary way
    h = q.prepare_weights(W, b, c, None, c8="only")
    codes, scales = _addresses(h)
    torch.cuda.synchronize()
    with _Capture(0):
        h.free()
    others = [q.prepare_weights(W, b, c, None, c8="only") for _ in range(3)]
    for o in others:
        assert _addresses(o)[0] != codes and _addresses(o)[1] != scales
        _check(o, ref, bias, "only")
    for o in others:
        o.free()


@pytest.mark.parametrize("mode", [0, 1, 2], ids=["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("kept", [True, False])
def test_preparing_on_a_captured_stream_is_refused(mode, kept):
    """Whether or not kept memory would fit."""
    W, b, c, ref, bias = _layer(1024, 768, 91)
    first = q.prepare_weights(W, b, c, None, c8=True)
    if kept:
        first.free()
    torch.cuda.synchronize()
    with _Capture(mode) as cap, torch.cuda.stream(torch.cuda.ExternalStream(cap.stream.value)):
        with pytest.raises(q.QvggtError) as e:
            q.prepare_weights(W, b, c, None, c8=True)
        status = e.value.status
        del e
    assert status == -7 and cap.ended == 0
    h = q.prepare_weights(W, b, c, None, c8=True)
    _check(h, ref, bias, True)
    h.free()
    first.free()


_RESET = r"""
import ctypes, sys
import numpy as np
L, rt = ctypes.CDLL(sys.argv[1]), ctypes.CDLL("libcudart.so.12")
vp = ctypes.c_void_p
L.qvggt_prepare_weights.argtypes = [vp, vp, vp, vp, ctypes.c_int, ctypes.c_int, ctypes.c_int, vp, ctypes.POINTER(vp)]
L.qvggt_free_weights.argtypes = [vp]
L.qvggt_free_weights.restype = None
N, K = 128, 1024

def device(a):
    p = vp()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, a.ctypes.data_as(vp), ctypes.c_size_t(a.nbytes), 1) == 0
    return p

def prepare():
    W, c = device(np.full((N, K), 0x3F80, np.uint16)), device(np.ones(K, np.float32))
    h = vp()
    st = L.qvggt_prepare_weights(W, None, c, None, N, K, 1, None, ctypes.byref(h))
    print(st, rt.cudaDeviceSynchronize())
    return h

a, b = prepare(), prepare()
L.qvggt_free_weights(a)                  # its memory is kept
assert rt.cudaDeviceReset() == 0
c = prepare()                            # must not get that memory
L.qvggt_free_weights(b)                  # of the context that is gone
d = prepare()
"""


def test_kept_memory_is_not_used_after_a_device_reset():
    """In a process of its own.  Whatever the runtime answers to launches after a reset, no launch touches memory of the old context."""
    from paper_2509_21302_b200 import buildlib
    r = subprocess.run([sys.executable, "-c", _RESET, buildlib.LIB], capture_output=True, text=True, timeout=120, cwd=os.path.dirname(buildlib.LIB))
    assert r.returncode == 0, r.stdout + r.stderr
    lines = [tuple(int(v) for v in x.split()) for x in r.stdout.split("\n") if x]
    assert lines[:2] == [(0, 0)] * 2 and len(lines) == 4 and all(st in (0, -5) and sync == 0 for st, sync in lines[2:]), lines

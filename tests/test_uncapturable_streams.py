"""Calls of more steps than the longest step graph on streams on which no
capture can begin: the legacy default stream (handle 1), and a stream that the
caller is capturing; and step graphs built beside other threads' work."""
import numpy as np
import pytest

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, pytest.mark.auto_plan]

KEYS = ("u", "v", "P", "r")


def _prob(nx, ny, seed=5):
    return W.smooth_random(nx, ny, W.clamped_free_edges(), seed=seed, amp=0.01, lam=0.3, mu=0.3)


def _same(got, ref):
    for k in KEYS:
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("nx,ny", [(70, 60), (420, 400)])
@pytest.mark.parametrize("n", [66, 150])
def test_long_calls_on_the_legacy_stream(nx, ny, n):
    with lbm.Body(_prob(nx, ny), storage="f32", stream=1) as a, lbm.Body(_prob(nx, ny), storage="f32") as b:
        for k in (n, 3, n):
            a.step(k)
            b.step(k)
        _same(a.read(), b.read())


@pytest.mark.parametrize("nx,ny", [(70, 60), (420, 400)])
@pytest.mark.parametrize("before", [5, 200])
def test_long_calls_recorded_by_a_caller(nx, ny, before):
    """Recorded before (5 steps) and after (200) the body has graphs of its own."""
    import torch
    s = torch.cuda.Stream()
    with lbm.Body(_prob(nx, ny), storage="f32", stream=s.cuda_stream) as a, lbm.Body(_prob(nx, ny), storage="f32") as b:
        a.step(before)
        lbm.lbm_sync(a.ctx)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            a.step(150)
        with torch.cuda.stream(s):
            g.replay()
        s.synchronize()
        a.step(100)
        b.step(before + 250)
        _same(a.read(), b.read())


def test_building_graphs_leaves_other_threads_legacy_work_alone():
    """Bodies on a blocking stream build their step graphs while another thread
    launches on the legacy default stream."""
    import ctypes
    import threading

    import torch
    cuda = ctypes.CDLL("libcuda.so.1")
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    h = ctypes.c_void_p()
    assert cuda.cuStreamCreate(ctypes.byref(h), 0) == 0  # CU_STREAM_DEFAULT: blocking
    stop, running, errors, launches = threading.Event(), threading.Event(), [], [0]

    def work():
        x = torch.zeros(1000, device="cuda")
        try:
            while not stop.is_set():
                x.add_(1.0)
                launches[0] += 1
                running.set()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    try:
        assert running.wait(60)  # its kernel is loaded
        with lbm.Body(_prob(70, 60), storage="f32") as b:
            b.step(200)
            ref = b.read()
        for _ in range(20):
            with lbm.Body(_prob(70, 60), storage="f32", stream=h.value) as a:
                a.step(200)
                _same(a.read(), ref)
    finally:
        stop.set()
        t.join()
        assert cuda.cuStreamDestroy_v2(h) == 0
    assert not errors, errors
    assert launches[0] > 100


@pytest.mark.parametrize("mode", ["relaxed", "thread_local", "global"])
@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("n", [20, 200])
def test_building_graphs_inside_a_capture_of_another_stream(mode, own, n):
    """A body steps on its own stream (the library's or the caller's) while the
    thread captures another one: neither disturbs the other."""
    import torch
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(10, device="cuda")
    with lbm.Body(_prob(420, 400), storage="f32", stream=0 if own else t.cuda_stream) as a, \
            lbm.Body(_prob(420, 400), storage="f32") as b:
        a.step(5)  # the plan's allocations come before the capture
        lbm.lbm_sync(a.ctx)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode=mode):
            x.add_(1.0)
            a.step(n)
            x.add_(1.0)
        b.step(5 + n)
        _same(a.read(), b.read())
        with torch.cuda.stream(s):
            g.replay()
        s.synchronize()
        assert float(x[0]) == 2.0


@pytest.mark.parametrize("n", [66, 150])
def test_long_batch_calls_on_the_legacy_stream(n):
    probs = [_prob(200, 130, 1), _prob(131, 90, 2)]
    bodies = [lbm.Body(p, storage="f32", stream=1) for p in probs]
    others = [lbm.Body(p, storage="f32") for p in probs]
    try:
        with lbm.Batch(bodies, stream=1) as a, lbm.Batch(others) as b:
            for k in (n, 3, n):
                a.step(k)
                b.step(k)
            a.sync()
            b.sync()
        for x, y in zip(bodies, others):
            _same(x.read(), y.read())
    finally:
        for x in bodies + others:
            x.close()


@pytest.mark.parametrize("before", [6, 200])
def test_long_batch_calls_recorded_by_a_caller(before):
    import torch
    s = torch.cuda.Stream()
    probs = [_prob(200, 130, 1), _prob(131, 90, 2)]
    bodies = [lbm.Body(p, storage="f32", stream=s.cuda_stream) for p in probs]
    others = [lbm.Body(p, storage="f32") for p in probs]
    try:
        with lbm.Batch(bodies, stream=s.cuda_stream) as a, lbm.Batch(others) as b:
            a.step(before)
            a.sync()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
                a.step(150)
            with torch.cuda.stream(s):
                g.replay()
            s.synchronize()
            a.step(100)
            b.step(before + 250)
            a.sync()
            b.sync()
        for x, y in zip(bodies, others):
            _same(x.read(), y.read())
    finally:
        for x in bodies + others:
            x.close()

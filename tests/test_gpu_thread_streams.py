"""Calls on cudaStreamPerThread from two threads, one of them capturing: the
handle is the same, the streams are not, so the library's own second streams must
not be shared between them.  The eager call succeeds, the capture stays whole, and
both results equal those of a call on an ordinary stream."""
import ctypes
import threading

import pytest

import scenegen

pytestmark = pytest.mark.gpu


class PerThread:
    cuda_stream = 2  # cudaStreamPerThread


def _beside_a_capture(torch, captured, eager):
    """Runs eager() in one thread while another has captured() in a thread-local
    capture of its per-thread stream, then launches that graph."""
    cu = ctypes.CDLL("libcuda.so.1")
    st = ctypes.c_void_p(PerThread.cuda_stream)
    in_capture, eager_done = threading.Event(), threading.Event()
    errors = []

    def ok(status, what):
        if status != 0:
            raise RuntimeError(f"{what}: {status}")

    def capturing():
        graph, ex = ctypes.c_void_p(), ctypes.c_void_p()
        try:
            torch.zeros(1, device="cuda")  # the context is current in this thread
            captured()                     # every kernel loaded before the capture
            ok(cu.cuStreamSynchronize(st), "synchronize")
            ok(cu.cuStreamBeginCapture_v2(st, 1), "begin capture")
            try:
                captured()
            finally:
                in_capture.set()
                eager_done.wait(30)
                status = cu.cuStreamEndCapture(st, ctypes.byref(graph))
            ok(status, "end capture")
            ok(cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)), "instantiate")
            ok(cu.cuGraphLaunch(ex, st), "launch")
            ok(cu.cuStreamSynchronize(st), "synchronize")
            cu.cuGraphExecDestroy(ex)
            cu.cuGraphDestroy(graph)
        except Exception as e:  # noqa: BLE001 (reported by the caller)
            errors.append(e)
        finally:
            in_capture.set()

    def eager_call():
        try:
            torch.zeros(1, device="cuda")
            assert in_capture.wait(30)
            eager()
            ok(cu.cuStreamSynchronize(st), "synchronize")
        except Exception as e:  # noqa: BLE001
            errors.append(e)
        finally:
            eager_done.set()

    threads = [threading.Thread(target=f) for f in (capturing, eager_call)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(90)
    assert not errors, errors


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_10096_gb300 as sff
    sff.build()
    return torch, sff


def test_sift_features(env):
    torch, sff = env
    w, h = 161, 83
    p = sff.default_params()
    dev = [torch.as_tensor(im).cuda() for im in scenegen.make_quad("planes", w, h, 5).images()]
    outs = [[torch.full((4, h, w, 4), float("nan"), device="cuda") for _ in range(4)] for _ in range(3)]
    wss = [torch.empty(sff.sift_workspace_bytes(w, h), dtype=torch.uint8, device="cuda") for _ in range(3)]
    sff.sift_features(dev, outs[0], wss[0], p)
    torch.cuda.synchronize()
    calls = [lambda k=k: sff.sift_features(dev, outs[k], wss[k], p, stream=PerThread()) for k in (1, 2)]
    _beside_a_capture(torch, *calls)
    for o in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs[0], o))


def test_run_batch(env):
    torch, sff = env
    q = scenegen.make_quad("planes", 161, 83, 6)
    dev = [torch.as_tensor(im).cuda() for im in q.images()]
    ms = [sff.QuadMatcher(q.width, q.height) for _ in range(3)]
    for m in ms:
        m.seeds.zero_()
    ms[0].run(*dev, seed=3)
    torch.cuda.synchronize()
    _beside_a_capture(torch, *[lambda m=m: m.run(*dev, seed=3, stream=PerThread()) for m in ms[1:]])
    for m in ms[1:]:
        for what in ("fwd", "fwd_cost", "inv", "inv_cost", "keep", "cerr", "seeds", "count"):
            assert torch.equal(getattr(ms[0], what), getattr(m, what)), what

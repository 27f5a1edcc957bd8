"""Resident launches of several handles at once (GPU): side by side where their
tiles fit the SMs together, ordinary steps where they do not, and never behind
work of a stream that is not theirs."""

import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import paper_1908_08386_gb300 as L
from paper_1908_08386_gb300 import workloads as WL

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KW = dict(nu=0.03, alpha=0.05, gbeta=1e-4)


def make(nx, ny, seed, stream=None, **kw):
    with torch.cuda.stream(stream or torch.cuda.Stream()):
        c = L.Cavity(nx, ny, **dict(KW, **kw))
        u, v = WL.random_velocity(ny, nx, seed, 0.01)
        c.set_state(*[a.astype(np.float32) for a in (u, v, WL.random_temperature(ny, nx, seed + 1))])
    return c


# two that fit side by side, two that do not, an FP64 one beside another
@pytest.mark.parametrize("a,b", [((64, 64, "f32"), (64, 64, "f32")), ((300, 280, "f32"), (64, 64, "f32x2")),
                                 ((64, 64, "f64"), (64, 64, "f64"))])
def test_a_handle_does_not_wait_for_work_of_another_stream(a, b):
    s = torch.cuda.Stream()
    x, y = make(*a[:2], 3, s, store=a[2]), make(*b[:2], 4, store=b[2])
    ref = make(*b[:2], 4, store=b[2], kernel="tma")
    for c in (x, y, ref):  # every kernel loaded: a first use waits for an idle device
        c.step(60)
        c.step(9)
        c.residual()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(3_000_000_000)  # over a second
        slept = torch.cuda.Event()
        slept.record()
    x.step(50)
    for n in (60, 9):
        y.step(n)
        ref.step(n)
    r = y.residual()
    assert not slept.query()
    torch.cuda.synchronize()
    assert r == ref.residual()
    assert np.array_equal(np.stack(y.fields()), np.stack(ref.fields()))
    for c in (x, y, ref):
        c.close()


def test_handles_of_many_sizes_on_shared_and_own_streams():
    """Asynchronous steps of handles that come and go, on two shared streams and
    on streams of their own, from one thread and from several: each result is
    the one of a handle alone."""
    shapes = [(64, 64, "f32"), (150, 141, "f32"), (40, 40, "f64"), (64, 64, "f32x2"), (300, 280, "f16"), (90, 30, "f32"),
              (64, 64, "f64"), (120, 120, "f32x2")]
    want = []
    for i, (nx, ny, st) in enumerate(shapes):
        ref = make(nx, ny, i, store=st, kernel="tma")
        ref.step(400)
        want.append(np.stack(ref.fields()))
        ref.close()
    shared = [torch.cuda.Stream() for _ in range(2)]

    def run(which, streams):
        for _ in range(3):
            cs = [(i, make(*shapes[i][:2], i, streams[k % len(streams)] if streams else None, store=shapes[i][2]))
                  for k, i in enumerate(which)]
            for n in (100, 8, 92, 200):
                for _, c in cs:
                    c.step(n)
            for i, c in cs:
                bad = not np.array_equal(np.stack(c.fields()), want[i])
                c.close()
                if bad:
                    wrong.append(i)

    wrong = []
    run(range(8), shared)
    run(range(8), shared[:1])
    run(range(8), None)
    ts = [threading.Thread(target=run, args=(w, st)) for w, st in
          ((range(0, 4), shared), (range(4, 8), shared), (range(8), None), (range(7, -1, -1), None))]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not wrong


def test_steps_beside_another_threads_capture():
    """A stream capture of another thread in its strictest mode outlives a call
    that looks for launches in flight."""
    a, b = make(64, 64, 1), make(64, 64, 2)
    torch.cuda.synchronize()
    g, x = torch.cuda.CUDAGraph(), torch.ones(1000, device="cuda")
    y = x * 2
    torch.cuda.synchronize()
    inside, stepped = threading.Event(), threading.Event()

    def go():
        inside.wait()
        for _ in range(20):
            a.step(10)
            b.step(10)
        stepped.set()

    t = threading.Thread(target=go)
    t.start()
    with torch.cuda.graph(g, capture_error_mode="global"):
        inside.set()
        assert stepped.wait(60)
        y = x * 3
    t.join()
    g.replay()
    torch.cuda.synchronize()
    assert float(y[0]) == 3.0 and a.steps == b.steps == 200
    a.close()
    b.close()


RESET = """
import ctypes
import paper_1908_08386_gb300 as L
rt = ctypes.CDLL("libcudart.so.13")
def residual():
    h = L.lbmfvm_create_lattice(L.make_grid(64, 64), None, 0.03, 0.05, 1e-4)
    L.lbmfvm_step(h, 50)
    r = L.lbmfvm_residual(h)
    L.lbmfvm_destroy(h)
    return r
first = residual()
assert rt.cudaDeviceReset() == 0
assert residual() == first
print("same")
"""


def test_new_handles_after_a_device_reset():
    """A program that closes its handles, resets its context and starts anew."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LD_LIBRARY_PATH="/usr/local/cuda/lib64:" + os.environ.get("LD_LIBRARY_PATH", ""))
    r = subprocess.run([sys.executable, "-c", RESET], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    if "libcudart" in r.stderr:
        pytest.skip("no shared CUDA runtime to call cudaDeviceReset of")
    assert r.stdout.strip() == "same", r.stderr

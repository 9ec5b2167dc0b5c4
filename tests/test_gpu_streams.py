"""FP64 sweeps of several meshes at once, each on its own stream and thread: the
results of each alone, and for small lattices room for one another on the GPU."""
import threading
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

SHAPES = {
    "small": (dict(n=(33, 30, 28), fem=((8, 8, 8), (24, 22, 20)), nsteps=120), 1),
    "refined": (dict(n=(24, 26, 31), fem=((5, 5, 5), (18, 20, 25)), nsteps=80, refine_frac=0.3), 2),
    "resident": (dict(n=(70, 66, 65), fem=((9, 6, 8), (51, 31, 33)), nsteps=60), 2),
    "per_axis": (dict(n=(41, 38, 45), fem=((4, 4, 4), (30, 30, 30)), nsteps=80, spacing=(0.03, 0.045, 0.038)), 1),
}


@pytest.fixture(scope="module")
def H():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb
    return hyb


def at_once(calls):
    """Runs the calls on a stream and a thread each; their results."""
    import torch
    out, bar = [None] * len(calls), threading.Barrier(len(calls))

    def go(q):
        with torch.cuda.stream(torch.cuda.Stream()):
            out[q] = calls[q](bar.wait)
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=go, args=(q,)) for q in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return out


@pytest.mark.parametrize("partner", sorted(SHAPES))
def test_two_meshes_on_two_streams(H, partner):
    import torch

    def solve(shape, nsrc):
        def call(ready, rounds=4):
            w = synth.small_problem(omega=14.0, courant=0.8, **shape)
            srcs = [synth.Source(synth.FACE_XP, 14.0), synth.Source(synth.FACE_ZM, 14.0, 1.0, (1.0, 2.0, 3.0))][:nsrc]
            a = torch.as_tensor(1.0 + np.random.default_rng(3).random(w.n_unknown), device="cuda")
            m = H.HybMesh.from_workload(w, precision="fp64")
            cot = torch.randn(m.new_trace(nsrc, w.nsteps).shape, device="cuda", dtype=torch.float64,
                              generator=torch.Generator(device="cuda").manual_seed(4))
            torch.cuda.current_stream().synchronize()
            ready()
            for _ in range(rounds):
                tr = m.forward(a, srcs, w.nsteps, w.dt)
                m.adjoint(cot)
                g = m.gradient(a, 0.0, 1.0)
            m.sync()
            m.close()
            return tr, g
        return call

    calls = [solve(*SHAPES["small"]), solve(*SHAPES[partner])]
    alone = [c(lambda: None, 1) for c in calls]
    for got, want in zip(at_once(calls), alone):
        assert torch.equal(got[0], want[0])
        # (a refined region's gradient terms are added in no fixed order)
        assert float((got[1] - want[1]).norm() / want[1].norm()) <= 1e-13


def test_small_sweeps_share_the_gpu(H):
    """Three small sweeps at once take less than twice the time of one: a sweep that
    held every SM would run them one after the other."""
    import torch
    w = synth.small_problem(n=(33, 33, 33), fem=((8, 8, 8), (24, 24, 24)), nsteps=3000, omega=14.0, courant=0.8)
    a = torch.full((w.n_unknown,), 1.5, device="cuda", dtype=torch.float64)

    def sweep(ready):
        m = H.HybMesh.from_workload(w, precision="fp64", ckpt_every=100)
        tr = m.new_trace(1, w.nsteps)
        for _ in range(3):  # (the first calls allocate and capture)
            m.forward(a, w.sources, w.nsteps, w.dt, trace=tr)
        m.sync()
        ready()
        t0 = time.perf_counter()
        for _ in range(4):
            m.forward(a, w.sources, w.nsteps, w.dt, trace=tr)
        m.sync()
        t1 = time.perf_counter()
        m.close()
        return t1 - t0

    one = min(at_once([sweep])[0] for _ in range(2))
    three = min(max(at_once([sweep] * 3)) for _ in range(2))
    print("one sweep %.2f ms, three at once %.2f ms" % (one * 1e3, three * 1e3))
    assert three < 2.0 * one


def test_small_pass_beside_an_fp64_inversion(H):
    """A short FP32 gradient beside an FP64 inversion that fills the GPU takes less than
    half of the inversion's time: the sweep's launches end often enough for it."""
    import torch

    def gradient(w, m, a, cot):
        m.forward(a, w.sources, w.nsteps, w.dt)
        m.adjoint(cot)
        m.sync()

    def ready(n, precision, nsteps):
        w = synth.small_problem(n=n, fem=(tuple(v // 4 for v in n), tuple(3 * v // 4 for v in n)), nsteps=nsteps,
                                omega=14.0, courant=0.8)
        m = H.HybMesh.from_workload(w, precision=precision)
        args = w, m, torch.full((w.n_unknown,), 1.5, device="cuda", dtype=torch.float64), m.new_trace(1, nsteps)
        for _ in range(3):  # (the first calls allocate and capture)
            gradient(*args)
        return args

    def timed(args):
        t0 = time.perf_counter()
        gradient(*args)
        return time.perf_counter() - t0

    big, small = [], []
    loaded, done = threading.Event(), threading.Event()

    def inversion():
        with torch.cuda.stream(torch.cuda.Stream()):
            args = ready((65, 65, 65), "fp64", 2000)
            big.append(min(timed(args) for _ in range(3)))
            loaded.set()
            while not done.is_set():
                gradient(*args)
            args[1].close()

    with torch.cuda.stream(torch.cuda.Stream()):
        args = ready((33, 33, 33), "fp32", 100)
        t = threading.Thread(target=inversion)
        t.start()
        try:
            assert loaded.wait(60)
            time.sleep(0.05)
            small = sorted(timed(args) for _ in range(7))
        finally:
            done.set()
            t.join()
        args[1].close()
    print("inversion alone %.1f ms, small pass beside it %.1f ms" % (big[0] * 1e3, small[3] * 1e3))
    assert small[3] < 0.5 * big[0]

"""Batches whose interior items are cut to leave room for the edge tiles' blocks
(eight of 65^3), for one wave (six of 70 x 81 x 62) and as one source's (two of
33^3), on a mesh that also runs several sources of one coefficient: every
problem's trace and gradient are those it has alone."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [((65, 65, 65), 8), ((70, 81, 62), 6), ((33, 33, 33), 2)])
def test_batch_matches_each_alone(n, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb as H
    w = synth.small_problem(n=n, fem=(tuple(v // 4 for v in n), tuple(3 * v // 4 for v in n)), nsteps=60, omega=25.0,
                            courant=0.8)
    a = torch.as_tensor(1.0 + np.random.default_rng(6).random((k, w.n_unknown)), device="cuda")
    srcs = [synth.Source(q % 6, 25.0) for q in range(k)]
    m = H.HybMesh.from_workload(w, precision="fp32")
    cot = torch.randn(m.new_trace(k, w.nsteps).shape, device="cuda",
                      generator=torch.Generator(device="cuda").manual_seed(2))
    m.forward(a[0], srcs, w.nsteps, w.dt)  # (the sources of one coefficient: a cut of their own)
    m.adjoint(cot)
    for _ in range(3):  # the last pass replays the captured sweeps
        trace = m.new_trace(k, w.nsteps)
        H.hyb_forward_batch(m.handle, a.data_ptr(), srcs, w.nsteps, w.dt, trace.data_ptr())
        H.hyb_adjoint(m.handle, cot.data_ptr(), 0)
        g = torch.empty_like(a)
        H.hyb_gradient_batch(m.handle, a.data_ptr(), 0.0, 1.0, g.data_ptr())
    m.sync()
    one = H.HybMesh.from_workload(w, precision="fp32")
    for q in range(k):
        tr = one.forward(a[q], srcs[q:q + 1], w.nsteps, w.dt)
        one.adjoint(cot[q:q + 1])
        assert torch.equal(tr[0], trace[q]), q
        assert torch.equal(one.gradient(a[q], 0.0, 1.0), g[q]), q
    one.close()
    m.close()

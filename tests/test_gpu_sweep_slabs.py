"""The sweep kernel (FP64 fields) with slabs of several planes, where a march
carries values from plane to plane, and with sweeps cut into several launches:
sixteen sources of one lattice.  Slabs of three planes (the last one partial)
against the FP64 oracle at the parity tests' 1e-12; slabs of sixteen and two
launches a sweep against each source alone, whose sweep takes one launch of
slabs of one plane or two: the rows' arithmetic is the same."""
import numpy as np
import pytest

import oracle
import synth
from helpers import rel_l2

pytestmark = pytest.mark.gpu

SLOTS = 16


@pytest.fixture(scope="module")
def H():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb
    return hyb


KINDS = {
    "plain": (dict(bc=(1, 1, 0, 1, 1, 1)), {}),
    "refined": (dict(refine_frac=0.1), {}),
    "telegraph": ({}, dict(model=1)),
    "per_axis": (dict(spacing=(0.03, 0.045, 0.038), bc=(1, 0, 1, 1, 1, 0)), {}),
    "paper": ({}, dict(adjoint_mode=1)),
}
SOURCES = [synth.Source(synth.FACE_XP, 40.0), synth.Source(synth.FACE_ZM, 40.0, 1.0, (1.0, 2.0, 3.0))]


@pytest.mark.parametrize("kind", ["plain", "refined", "per_axis", "paper"])
def test_three_planes_a_slab(H, kind):
    import torch
    shape, kw = KINDS[kind]
    w = synth.small_problem(n=(62, 60, 60), fem=((3, 3, 4), (57, 56, 54)), nsteps=30, courant=0.8, **shape)
    a = 1.0 + np.random.default_rng(2).random(w.n_unknown)
    P = oracle.problem_from_workload(w)
    want_tr, want_g, cots = [], 0.0, []
    for q, src in enumerate(SOURCES):
        r = P.forward(a, src, w.nsteps, w.dt, keep_hist=True)
        c = synth.random_cotangent(1, w.nsteps, r["trace"].shape[1], seed=70 + q)[0]
        adj = P.adjoint_paper if kind == "paper" else P.adjoint
        want_g = want_g + SLOTS // 2 * adj(a, src, w.nsteps, w.dt, c, r["hist"])
        want_tr.append(r["trace"])
        cots.append(torch.from_numpy(c))
    for ckpt in (0, 8):
        m = H.HybMesh.from_workload(w, precision="fp64", ckpt_every=ckpt, **kw)
        tr = m.forward(a, SOURCES * (SLOTS // 2), w.nsteps, w.dt)
        cot = torch.zeros_like(tr)
        for s in range(SLOTS):
            t = want_tr[s % 2]
            assert rel_l2(tr[s, :, : t.shape[1]].cpu().numpy(), t) <= 1e-12, (ckpt, s)
            cot[s, :, : t.shape[1]] = cots[s % 2]
        m.adjoint(cot)
        assert rel_l2(m.gradient(a, 0.0, 1.0).cpu().numpy(), want_g) <= 1e-12, ckpt
        m.sync()
        m.close()


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_sixteen_planes_a_slab_and_two_launches(H, kind):
    import torch
    shape, kw = KINDS[kind]
    w = synth.small_problem(n=(112, 105, 104), fem=((10, 9, 8), (40, 38, 44)), nsteps=280, courant=0.8, **shape)
    srcs = [synth.Source(q % 6, 30.0 + q) for q in range(SLOTS)]
    a = (0.0 if kind == "telegraph" else 1.0) + np.random.default_rng(8).random(w.n_unknown)
    m = H.HybMesh.from_workload(w, precision="fp64", **kw)
    one = H.HybMesh.from_workload(w, precision="fp64", **kw)
    tr = m.forward(a, srcs, w.nsteps, w.dt)
    cot = torch.randn(tr.shape, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(1))
    m.adjoint(cot)
    g, want = m.gradient(a, 0.0, 1.0), 0.0
    for s in range(SLOTS):
        t = one.forward(a, srcs[s:s + 1], w.nsteps, w.dt)
        assert torch.equal(t[0], tr[s]), s
        one.adjoint(cot[s:s + 1])
        want = want + one.gradient(a, 0.0, 1.0)
    m.sync()
    # the sixteen gradients summed in another order
    assert float((g - want).norm() / want.norm()) <= 1e-14 * SLOTS
    m.close()
    one.close()

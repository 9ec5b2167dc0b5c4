"""The paper's adjoint in FP32, whose step launches carry the same-index pairing
in their trailing blocks: one voxel block and several, refined voxels behind
them, one and three slots, stored and recomputed history, against the FP64
oracle."""
import numpy as np
import pytest

import oracle
import synth
from helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb
    return hyb


SHAPES = {
    "one_block": dict(n=(9, 10, 11), fem=((3, 3, 3), (6, 6, 6)), nsteps=40),
    "several_blocks": dict(n=(37, 21, 19), fem=((5, 4, 4), (30, 16, 15)), nsteps=40),
    "refined": dict(n=(12, 11, 13), fem=((2, 2, 2), (9, 8, 10)), nsteps=40, refine_frac=0.5, bc=(0, 1, 0, 1, 1, 1)),
}


@pytest.mark.parametrize("ckpt", [0, 7])
@pytest.mark.parametrize("n_src", [1, 3])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_fp32_paper_gradient(H, name, n_src, ckpt):
    import torch
    w = synth.small_problem(omega=12.0, courant=0.8, **SHAPES[name])
    srcs = [synth.Source(synth.FACE_ZP, 12.0), synth.Source(synth.FACE_XM, 9.0),
            synth.Source(synth.FACE_ZM, 14.0, 1.0, (1.0, 1.0, 1.0))][:n_src]
    a = 1.0 + 2.0 * np.random.default_rng(5).random(w.n_unknown)
    m = H.HybMesh.from_workload(w, precision="fp32", ckpt_every=ckpt, adjoint_mode=H.HYB_ADJ_PAPER)
    tr = m.forward(a, srcs, w.nsteps, w.dt)
    P = oracle.problem_from_workload(w)
    cot, want = torch.zeros_like(tr), 0.0
    for s, src in enumerate(srcs):
        r = P.forward(a, src, w.nsteps, w.dt, keep_hist=True)
        c = synth.random_cotangent(1, w.nsteps, r["trace"].shape[1], seed=60 + s)[0]
        cot[s, :, : c.shape[1]] = torch.from_numpy(c)
        want = want + P.adjoint_paper(a, src, w.nsteps, w.dt, c, r["hist"])
    m.adjoint(cot)
    # FP32 rounding of 40 steps and of the cotangent, at the parity tests' FP32 tolerance
    assert rel_l2(m.gradient(a, 0.0, 1.0).cpu().numpy(), want) <= 1e-4
    m.close()

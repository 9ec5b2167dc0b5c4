"""Where the paper's adjoint in FP32 pairs: inside the step's launch with a small
FEM block, by launches of its own with a large one (which the step's blocks
would hold up), on both sides of the line, and the gradient there against the
FP64 fields'."""
import numpy as np
import pytest

import synth
from helpers import rel_l2

pytestmark = pytest.mark.gpu

SHAPES = {  # (kernels per adjoint level: the step, and the pairing's own)
    "small_block": (dict(n=(60, 41, 50), fem=((2, 2, 2), (57, 38, 47))), 1),
    "large_block": (dict(n=(121, 112, 108), fem=((2, 2, 2), (118, 109, 105))), 2),
    "many_refined": (dict(n=(44, 41, 42), fem=((4, 4, 4), (39, 36, 37)), refine_frac=0.6), 3),
    "few_refined": (dict(n=(44, 41, 42), fem=((4, 4, 4), (39, 36, 37)), refine_frac=0.05), 1),
}


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_pairing_place(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb as H
    shape, per_level = SHAPES[name]
    w = synth.small_problem(omega=25.0, courant=0.8, nsteps=60, **shape)
    a = 1.0 + 2.0 * np.random.default_rng(9).random(w.n_unknown)
    got, cot = {}, None
    for precision in ("fp64", "fp32"):
        m = H.HybMesh.from_workload(w, precision=precision, adjoint_mode=H.HYB_ADJ_PAPER)
        tr = m.forward(a, w.sources, w.nsteps, w.dt)
        if cot is None:
            cot = torch.randn(tr.shape, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda",
                              dtype=torch.float64).float()
        before = m.launches()
        m.adjoint(cot)
        if precision == "fp32":  # levels 59 .. 1 pair; the first level does not, and level 0 pairs last
            level0 = 2 if shape.get("refine_frac") else 1
            assert m.launches() - before == 1 + 59 * per_level + level0
        got[precision] = m.gradient(a, 0.0, 1.0).cpu().numpy()
        m.close()
    # FP32 rounding of 60 forward and 60 adjoint levels, at the parity tests' FP32 tolerance
    assert rel_l2(got["fp32"], got["fp64"]) <= 1e-4

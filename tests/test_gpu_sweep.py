"""The sweep kernel (FP64 fields) and the tile kernel with per-axis steps (FP32)
where their pieces meet:
lattices down to 5 nodes, x extents at every remainder of the 16-byte groups,
rows longer than an item's run (staged in three pieces), items that end inside
a row, slabs of several planes and several launches' worth of levels, with FEM
blocks that touch the faces' neighbours, reflecting and absorbing faces, against
the FP64 oracle at 1e-12 (the parity tests' FP64 tolerance) and, per-axis steps
in FP32, at the FP32 tolerances."""
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
    "least_5": dict(n=(5, 5, 5), fem=((0, 0, 0), (4, 4, 4)), bc=(1, 1, 1, 1, 1, 1)),
    "thin_5x9x6": dict(n=(5, 9, 6), fem=((1, 2, 1), (3, 6, 4)), bc=(0, 1, 1, 0, 1, 1)),
    "x_rem0_16": dict(n=(16, 7, 9), fem=((1, 1, 2), (14, 5, 6)), bc=(1, 0, 1, 1, 1, 0)),
    "x_rem1_17": dict(n=(17, 8, 6), fem=((0, 1, 0), (16, 6, 5)), bc=(1, 1, 0, 1, 1, 1)),
    "x_rem2_18": dict(n=(18, 6, 8), fem=((3, 1, 2), (12, 4, 6)), bc=(1, 1, 1, 1, 0, 1)),
    "x_rem3_19": dict(n=(19, 9, 7), fem=((2, 2, 1), (17, 7, 5)), bc=(0, 0, 1, 1, 1, 1)),
    "long_rows_1100": dict(n=(1100, 6, 7), fem=((530, 1, 2), (560, 4, 5)), bc=(1, 1, 1, 1, 1, 1)),
    "slabs_70x38x41": dict(n=(70, 38, 41), fem=((9, 6, 8), (51, 31, 33)), bc=(1, 1, 1, 0, 1, 1)),
}
SPACING = (0.03, 0.045, 0.038)


@pytest.mark.parametrize("steps", ["equal", "per_axis", "per_axis_fp32"])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_sweep_matches_the_oracle(H, name, steps):
    """Traces of three sources, and the gradient of a seeded random cotangent
    on them (no residual, whose cancellation would hide or mimic errors)."""
    import torch
    w = synth.small_problem(nsteps=60, omega=14.0, courant=0.8, spacing=None if steps == "equal" else SPACING,
                            **SHAPES[name])
    srcs = [synth.Source(synth.FACE_XP, 14.0), synth.Source(synth.FACE_ZM, 14.0, 1.0, (1.0, 2.0, 3.0)),
            synth.Source(synth.FACE_YM, 11.0)]
    a = 1.0 + 2.0 * np.random.default_rng(31).random(w.n_unknown)
    fp32 = steps.endswith("fp32")
    m = H.HybMesh.from_workload(w, precision="fp32" if fp32 else "fp64")
    tr = m.forward(a, srcs, w.nsteps, w.dt)
    P = oracle.problem_from_workload(w)
    cot, g = torch.zeros_like(tr), 0.0
    for s, src in enumerate(srcs):
        r = P.forward(a, src, w.nsteps, w.dt, keep_hist=True)
        assert rel_l2(tr[s, :, : r["trace"].shape[1]].double().cpu().numpy(), r["trace"]) <= (1e-4 if fp32 else 1e-12), s
        c = synth.random_cotangent(1, w.nsteps, r["trace"].shape[1], seed=40 + s)[0]
        cot[s, :, : c.shape[1]] = torch.from_numpy(c)
        g = g + P.adjoint(a, src, w.nsteps, w.dt, c, r["hist"])
    m.adjoint(cot)
    got = m.gradient(a, 0.0, 1.0).cpu().numpy()
    m.sync()
    m.close()
    assert rel_l2(got, g) <= (1e-3 if fp32 else 1e-12)

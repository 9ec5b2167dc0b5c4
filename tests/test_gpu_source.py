"""The plane-wave flux of FP32 fields, whose delay is formed in pairs of FP32
numbers: waves through one, two and three faces, with the pulse's start and end
on the lattice, per-axis steps too, against the FP64 fields' traces on the source
face."""
import pytest

import synth

pytestmark = pytest.mark.gpu

WAVES = {
    "x": (synth.FACE_XM, None), "y": (synth.FACE_YP, None), "z": (synth.FACE_ZP, None),
    "two_faces": (synth.FACE_XP, (-1.0, 0.4, 0.0)), "three_faces": (synth.FACE_ZM, (0.3, -0.5, 0.8)),
}


@pytest.mark.parametrize("spacing", [None, (0.03, 0.045, 0.038)])
@pytest.mark.parametrize("wave", sorted(WAVES))
def test_fp32_flux_follows_fp64(wave, spacing):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb
    face, direction = WAVES[wave]
    w = synth.small_problem(n=(37, 21, 40), fem=None, nsteps=60, omega=14.0, courant=0.8, spacing=spacing)
    src = synth.Source(face, 14.0) if direction is None else synth.Source(face, 14.0, 1.0, direction)
    out = []
    for precision in ("fp32", "fp64"):
        m = hyb.HybMesh.from_workload(w, precision=precision)
        out.append(m.forward(torch.zeros(0, dtype=torch.float64), [src], w.nsteps, w.dt).double())
        m.close()
    # 60 levels of FP32 rounding (2^-24 each) on the rows; the flux adds one rounding of its argument a level
    assert float((out[0] - out[1]).norm() / out[1].norm()) <= 1e-5

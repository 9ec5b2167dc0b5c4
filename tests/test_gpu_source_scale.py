"""The plane-wave flux of FP32 fields in other units of length and time (with
omega and the pulse's end beyond FP32's range among them): the scheme knows only
ratios, so the trace is that of unit 1."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [1e-40, 1e-32, 1e-15, 1e20, 1e40])
def test_fp32_flux_in_other_units(unit):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb
    out = []
    for precision, u in (("fp32", unit), ("fp64", 1.0)):
        m = hyb.HybMesh((37, 21, 40), 0.03 * u, precision=precision, a_max=2.0)
        src = synth.Source(synth.FACE_ZM, 14.0 / u, 1.0 / u, (0.3, -0.5, 0.8))
        out.append(m.forward(torch.zeros(0, dtype=torch.float64), [src], 60, 0.8 * m.info.dt_max).double())
        m.close()
    # 60 levels of FP32 rounding (2^-24 each) on the rows; the flux adds one rounding of its argument a level
    assert float((out[0] - out[1]).norm() / out[1].norm()) <= 1e-5

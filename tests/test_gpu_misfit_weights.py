"""FP32 cotangents of the misfit where the weight tau h^2 is far from 1: beyond
FP32's range with equal entries among the data, and so small that its FP32
parts would be rounded; one rounding of the FP64 product each."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,scale", [(1e20, 1e-25), (2e10, 1e-3), (1.0, 1.0), (3e-11, 1e5), (2e-12, 1e20),
                                     (5e-14, 1e29), (1e-18, 1e30)])
def test_cotangent_of_extreme_weights(h, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb as H
    n, nsteps, dt = (33, 20, 9), 4, 0.1 * h
    m = H.HybMesh(n, h, None, None, (1,) * 6, "fp32", 0, 2.0)
    m.forward(torch.zeros(0, dtype=torch.float64, device="cuda"), [synth.Source(5, 1.0 / h)], nsteps, dt)
    gen = torch.Generator(device="cuda").manual_seed(8)
    tr = scale * torch.randn((1, nsteps + 1, m.obs_stride), generator=gen, device="cuda")
    obs = scale * torch.randn(tr.shape, generator=gen, device="cuda")
    obs[:, :, ::5] = tr[:, :, ::5]
    J, cot = m.misfit(tr, obs, 1, want_cot=True)
    w = np.full((n[1], n[0]), dt * (h * h))
    w[0] *= 0.5
    w[-1] *= 0.5
    w[:, 0] *= 0.5
    w[:, -1] *= 0.5
    w = w.ravel()
    r = (tr.double() - obs.double()).cpu().numpy()[0, 1:, : w.size]
    # sums of FP64 products in another order; one rounding to FP32, relative, and below its normal range absolute
    assert abs(J - 0.5 * float((w * r * r).sum())) <= 1e-12 * J
    np.testing.assert_allclose(cot.double().cpu().numpy()[0, 1:, : w.size], w * r, rtol=6e-8, atol=1e-45)
    m.close()

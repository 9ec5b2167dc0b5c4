"""The misfit reduction's blocks of columns and rows: traces whose rows end
inside and past a block of 512 columns, one step, several sources with
faces of different extents, both weights, against the same sums in numpy."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb
    return hyb


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("weights", [0, 1])
@pytest.mark.parametrize("n,nsteps", [((3, 4, 5), 1), ((32, 16, 9), 7), ((27, 19, 6), 3), ((33, 31, 70), 40)])
def test_misfit_and_cotangent(H, n, nsteps, weights, precision):
    import torch
    h, dt = 0.1, 0.01
    m = H.HybMesh(n, h, None, None, (1,) * 6, precision, 0, 2.0)
    srcs = [synth.Source(f, 12.0) for f in (5, 0, 3)]
    a = torch.zeros(0, dtype=torch.float64, device="cuda")
    m.forward(a, srcs, nsteps, dt)
    gen = torch.Generator(device="cuda").manual_seed(3)
    tr = torch.randn((3, nsteps + 1, m.obs_stride), generator=gen, device="cuda", dtype=torch.float64).to(m.dtype)
    obs = torch.randn(tr.shape, generator=gen, device="cuda", dtype=torch.float64).to(m.dtype)
    J, cot = m.misfit(tr, obs, weights, want_cot=True)
    want_cot, want_J = np.zeros(tr.shape), 0.0
    for s, src in enumerate(srcs):
        p, q = [n[d] for d in range(3) if d != src.face // 2]
        w = np.ones((q, p))
        if weights:
            w *= dt * h * h
            w[0] *= 0.5
            w[-1] *= 0.5
            w[:, 0] *= 0.5
            w[:, -1] *= 0.5
        w = w.ravel()
        r = (tr[s].double() - obs[s].double()).cpu().numpy()[1:, : p * q]
        want_cot[s, 1:, : p * q] = w * r
        want_J += 0.5 * float((w * r * r).sum())
    # J: sums of FP64 products in another order; the cotangent: one rounding to the field's precision
    assert abs(J - want_J) <= 1e-12 * want_J
    tol = 1e-15 if precision == "fp64" else 6e-8
    np.testing.assert_allclose(cot.double().cpu().numpy(), want_cot, rtol=tol, atol=0)
    m.close()


def test_cg_step_with_more_partials_than_the_reductions(H):
    """Two faces of 1025^2 entries: the misfit wants a larger buffer of partial
    sums than the other reductions of a CG step, in the middle of the step.
    The report against the same step's gradient in separate calls."""
    import torch
    n, h, nsteps, dt, gamma = (1025, 1025, 9), 0.1, 48, 0.025, 0.01
    m = H.HybMesh(n, h, (2, 2, 2), (6, 6, 6), (1,) * 6, "fp64", 0, 4.0)
    srcs = [synth.Source(f, 12.0) for f in (4, 5)]
    gen = torch.Generator(device="cuda").manual_seed(4)
    a = 1.0 + torch.rand(m.n_unknown, generator=gen, device="cuda", dtype=torch.float64)
    obs = torch.randn((2, nsteps + 1, m.obs_stride), generator=gen, device="cuda", dtype=torch.float64)
    # the step first: its misfit has to grow the buffer itself
    step = a.clone()
    rep = m.cg_step(step, obs, srcs, nsteps, dt, m.new_cg_state(), gamma=gamma, a0=1.0, a_min=1.0, a_max=4.0)
    tr = m.forward(a, srcs, nsteps, dt)
    J, cot = m.misfit(tr, obs, 1, want_cot=True)
    m.adjoint(cot)
    g = m.gradient(a, gamma=gamma, a0=1.0)
    vol = h ** 3
    want_J = J + 0.5 * gamma * vol * float(((a - 1.0) ** 2).sum())
    want_g = float((g @ g) / vol) ** 0.5
    # the same arithmetic, sums in another order
    assert abs(rep.J - want_J) <= 1e-12 * want_J
    assert abs(rep.gnorm - want_g) <= 1e-12 * want_g
    m.close()

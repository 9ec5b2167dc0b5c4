"""Tall lattices driven at their top: FP32 fields of 2^31 padded nodes and more,
whose node offsets no longer fit 32 bits, and FP64 fields of 2^23 planes and
more, against the same problem with FP64 fields on a short lattice with the same
top (a wave moves at most one node a step, so neither sees its bottom)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

STEPS = 30
KINDS = {
    "plain": {},
    "refined": dict(refine=True),
    "telegraph": dict(model=1),
    "per_axis": dict(spacing=(0.03, 0.045, 0.038)),
    "paper": dict(adjoint_mode=1),
}


def solve(H, precision, nx, ny, nz, kind):
    """Trace on the top face and gradient, with the FEM block 24 to 5 planes
    below the top of the lattice."""
    import torch
    kw = dict(KINDS[kind])
    lo = (nx // 4, ny // 4, nz - 24)
    hi = (nx - 1 - nx // 4, ny - 1 - ny // 4, nz - 5)
    ud = synth.unknown_dims(lo, hi)
    rng = np.random.default_rng(7)
    a = 1.0 + rng.random(ud[0] * ud[1] * ud[2])
    if kind == "telegraph":
        a -= 1.0
    refine = (rng.random(a.size) < 0.2) if kw.pop("refine", False) else None
    m = H.HybMesh((nx, ny, nz), 0.03, lo, hi, (1,) * 6, precision, 0, 2.0, refine=refine, **kw)
    dt = 0.5 * m.info.dt_max
    srcs = [synth.Source(synth.FACE_ZP, 20.0)]
    tr = m.forward(a, srcs, STEPS, dt)
    cot = torch.zeros_like(tr)
    c = torch.randn((STEPS + 1, nx * ny), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda",
                    dtype=torch.float64)
    cot[0, :, : nx * ny] = c.to(cot.dtype)
    m.adjoint(cot)
    g = m.gradient(a, 0.0, 1.0)
    m.sync()
    out = tr[0, :, : nx * ny].clone(), g
    m.close()
    del tr, cot
    torch.cuda.empty_cache()
    return out


def pair(precision, nx, ny, nz, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb as H
    tall, short = solve(H, precision, nx, ny, nz, kind), solve(H, "fp64", nx, ny, 72, kind)
    # the parity tests' tolerances of the precision
    for got, want, tol in zip(tall, short, (1e-4, 1e-3) if precision == "fp32" else (1e-12, 1e-12)):
        assert float((got.double() - want).norm() / want.norm()) <= tol


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_fp32_tall(kind):
    pair("fp32", 72, 66, (1 << 31) // (72 * 66) + 150, kind)


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_fp64_tall(kind):
    pair("fp64", 8, 8, (1 << 23) + 40, kind)

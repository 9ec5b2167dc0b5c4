"""Fields of 2^31 padded nodes and more: a tall lattice driven at its top, where
the node offsets no longer fit 32 bits, against the same problem with FP64 fields
on a short lattice with the same top (a wave moves at most one node a step, so
neither sees its bottom)."""
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


def solve(H, precision, nx, ny, nz, top, kind):
    """Trace on the top face and gradient, with the FEM block 24 planes to 4
    planes below the top of the lattice (top) or above its bottom."""
    import torch
    kw = dict(KINDS[kind])
    lo = (20, 18, nz - 24 if top else 4)
    hi = (nx - 21, ny - 19, nz - 5 if top else 23)
    ud = synth.unknown_dims(lo, hi)
    rng = np.random.default_rng(7)
    a = 1.0 + rng.random(ud[0] * ud[1] * ud[2])
    if kind == "telegraph":
        a -= 1.0
    refine = (rng.random(a.size) < 0.2) if kw.pop("refine", False) else None
    m = H.HybMesh((nx, ny, nz), 0.03, lo, hi, (1,) * 6, precision, 0, 2.0, refine=refine, **kw)
    dt = 0.5 * m.info.dt_max
    srcs = [synth.Source(synth.FACE_ZP if top else synth.FACE_ZM, 20.0)]
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


def pair(precision, nx, ny, nz, top, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_01399_gb300 import hyb as H
    tall, short = solve(H, precision, nx, ny, nz, top, kind), solve(H, "fp64", nx, ny, 72, top, kind)
    # the parity tests' tolerances of the precision
    for got, want, tol in zip(tall, short, (1e-4, 1e-3) if precision == "fp32" else (1e-12, 1e-12)):
        assert float((got.double() - want).norm() / want.norm()) <= tol


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_fp32_tall(kind):
    pair("fp32", 72, 66, (1 << 31) // (72 * 66) + 150, True, kind)

"""What a user of this framework has it do, as timed cases.

Each case is one pass through the public entry points (``HybMesh``,
``autograd.hyb_trace``, the batched C ABI): a forward solve, a gradient
evaluation (forward, misfit, adjoint, gradient), a batch of independent
gradients as the serving engine runs it, one iteration of the conjugate
gradient loop, or the data misfit of recorded traces.  Sizes, step counts,
boundary conditions and sources are those of the repository's workloads
(``synth``) or ragged ones of the same kind; the coefficient and the data are
made from the seed.  Long runs are cut to fewer time steps.

``exact`` solves the same discrete problem in 64 bits with plain torch: the
7-point rows and Kuhn/bisected element rows as one symmetric operator
K u = sum over edges, its lumped mass, the absorbing rows face by face, the
adjoint as the literal transpose.
"""
import math

import torch

from paper_1509_01399_gb300 import hyb as H
from paper_1509_01399_gb300.autograd import hyb_trace

ABC6 = "111111"


def listed():
    return [
        # the repository's small reference problem: 33^3, one source, FP64, 400 steps (latency and launches)
        _case("grad_33_fp64", "grad", (33, 33, 33), "fp64", 400, fem="half", omega=40.0, a_max=4.0, cfl=0.866),
        # the waveguide of the reconstruction study (FP64, reflecting sides, Model Problem 1's initial state): a CG step
        _case("study_cg_fp64", "cg", (69, 17, 17), "fp64", 500, fem="margin2", omega=40.0, a_max=5.0, cfl=0.232,
              bc="110000", face=0, initial=True, weights=1),
        # serving: eight requests of the 65^3 class in one batch (FP32, each its own coefficient)
        _case("serve_65_x8_fp32", "batch", (65, 65, 65), "fp32", 400, nsrc=8, fem="half", omega=40.0, a_max=3.0),
        # the inverse problem on 129^3 with refined voxels around the inclusions (FP32): a CG step, stored history
        _case("cg_129_refined_fp32", "cg", (129, 129, 129), "fp32", 750, fem="half", omega=40.0, a_max=5.0,
              cfl=0.53, refine=0.003, weights=1),
        # the differentiable solve of the autograd form: 97^3, FP64, checkpoints every 50 steps
        _case("autograd_97_fp64", "autograd", (97, 97, 97), "fp64", 300, ckpt=50, fem="half", omega=40.0, a_max=4.0),
        # the large batched inversion: 257^3, eight sources, a sixth of the voxels refined, checkpoints: a CG step
        _case("cg_257_x8_refined_fp32", "cg", (257, 257, 257), "fp32", 400, nsrc=8, ckpt=50, fem="half", omega=40.0,
              a_max=2.5, cfl=0.55, refine=0.17, weights=1),
        # data generation on a ragged lattice: forward only, one oblique source, FP32
        _case("forward_ragged_fp32", "forward", (250, 171, 215), "fp32", 200, fem="half", omega=30.0, a_max=2.0,
              diag=True),
        # a double-precision gradient on a ragged mid-size lattice, two sources, quadrature weights
        _case("grad_ragged_fp64", "grad", (131, 118, 143), "fp64", 100, nsrc=2, fem="half", omega=30.0, a_max=3.0,
              weights=1),
        # per-axis steps: the anisotropic box with its eight sources, differentiable solve with FP32 sigma
        _case("aniso_257x193x321_x8_fp32", "autograd", (257, 193, 321), "fp32", 350, nsrc=8, ckpt=50, fem="half",
              omega=40.0, a_max=2.5, aniso=True),
        # the telegraph (damped) model, four sources, FP32, checkpoints
        _case("telegraph_193_x4_fp32", "autograd", (193, 193, 193), "fp32", 300, nsrc=4, ckpt=50, fem="half",
              omega=40.0, a_max=2.5, model="telegraph"),
        # the paper's own adjoint scheme on a ragged small lattice, mixed boundary conditions
        _case("paper_adjoint_ragged_fp32", "autograd", (66, 49, 57), "fp32", 300, fem="half", omega=25.0, a_max=4.0,
              bc="110011", adjoint="paper"),
        # the data misfit with its cotangent on recorded traces of eight sources
        _case("misfit_129_x8_fp32", "misfit", (129, 129, 129), "fp32", 600, nsrc=8, fem="half", omega=40.0,
              a_max=3.0, weights=1),
    ]


def _case(name, call, n, prec, steps, nsrc=1, ckpt=0, fem="half", omega=40.0, a_max=3.0, cfl=0.9, bc=ABC6, face=5,
          refine=0.0, weights=0, diag=False, aniso=False, model="wave", adjoint="exact", initial=False):
    return dict(name=name, call=call, nx=n[0], ny=n[1], nz=n[2], prec=prec, steps=steps, nsrc=nsrc, ckpt=ckpt,
                fem=fem, omega=omega, a_max=a_max, cfl=cfl, bc=bc, face=face, refine=refine, weights=weights,
                diag=diag, aniso=aniso, model=model, adjoint=adjoint, initial=initial)


def draw(rng):
    call = rng.choice(["grad", "cg", "batch", "autograd", "autograd", "forward", "misfit"])
    prec = "fp64" if call in ("grad", "cg", "autograd") and rng.random() < 0.35 else "fp32"
    top = 140 if prec == "fp64" else 260
    side = lambda: int(round(math.exp(rng.uniform(math.log(25), math.log(top)))))  # noqa: E731
    base = side()
    n = [max(20, min(300, int(base * rng.uniform(0.7, 1.4)))) for _ in range(3)]
    nodes = n[0] * n[1] * n[2]
    nsrc = rng.choice([1, 1, 2, 3, 4, 8])
    budget = 1.2e10 if prec == "fp32" else 8e8  # node-steps of one sweep
    while nodes * nsrc * 40 > budget and nsrc > 1:
        nsrc -= 1
    steps = max(20, int(min(math.exp(rng.uniform(math.log(20), math.log(600))), budget / (nodes * nsrc))))
    c = _case("", call, n, prec, steps, nsrc=nsrc, omega=rng.choice([20.0, 30.0, 40.0]),
              a_max=rng.choice([2.0, 3.0, 5.0]), cfl=round(rng.uniform(0.6, 0.9), 3))
    del c["name"]
    c["fem"] = rng.choice(["half", "half", "third", "margin2"])
    if call in ("grad", "autograd", "cg", "batch"):  # time for the waves of both sweeps to cross to the block
        need = 1.8 * {"half": 0.25, "third": 0.34, "margin2": 0.05}[c["fem"]] * max(n) * math.sqrt(3 * c["a_max"]) / c["cfl"]
        c["steps"] = steps = max(steps, int(need))
        while nodes * nsrc * steps > budget and nsrc > 1:
            nsrc -= 1
        c["nsrc"] = nsrc
    c["ckpt"] = rng.choice([0, 0, 25, 50]) if call in ("grad", "autograd", "cg") else 0
    if nodes * nsrc * steps > 4e8 and call != "batch":
        c["ckpt"] = 25
    c["weights"] = rng.choice([0, 1]) if call in ("grad", "cg", "batch", "misfit") else 0
    c["bc"] = rng.choice([ABC6, ABC6, ABC6, "110011", "001111", "000011"])
    c["face"] = rng.randrange(6)
    c["diag"] = rng.random() < 0.25
    kind = rng.choice(["plain", "plain", "refine", "aniso", "telegraph", "paper"])
    if call in ("grad", "autograd", "cg"):
        if kind == "refine" and c["fem"] != "margin2":
            c["refine"], c["cfl"] = round(rng.uniform(0.001, 0.2), 4), 0.53
        elif kind == "aniso":
            c["aniso"] = True
        elif kind == "telegraph" and call != "cg":
            c["model"] = "telegraph"
        elif kind == "paper" and call != "cg":
            c["adjoint"] = "paper"
    return c


# ---- inputs ----
class _Source:
    def __init__(self, face, omega, direction=None):
        self.face, self.omega, self.amp, self.direction = face, omega, 1.0, direction


def _geometry(case):
    n = (case["nx"], case["ny"], case["nz"])
    if case["fem"] == "margin2":
        lo, hi = (2, 2, 2), tuple(v - 3 for v in n)
    elif case["fem"] == "third":
        lo, hi = tuple(v // 3 for v in n), tuple(v - 1 - v // 3 for v in n)
    else:
        lo, hi = tuple((v - 1) // 4 for v in n), tuple(3 * (v - 1) // 4 for v in n)
    ud = tuple(hi[d] - lo[d] - 2 for d in range(3))
    if case["aniso"]:
        hv = tuple(2.0 / (v - 1) for v in n)
    else:
        hv = (2.0 / (max(n) - 1),) * 3
    dt = case["cfl"] / math.sqrt(case["a_max"] * sum(1.0 / (h * h) for h in hv))
    return n, lo, hi, ud, hv, dt


def _sources(case):
    d3 = [(1.0, 1.0, 1.0), (-1.0, -1.0, -1.0), (1.0, 0.0, 1.0), (0.0, -1.0, -1.0)]
    out = []
    for s in range(case["nsrc"]):
        if case["call"] == "batch" or s < 6 and not (case["diag"] and s % 2 == 0):
            face = case["face"] if case["call"] == "batch" else (case["face"] + s) % 6
            out.append(_Source(face, case["omega"]))
        else:
            d = d3[s // 2 % 4 if case["diag"] else s % 2]
            ax = 2 if d[2] else 0
            out.append(_Source(2 * ax + (0 if d[ax] > 0 else 1), case["omega"], d))
    return out


def _bumps(case, gen, ud, hv, amp):
    """Smooth sigma >= 0 on the unknown voxels: four to eight Gaussian bumps."""
    ax = [torch.arange(ud[d], device="cuda", dtype=torch.float64) * hv[d] for d in range(3)]
    sig = torch.zeros(ud[2], ud[1], ud[0], device="cuda", dtype=torch.float64)
    r = torch.rand(8, 5, generator=gen, device="cuda", dtype=torch.float64).cpu().tolist()
    for b in range(4 + int(r[0][4] * 5) if r[0][4] < 1 else 8):
        p = r[min(b, 7)]
        w = 0.05 + 0.1 * p[3]
        e = [torch.exp(-((ax[d] - p[d] * float(ax[d][-1])) ** 2) / (2 * w * w)) for d in range(3)]
        sig += (0.2 + 0.8 * p[4]) * (e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :])
    return (sig * (amp / float(sig.max()))).reshape(-1)


def _inputs(case, seed):
    n, lo, hi, ud, hv, dt = _geometry(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * int(seed) + 17)
    amp = 0.5 * (case["a_max"] - 1.0)
    nset = case["nsrc"] if case["call"] == "batch" else 1
    true = torch.stack([_bumps(case, gen, ud, hv, amp) for _ in range(nset)])
    refine = None
    if case["refine"] > 0:
        k = max(1, int(case["refine"] * true.shape[1]))
        refine = torch.zeros(true.shape[1], dtype=torch.uint8, device="cuda")
        refine[torch.topk(true[0], k).indices] = 1
    # the current guess of the coefficient: part of the perturbation, rounded to FP32 (an FP32 parameter)
    sigma = (0.4 * true).float()
    if case["call"] == "misfit":
        sigma = sigma * 0
    srcs = _sources(case)
    stride = max(n[0] * n[1], n[0] * n[2], n[1] * n[2])
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    shape = (len(srcs), case["steps"] + 1, stride)
    t = torch.arange(case["steps"] + 1, device="cuda", dtype=torch.float64) * dt
    obs = torch.zeros(shape, dtype=dtype, device="cuda")
    for s, src in enumerate(srcs):  # the background plane wave on the observation face, an echo, and 3 % noise
        a = src.face >> 1
        p, q = [d for d in range(3) if d != a]
        w = src.omega
        f = lambda s_: torch.where((s_ >= 0) & (s_ <= 2 * math.pi / w), (1 - torch.cos(w * s_)) / w, 0 * s_)  # noqa: E731
        delay = torch.zeros(n[q], n[p], device="cuda", dtype=torch.float64)
        if src.direction:
            nrm = math.sqrt(sum(v * v for v in src.direction))
            for d in (p, q):
                v = src.direction[d] / nrm
                i = torch.arange(n[d], device="cuda", dtype=torch.float64)
                along = abs(v) * hv[d] * (i if v >= 0 else n[d] - 1 - i)
                delay = delay + (along[None, :] if d == p else along[:, None])
        m = n[p] * n[q]
        wave = f(t[:, None] - delay.reshape(1, -1)) if src.direction else f(t)[:, None]
        echo = 0.15 * f(t - 0.35 * float(t[-1]))[:, None]
        noise = torch.randn(len(t), m, generator=gen, device="cuda", dtype=torch.float32) * (0.06 / w)
        obs[s, :, :m] = (wave + echo + noise).to(dtype)
        obs[s, 0] = 0
    u0 = None
    if case["initial"]:
        r2 = sum(((torch.arange(n[d], device="cuda", dtype=torch.float64) - 0.5 * (n[d] - 1)) * hv[d])
                 .reshape([-1 if e == 2 - d else 1 for e in range(3)]) ** 2 for d in range(3))
        u0 = torch.exp(-r2).contiguous()
    return dict(n=n, lo=lo, hi=hi, ud=ud, hv=hv, dt=dt, sigma=sigma, refine=refine, srcs=srcs, obs=obs, u0=u0, gen=gen)


def prepare(case, seed):
    v = _inputs(case, seed)
    m = H.HybMesh(v["n"], v["hv"][0], v["lo"], v["hi"], tuple(int(b) for b in case["bc"]), case["prec"], case["ckpt"],
                  case["a_max"], (-1.0, -1.0, -1.0), refine=None if v["refine"] is None else v["refine"].cpu().numpy(),
                  adjoint_mode=H.HYB_ADJ_PAPER if case["adjoint"] == "paper" else H.HYB_ADJ_EXACT,
                  model=H.HYB_MODEL_TELEGRAPH if case["model"] == "telegraph" else H.HYB_MODEL_WAVE,
                  spacing=v["hv"] if case["aniso"] else None)
    st = dict(case=case, mesh=m, srcs=v["srcs"], dt=v["dt"], obs=v["obs"])
    if v["u0"] is not None:
        m.set_initial(v["u0"], v["u0"])
    coef = v["sigma"].double() + (0.0 if case["model"] == "telegraph" else 1.0)
    call = case["call"]
    if call in ("grad", "forward"):
        st["a"] = coef[0].contiguous()
    elif call == "batch":
        st["a"] = coef.contiguous()
    elif call == "autograd":
        # an FP32 mesh is driven by an FP32 parameter, an FP64 mesh by an FP64 one
        st["sigma"] = (v["sigma"][0].double() if case["prec"] == "fp64" else v["sigma"][0].clone()).requires_grad_(True)
        st["shift"] = case["model"] == "telegraph"
    elif call == "cg":
        st["a0"] = coef[0].contiguous()
        st["a"] = st["a0"].clone()
        st["cg"] = m.new_cg_state()
    elif call == "misfit":
        # traces recorded by an earlier solve: here the data themselves, with the echo scaled and noise of their own
        m.forward(coef[0].contiguous(), v["srcs"], case["steps"], v["dt"])
        noise = torch.randn(v["obs"].shape, generator=v["gen"], device="cuda", dtype=torch.float32) * 1e-3
        st["trace"] = (0.9 * v["obs"] + noise.to(v["obs"].dtype)).contiguous()
    return st


def run(state):
    case, m, srcs, dt, steps = state["case"], state["mesh"], state["srcs"], state["dt"], state["case"]["steps"]
    call = case["call"]
    if call == "forward":
        trace = m.forward(state["a"], srcs, steps, dt)
        return {"trace": trace, "u": m.field(H.HYB_FIELD_U_LAST, 0)}
    if call == "grad":
        trace = m.forward(state["a"], srcs, steps, dt)
        J, cot = m.misfit(trace, state["obs"], case["weights"], want_cot=True)
        m.adjoint(cot)
        g = m.gradient(state["a"], 0.01, 1.0)
        return {"trace": trace, "J": J, "g": g if case["prec"] == "fp64" else g.float()}
    if call == "batch":
        k = len(srcs)
        trace = m.new_trace(k, steps)
        H.hyb_forward_batch(m.handle, state["a"].data_ptr(), srcs, steps, dt, trace.data_ptr())
        cot = torch.empty_like(trace)
        J = H.hyb_misfit_batch(m.handle, trace.data_ptr(), state["obs"].data_ptr(), case["weights"], k, cot.data_ptr())
        H.hyb_adjoint(m.handle, cot.data_ptr(), 0)
        g = torch.empty_like(state["a"])
        H.hyb_gradient_batch(m.handle, state["a"].data_ptr(), 0.0, 1.0, g.data_ptr())
        # an FP32 mesh's gradient is kept as the FP32 vector that a request's answer carries
        return {"trace": trace, "J": J, "g": g.float()}
    if call == "autograd":
        sigma = state["sigma"]
        sigma.grad = None
        # (hyb_trace adds the background a = 1; the telegraph model's coefficient is sigma itself)
        trace = hyb_trace(sigma - 1.0 if state["shift"] else sigma, m, srcs, steps, dt)
        r = trace - state["obs"]
        loss = 0.5 * (r * r).sum()
        loss.backward()
        return {"trace": trace.detach(), "grad": sigma.grad}
    if call == "cg":
        a = state["a"].copy_(state["a0"])
        st = state["cg"]
        st.gnorm2, st.alpha, st.J, st.iter = 0.0, 0.0, 0.0, 0
        rep = m.cg_step(a, state["obs"], srcs, steps, dt, st, gamma=0.01, a0=1.0, a_min=1.0, weights=case["weights"])
        return {"a": a if case["prec"] == "fp64" else a.float(), "J": rep.J, "gnorm": rep.gnorm}
    J, cot = m.misfit(state["trace"], state["obs"], case["weights"], want_cot=True)
    return {"J": J, "cot": cot}


def work(case):
    n, lo, hi, ud, hv, dt = _geometry(case)
    e = 8 if case["prec"] == "fp64" else 4
    N = n[0] * n[1] * n[2]
    own = math.prod(hi[d] - lo[d] - 1 for d in range(3))
    stride = max(n[0] * n[1], n[0] * n[2], n[1] * n[2])
    tb = case["nsrc"] * (case["steps"] + 1) * stride * e
    if case["call"] == "misfit":
        return {"bytes": 3 * tb, "flops": 4 * tb // e}
    # a level reads u^k, u^{k-1} (and the coefficient on FEM-owned nodes) and writes u^{k+1}; a transposed level
    # also reads the state of the FEM-owned nodes
    fwd, adj = e * (3 * N + own), e * (3 * N + 2 * own)
    levels = case["nsrc"] * case["steps"]
    nf = 3 if case["call"] == "cg" else 1
    if case["ckpt"] and case["call"] != "forward":
        nf = nf if case["call"] != "cg" else 2
        nf += 1  # the recomputed segments
    elif case["call"] == "cg":
        nf = 2
    na = 0 if case["call"] == "forward" else 1
    flops = levels * (nf * (10 * N + 8 * own) + na * (10 * N + 60 * own))
    return {"bytes": levels * (nf * fwd + na * adj) + tb, "flops": flops}


# ---- the same discrete problem in 64 bits ----
class _Exact:
    """Nodes u[z, y, x] plus the centre nodes of refined voxels."""

    def __init__(self, case, v, a):
        self.case, self.n, self.hv, self.dt = case, v["n"], v["hv"], v["dt"]
        dev, f64 = "cuda", torch.float64
        n, lo, hi, ud = v["n"], v["lo"], v["hi"], v["ud"]
        self.fl = [lo[d] + 1 for d in range(3)]
        self.ud = ud
        tel = case["model"] == "telegraph"
        av = torch.ones(n[2] - 1, n[1] - 1, n[0] - 1, device=dev, dtype=f64)
        box = tuple(slice(self.fl[d], self.fl[d] + ud[d]) for d in (2, 1, 0))
        if not tel:
            av[box] = a.reshape(ud[2], ud[1], ud[0])
        self.kap = [self.hv[0] ** 2 / h ** 2 for h in self.hv]
        # edge weights along each axis: 1 off the unknown voxels' edges, sums of a_c / 3 and a_c / 6 on them,
        # halved by the missing voxels on the outer faces (K of the whole box, symmetric)
        self.W = []
        for d in range(3):
            shape = [n[2], n[1], n[0]]
            shape[2 - d] -= 1
            w = torch.zeros(shape, device=dev, dtype=f64)
            o = [e for e in (2, 1, 0) if e != d]  # the two other axes
            for b0 in (0, 1):
                for b1 in (0, 1):
                    at = [slice(None)] * 3
                    at[2 - o[0]] = slice(b0, n[o[0]] - 1 + b0)
                    at[2 - o[1]] = slice(b1, n[o[1]] - 1 + b1)
                    w[tuple(at)] += av * (1.0 / 3.0 if b0 == b1 else 1.0 / 6.0)
            # the outer boundary rows are finite-difference rows: weights 1, halved per boundary axis
            ones = torch.ones_like(w)
            for e in o:
                for end in (0, n[e] - 1):
                    at = [slice(None)] * 3
                    at[2 - e] = end
                    ones[tuple(at)] *= 0.5
            edge = torch.zeros_like(w, dtype=torch.bool)
            for e in o:
                for end in (0, n[e] - 1):
                    at = [slice(None)] * 3
                    at[2 - e] = end
                    edge[tuple(at)] = True
            self.W.append(torch.where(edge, ones, w) * self.kap[d])
        M = torch.ones(n[2], n[1], n[0], device=dev, dtype=f64)
        self.D = M
        for d in range(3):
            for end in (0, n[d] - 1):
                at = [slice(None)] * 3
                at[2 - d] = end
                M[tuple(at)] *= 0.5
        self.N = M.numel()
        self.M = M.reshape(-1)
        self.nc = 0
        if v["refine"] is not None:
            ids = torch.nonzero(v["refine"]).reshape(-1)
            self.nc = ids.numel()
            x, y, z = ids % ud[0], ids // ud[0] % ud[1], ids // (ud[0] * ud[1])
            K8, m8, K9, m9 = _voxel_matrices()
            corner = [(z + self.fl[2] + (c >> 2)) * n[1] * n[0] + (y + self.fl[1] + (c >> 1 & 1)) * n[0]
                      + x + self.fl[0] + (c & 1) for c in range(8)]
            self.ridx = torch.stack(corner + [self.N + torch.arange(self.nc, device=dev)], 1)
            self.ra = a[ids]
            self.rids = ids
            self.K9 = K9.to(dev)
            self.dK = K9.clone()
            self.dK[:8, :8] -= K8
            self.dK = self.dK.to(dev)
            self.M = torch.cat([self.M, torch.zeros(self.nc, device=dev, dtype=f64)])
            dm = m9.clone()
            dm[:8] -= m8
            self.M.index_add_(0, self.ridx.reshape(-1), dm.to(dev).repeat(self.nc))
        self.c2 = self.dt ** 2 / self.hv[0] ** 2
        self.s = None
        if tel:
            s = torch.zeros(n[2], n[1], n[0], device=dev, dtype=f64)
            sg = a.reshape(ud[2], ud[1], ud[0])
            for c in range(8):
                at = tuple(slice(self.fl[d] + (c >> d & 1), self.fl[d] + (c >> d & 1) + ud[d]) for d in (2, 1, 0))
                s[at] += sg * (0.25 if c in (0, 7) else 1.0 / 12.0)
            self.s = (0.5 * self.dt * s).reshape(-1)
        # nodes by the number of outer faces they lie on (the absorbing rows' levels)
        self.groups = []
        for cz in (0, 1, 2):
            for cy in (0, 1, 2):
                for cx in (0, 1, 2):
                    pos = (cz, cy, cx)
                    faces = [2 * d + (1 if pos[2 - d] == 2 else 0) for d in range(3) if pos[2 - d] != 1]
                    if faces:
                        at = tuple(slice(0, 1) if p == 0 else slice(1, n[2 - i] - 1) if p == 1 else
                                   slice(n[2 - i] - 1, n[2 - i]) for i, p in enumerate(pos))
                        self.groups.append((len(faces), faces, at))
        self.groups.sort(key=lambda g: g[0])
        self.abc = [f for f in range(6) if case["bc"][f] == "1"]

    def lap(self, u):
        """-M^{-1} K u in units of 1 / dx_1^2 (u: N + nc values)."""
        return self.minus_K(u) / self.M

    def minus_K(self, u):
        n = self.n
        g = u[: self.N].reshape(n[2], n[1], n[0])
        out = torch.zeros_like(u)
        o = out[: self.N].reshape(n[2], n[1], n[0])
        for d in range(3):
            f = self.W[d] * torch.diff(g, dim=2 - d)
            o.narrow(2 - d, 0, n[d] - 1).add_(f)
            o.narrow(2 - d, 1, n[d] - 1).sub_(f)
        if self.nc:
            y = (u[self.ridx] @ self.dK) * self.ra[:, None]
            out.index_add_(0, self.ridx.reshape(-1), -y.reshape(-1))
        return out

    # the plane wave of one source
    def wave(self, src):
        n = self.n
        d = list(src.direction or (0.0, 0.0, 0.0))
        if not any(d):
            d[src.face >> 1] = -1.0 if src.face & 1 else 1.0
        nrm = math.sqrt(sum(v * v for v in d))
        d = [v / nrm for v in d]
        t1 = 2 * math.pi / src.omega
        fac, tsw = {}, {}
        for f in range(6):
            dn = d[f >> 1] * (1.0 if f & 1 else -1.0)
            if dn < 0:
                fac[f] = -dn
                tsw[f] = t1 + sum(abs(d[e]) * (n[e] - 1) * self.hv[e] for e in range(3) if e != f >> 1)
        delay = torch.zeros(n[2], n[1], n[0], device="cuda", dtype=torch.float64)
        for e in range(3):
            i = torch.arange(n[e], device="cuda", dtype=torch.float64)
            along = d[e] * self.hv[e] * (i if d[e] >= 0 else i - (n[e] - 1))
            delay = delay + along.reshape([-1 if q == 2 - e else 1 for q in range(3)])
        return dict(fac=fac, tsw=tsw, delay=delay, t1=t1, omega=src.omega)

    def masks(self, w, k):
        t = k * self.dt
        flux = [f for f in w["fac"] if t <= w["tsw"][f]]
        return [f for f in self.abc if f not in flux], flux

    def face_at(self, f):
        at = [slice(None)] * 3
        d = f >> 1
        at[2 - d] = slice(self.n[d] - 1, self.n[d]) if f & 1 else slice(0, 1)
        return tuple(at)

    def inward(self, at, f):
        q = list(at)
        d = f >> 1
        q[2 - d] = slice(self.n[d] - 2, self.n[d] - 1) if f & 1 else slice(1, 2)
        return tuple(q)

    def r_of(self, f):
        h = self.hv[f >> 1]
        return (h - self.dt) / (h + self.dt)

    def step(self, w, k, u, p, force=None):
        """u^{k+1} from u^k and u^{k-1}; force: None, or the paper adjoint's term (every face reflects)."""
        if self.s is not None:
            new = self.c2 * self.lap(u) + 2 * u - p
            new = torch.where(self.s > 0, u + ((u - p) * (1 - self.s) + self.c2 * self.lap(u)) / (1 + self.s), new)
        else:
            new = u + ((u - p) + self.c2 * self.lap(u))
        n = self.n
        g = new[: self.N].reshape(n[2], n[1], n[0])
        if force is not None:
            g += force
            return new
        ub = u[: self.N].reshape(n[2], n[1], n[0])
        absorb, flux = self.masks(w, k)
        for f in flux:
            at = self.face_at(f)
            s = k * self.dt - w["delay"][at]
            on = (s >= 0) & (s <= w["t1"])
            g[at] += torch.where(on, self.dt ** 2 * 2.0 / self.hv[f >> 1] * w["fac"][f] * torch.sin(w["omega"] * s), 0 * s)
        for _, faces, at in self.groups:
            fb = [f for f in faces if f in absorb]
            if fb:
                acc = 0
                for f in fb:
                    q = self.inward(at, f)
                    acc = acc + ub[q] - self.r_of(f) * g[q]
                g[at] = sum(self.r_of(f) for f in fb) / len(fb) * ub[at] + acc / len(fb)
        return new

    def step_t(self, w, j, l1, l2, c):
        """lambda^j from lambda^{j+1}, lambda^{j+2} and the cotangent on the lattice."""
        n = self.n
        shape = (n[2], n[1], n[0])
        keep, _ = self.masks(w, j)
        x = l1.clone()
        for f in keep:
            x[: self.N].reshape(shape)[self.face_at(f)] = 0
        m = x / (self.M)
        if self.s is None:
            rhs = 2 * x + self.c2 * self.minus_K(m)
        else:
            rhs = 2 * x + self.c2 * self.minus_K(m)
        g = rhs[: self.N].reshape(shape)
        lb = l1[: self.N].reshape(shape)
        for _, faces, at in self.groups:
            fb = [f for f in faces if f in keep]
            if fb:
                g[at] += sum(self.r_of(f) for f in fb) / len(fb) * lb[at]
                for f in fb:
                    g[self.inward(at, f)] += lb[at] / len(fb)
        off, _ = self.masks(w, j + 1)
        y = l2 if self.s is None else l2 * (1 - self.s)
        y = y.clone()
        for f in off:
            y[: self.N].reshape(shape)[self.face_at(f)] = 0
        rhs -= y
        g += c
        solve, _ = self.masks(w, j - 1)
        for _, faces, at in reversed(self.groups):
            fb = [f for f in faces if f in solve]
            for f in fb:
                g[self.inward(at, f)] -= self.r_of(f) / len(fb) * g[at]
        return rhs if self.s is None else rhs / (1 + self.s)

    def rows(self, face):
        return (lambda g: g[self.face_at(face)].reshape(-1))

    def start(self, v):
        z = torch.zeros(self.N + self.nc, device="cuda", dtype=torch.float64)
        if v["u0"] is None:
            return z, z.clone()
        z[: self.N] = v["u0"].reshape(-1)
        return z, z.clone()

    def box(self, u):
        fl, ud, n = self.fl, self.ud, self.n
        g = u[: self.N].reshape(n[2], n[1], n[0])
        return g[fl[2]:fl[2] + ud[2] + 1, fl[1]:fl[1] + ud[1] + 1, fl[0]:fl[0] + ud[0] + 1].clone(), u[self.N:].clone()

    def forward(self, v, src, hist=None):
        n, case = self.n, self.case
        w = self.wave(src)
        p, u = self.start(v)
        rows = self.rows(src.face)
        shape = (n[2], n[1], n[0])
        trace = [rows(u[: self.N].reshape(shape))]
        for k in range(case["steps"]):
            if hist is not None and self.s is None:
                hist.append(self.box(u))
            new = self.step(w, k, u, p)
            if hist is not None and self.s is not None:
                hist.append(self.box(new - p))
            p, u = u, new
            trace.append(rows(u[: self.N].reshape(shape)))
        return torch.stack(trace), u

    def pair(self, acc, b, lam):
        """Adds the pairing of the stored box b and lambda (scaled by 1 / mass) level by level."""
        l, lc = self.box(lam)
        if self.s is not None:
            acc["p"] += b[0] * l
            return
        for d in range(3):
            acc["e"][d] += torch.diff(b[0], dim=2 - d) * torch.diff(l, dim=2 - d) * self.kap[d]
        if self.nc:
            full = torch.zeros(self.N + self.nc, device="cuda", dtype=torch.float64)
            n, fl, ud = self.n, self.fl, self.ud
            full[: self.N].reshape(n[2], n[1], n[0])[fl[2]:fl[2] + ud[2] + 1, fl[1]:fl[1] + ud[1] + 1,
                                                     fl[0]:fl[0] + ud[0] + 1] = b[0]
            full[self.N:] = b[1]
            acc["r"] += ((full[self.ridx] @ self.K9) * lam[self.ridx]).sum(1)

    def gradient(self, v, src, cot, hist):
        """dJ/da of one source from the cotangent rows [steps + 1, face]."""
        n, N, ud, case = self.n, self.case["steps"], self.ud, self.case
        w = self.wave(src)
        z = lambda *s: torch.zeros(*s, device="cuda", dtype=torch.float64)  # noqa: E731
        bs = [ud[2] + 1, ud[1] + 1, ud[0] + 1]
        acc = {"e": [z(*[bs[i] - (1 if i == 2 - d else 0) for i in range(3)]) for d in range(3)], "p": z(*bs),
               "r": z(self.nc)}
        at = self.face_at(src.face)
        shape = (n[2], n[1], n[0])
        l1, l2 = z(self.N + self.nc), z(self.N + self.nc)
        paper = case["adjoint"] == "paper"
        if paper:  # lambda^N = lambda^{N+1} = 0; pairs (u^j, lambda^j), then lambda^{j-1}
            for j in range(N, -1, -1):
                if j <= N - 1:
                    self.pair(acc, hist[j], l1)
                if j >= 1:
                    force = z(*shape)
                    force[at] = -self.dt * cot[j].reshape(force[at].shape) / (self.hv[0] ** 3 * self.D[at])
                    l1, l2 = self.step(None, None, l1, l2, force), l1
            scale = self.dt * self.hv[0]
        else:
            for j in range(N, 0, -1):
                c = z(*shape)
                c[at] = cot[j].reshape(c[at].shape)
                l1, l2 = self.step_t(w, j, l1, l2, c), l1
                self.pair(acc, hist[j - 1], l1 if self.s is not None else l1 / self.M)
            scale = -self.c2
        if self.s is not None:
            g = z(ud[2], ud[1], ud[0])
            for c in range(8):
                q = tuple(slice(c >> d & 1, (c >> d & 1) + ud[d]) for d in (2, 1, 0))
                g += acc["p"][q] * (0.25 if c in (0, 7) else 1.0 / 12.0)
            return (-0.5 * self.dt * g).reshape(-1)
        g = z(ud[2], ud[1], ud[0])
        for d in range(3):
            o = [e for e in (2, 1, 0) if e != d]
            for b0 in (0, 1):
                for b1 in (0, 1):
                    q = [slice(None)] * 3
                    q[2 - o[0]] = slice(b0, ud[o[0]] + b0)
                    q[2 - o[1]] = slice(b1, ud[o[1]] + b1)
                    g += acc["e"][d][tuple(q)] * (1.0 / 3.0 if b0 == b1 else 1.0 / 6.0)
        g = g.reshape(-1)
        if self.nc:
            g[self.rids] = acc["r"]
        return scale * g


def _voxel_matrices():
    """Unit-voxel stiffness and lumped masses: six Kuhn tetrahedra (8 nodes), each bisected at the centre (9 nodes)."""
    P = torch.tensor([[c & 1, c >> 1 & 1, c >> 2] for c in range(8)] + [[0.5] * 3], dtype=torch.float64)
    K8, m8 = torch.zeros(8, 8, dtype=torch.float64), torch.zeros(8, dtype=torch.float64)
    K9, m9 = torch.zeros(9, 9, dtype=torch.float64), torch.zeros(9, dtype=torch.float64)
    for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)):
        v = [0, 1 << a, 1 << a | 1 << b, 7]
        for K, m, t in ((K8, m8, v), (K9, m9, v[:3] + [8]), (K9, m9, [8] + v[1:])):
            X = torch.cat([torch.ones(4, 1, dtype=torch.float64), P[t]], 1)
            g = torch.linalg.inv(X)[1:]  # columns: gradients of the barycentric functions
            vol = abs(float(torch.linalg.det(X))) / 6
            for i in range(4):
                m[t[i]] += vol / 4
                for j in range(4):
                    K[t[i], t[j]] += vol * float(g[:, i] @ g[:, j])
    return K8, m8, K9, m9


def _weights(case, v, src):
    n, hv = v["n"], v["hv"]
    a = src.face >> 1
    p, q = [d for d in range(3) if d != a]
    w = torch.ones(n[q], n[p], device="cuda", dtype=torch.float64)
    if not case["weights"]:
        return w.reshape(-1), 1.0
    w *= hv[p] * hv[q]
    w[0] *= 0.5
    w[-1] *= 0.5
    w[:, 0] *= 0.5
    w[:, -1] *= 0.5
    return w.reshape(-1), v["dt"]


def exact(case, seed):
    n, _, _, _, _, _ = _geometry(case)
    sweeps = {"forward": 1, "misfit": 0, "cg": 5}.get(case["call"], 4)
    cost = n[0] * n[1] * n[2] * case["nsrc"] * case["steps"] * sweeps * (2 if case["refine"] else 1)
    if cost / 1.5e10 + case["steps"] * case["nsrc"] * sweeps * 1.5e-3 > 25:
        return None  # over about 20 seconds
    with torch.no_grad():
        return _exact(case, seed)


def _exact(case, seed):
    v = _inputs(case, seed)
    srcs, call, steps = v["srcs"], case["call"], case["steps"]
    coef = v["sigma"].double() + 1.0
    if case["model"] == "telegraph":  # (as the program forms it from its parameter)
        coef = (v["sigma"] - 1.0).double() + 1.0 if call == "autograd" and case["prec"] == "fp32" else v["sigma"].double()
    if call == "misfit":
        noise = torch.randn(v["obs"].shape, generator=v["gen"], device="cuda", dtype=torch.float32) * 1e-3
        tr = (0.9 * v["obs"] + noise.to(v["obs"].dtype))
        J, cot = 0.0, torch.zeros(v["obs"].shape, device="cuda", dtype=torch.float64)
        for s, src in enumerate(srcs):
            w, wt = _weights(case, v, src)
            m = w.numel()
            r = tr[s, 1:, :m].double() - v["obs"][s, 1:, :m].double()
            cot[s, 1:, :m] = wt * w * r
            J += 0.5 * float((wt * w * r * r).sum())
        return {"J": J, "cot": cot}

    def evaluate(a, want_grad, want_trace=True):
        """Traces, misfit per source and gradient per source at the coefficient(s) a."""
        trace = torch.zeros(v["obs"].shape, device="cuda", dtype=torch.float64) if want_trace else None
        Js, gs, last = [], [], None
        op = None
        for s, src in enumerate(srcs):
            if op is None or call == "batch":
                op = _Exact(case, v, a[s] if call == "batch" else a[0])
            hist = [] if want_grad else None
            tr, u = op.forward(v, src, hist)
            w, wt = _weights(case, v, src)
            m = w.numel()
            r = tr - v["obs"][s, :, :m].double()
            r[0] = 0
            Js.append(0.5 * float((wt * w * r * r).sum()))
            if want_grad:
                gs.append(op.gradient(v, src, wt * w * r, hist))
            if want_trace:
                trace[s, :, :m] = tr
            if s == 0:
                last = u[: op.N].reshape(v["n"][2], v["n"][1], v["n"][0]).clone()
        return trace, Js, gs, last

    vol = v["hv"][0] * v["hv"][1] * v["hv"][2]
    if call == "forward":
        trace, _, _, u = evaluate(coef, False)
        return {"trace": trace, "u": u}
    if call == "grad":
        trace, J, g, _ = evaluate(coef, True)
        return {"trace": trace, "J": sum(J), "g": sum(g) + 0.01 * vol * (coef[0] - 1.0)}
    if call == "batch":
        trace, J, g, _ = evaluate(coef, True)
        return {"trace": trace, "J": J, "g": torch.stack(g)}
    if call == "autograd":
        trace, _, g, _ = evaluate(coef, True)
        return {"trace": trace, "grad": sum(g)}
    # one CG iteration from the start: projected steepest descent, a trial step, the parabola's minimum
    a = coef[0]
    lo, hi, gamma = 1.0, case["a_max"], 0.01
    _, J, g, _ = evaluate(coef, True, False)
    g = sum(g) + gamma * vol * (a - 1.0)
    F = lambda J_, a_: sum(J_) + 0.5 * gamma * vol * float(((a_ - 1.0) ** 2).sum())  # noqa: E731
    F0 = F(J, a)
    out = lambda d_: ((a <= lo) & (d_ < 0)) | ((a >= hi) & (d_ > 0))  # noqa: E731
    d = torch.where(out(-g), 0 * g, -g / vol)
    d = torch.where(out(d), 0 * d, d)
    slope, at = float((g * d).sum()), 0.5 / float(d.abs().max())
    trial = (a + at * d).clamp(lo, hi)
    _, Jt, _, _ = evaluate(trial[None], False, False)
    curve = F(Jt, trial) - F0 - slope * at
    alpha = at if curve <= 0 else -slope * at * at / (2 * curve)
    alpha = min(max(alpha, 0.0), 4 * at)
    return {"a": (a + alpha * d).clamp(lo, hi), "J": F0, "gnorm": math.sqrt(float((g * g).sum()) / vol)}

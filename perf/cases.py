"""Performance cases: the work a user of the solver has it do, through its public entry points.

A case is a dict of plain values. Three kinds:
  plan   one field advanced `steps` time steps by `Plan.run` (or `Plan.step`): 2D and 3D, FP32 and
         FP64, ETDRK1 and ETDRK2, Dirichlet and periodic boundaries, the FFT and the tensor-core routes;
  batch  many independent 2D problems of uneven size advanced together by `Batch.run`;
  sno    the spectral neural operator: a forward pass (inference) or the loss gradient (training).
Sizes are those of the repository's own workloads (paper_2209_11922_gb300/inputs.py, bench.py, the
tests), or other supported lengths (2^k and 3 2^k) between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2209_11922_gb300.etd import Batch, Plan
from paper_2209_11922_gb300.sno import PARAM_NAMES, Sno, param_shapes

BATCH_SIZES = (64, 96, 128, 192, 256, 384)   # mesh lengths of the batched workload


def _plan(name, N, D, tau, scheme, dtype, steps, amp=0.9, **kw):
    nz = N[2] if len(N) == 3 else 0
    c = {"kind": "plan", "nx": N[0], "ny": N[1], "nz": nz, "D": D, "tau": tau, "scheme": scheme,
         "dtype": dtype, "steps": steps, "amp": amp, "bc": "dirichlet", "route": "auto",
         "flory_huggins": False, "source": False, **kw}
    return {"name": name, **c} if name else c


def _batch(name, count, steps, seed, scheme=2):
    c = {"kind": "batch", "count": count, "steps": steps, "tau": 1e-2, "scheme": scheme, "mesh_seed": seed}
    return {"name": name, **c} if name else c


def _sno(name, N, C, M, L, batch, grad):
    c = {"kind": "sno", "N": N, "C": C, "M": M, "L": L, "batch": batch, "grad": grad}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one time step of a small ragged field, as a program that looks at every step does it
        _plan("step_2d_128x96_f32", (128, 96), 1e-2, 1e-2, 2, "f32", 1),
        # the small FP64 configuration, its whole run to T = 1
        _plan("run_2d_64_f64", (64, 64), 1e-2, 1e-2, 2, "f64", 100),
        # the headline: the 2D 1024^2 run in FP32
        _plan("run_2d_1024_f32", (1024, 1024), 1e-4, 5e-3, 2, "f32", 64, amp=0.05),
        # the same mesh in FP64, with the first-order scheme
        _plan("run_2d_1024_f64_rk1", (1024, 1024), 1e-4, 5e-3, 1, "f64", 32, amp=0.05),
        # a ragged anisotropic mesh, first-order scheme
        _plan("run_2d_768x192_f32_rk1", (768, 192), 1e-3, 1e-2, 1, "f32", 50),
        # the manufactured-solution mesh with a time-dependent source, FP64
        _plan("run_2d_2048x1024_f64_source", (2048, 1024), 1e-2, 1.0 / 128, 2, "f64", 6, amp=0.5, source=True),
        # the 3D run
        _plan("run_3d_256_f32", (256, 256, 256), 1e-3, 1e-2, 2, "f32", 8),
        # the 3D run on the split-BF16 tensor-core transforms
        _plan("run_3d_256_f32_bf16x3", (256, 256, 256), 1e-3, 1e-2, 2, "f32", 6, route="gemm_bf16x3"),
        # grain coarsening: periodic cube with the Flory-Huggins reaction, 32 steps between two looks at the field
        _plan("run_3d_128_periodic_fh_f32", (128, 128, 128), 1e-4, 20.0 / 2048, 2, "f32", 32,
              bc="periodic", flory_huggins=True),
        # the batched workload: 512 problems of uneven mesh and diffusion
        _batch("batch_512_f32", 512, 20, 1),
        # the learned coarse propagator applied to the 64 fields of a Parareal sweep
        _sno("sno_forward_256_b64", 256, 32, 24, 4, 64, False),
        # its training gradient
        _sno("sno_gradient_256_b32", 256, 32, 24, 4, 32, True),
    ]


def _lengths(lo, hi):
    out = sorted({2 ** k for k in range(2, 12)} | {3 * 2 ** k for k in range(1, 10)})
    return [n for n in out if lo <= n <= hi]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["plan2", "plan2", "plan2", "plan3", "plan3", "batch", "sno"])
    if kind == "batch":
        return _batch(None, max(2, round(_logu(rng, 4, 512))), rng.randint(2, 20), rng.randrange(1, 10 ** 6),
                      rng.choice([1, 2, 2]))
    if kind == "sno":
        grad = rng.random() < 0.4
        N = rng.choice([64, 96, 128, 192, 256])
        B = max(1, round(_logu(rng, 1, 32 if grad else 64)))
        return _sno(None, N, rng.choice([16, 32]), rng.choice([12, 16, 24]), rng.randint(2, 4), B, grad)
    dtype = rng.choice(["f32", "f32", "f64"])
    scheme = rng.choice([1, 2, 2])
    bc = rng.choice(["dirichlet", "dirichlet", "periodic"])
    fh = bc == "periodic" and rng.random() < 0.5
    D = _logu(rng, 1e-4, 1e-2)
    tau = _logu(rng, 4e-3, 1e-2)
    if kind == "plan2":
        N = [rng.choice(_lengths(32, 2048)) for _ in range(2)]
        cost = N[0] * N[1] * (16 if dtype == "f64" else 1)
        steps = max(1, min(100, round(_logu(rng, 1, 100)), int(1e9 / cost)))
    else:
        N = [rng.choice(_lengths(24, 256)) for _ in range(3)]
        cost = N[0] * N[1] * N[2] * (16 if dtype == "f64" else 1) * 2
        steps = max(1, min(50, round(_logu(rng, 1, 50)), int(4e8 / cost)))
    route = "auto"
    if dtype == "f32" and all(n % 32 == 0 for n in N) and rng.random() < 0.15:
        route = "gemm_bf16x3"
    source = kind == "plan2" and bc == "dirichlet" and route == "auto" and rng.random() < 0.2
    return _plan(None, tuple(N), D, tau, scheme, dtype, steps, amp=rng.choice([0.05, 0.5, 0.9]), bc=bc,
                 route=route, flory_huggins=fh, source=source)


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(shape, amp, g, dtype=torch.float32):
    return (2.0 * torch.rand(shape, generator=g, device="cuda", dtype=dtype) - 1.0) * amp


def _dims(case):
    return [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] else [])


def _reaction(case):
    # Flory-Huggins with theta = 0.8, theta_c = 1.6, or Allen-Cahn
    return (1.6, 0.0, -0.8) if case["flory_huggins"] else (1.0, -1.0, 0.0)


def _source(case):
    """Separable source amp exp(-rate t) g_x g_y of the manufactured-solution runs."""
    gs = [np.sin(math.pi * np.arange(1, n) / n) for n in _dims(case)]
    return 0.25, 1.0, gs


def _meshes(case):
    r = np.random.default_rng(case["mesh_seed"])
    N = [(int(r.choice(BATCH_SIZES)), int(r.choice(BATCH_SIZES))) for _ in range(case["count"])]
    D = [float(d) for d in np.exp(r.uniform(math.log(1e-4), math.log(1e-2), case["count"]))]
    return N, D


def _field(case, seed):
    cut = 0 if case["bc"] == "periodic" else 1
    shape = tuple(n - cut for n in reversed(_dims(case)))
    return _uniform(shape, case["amp"], _gen(seed), torch.float64 if case["dtype"] == "f64" else torch.float32)


def _batch_fields(case, seed):
    N, D = _meshes(case)
    flat = _uniform((sum((a - 1) * (b - 1) for a, b in N),), 0.9, _gen(seed))
    return N, D, flat


def _views(flat, N):
    out, off = [], 0
    for a, b in N:
        out.append(flat[off:off + (a - 1) * (b - 1)].view(b - 1, a - 1))
        off += (a - 1) * (b - 1)
    return out


def _sno_data(case, seed):
    """Weights of the operator's usual initial scales, fields, diffusion coefficients and training targets."""
    C, M, L, B, n = case["C"], case["M"], case["L"], case["batch"], case["N"] - 1
    g = _gen(seed)
    scale = {"Wl": 1.0, "bl": 0.1, "Wm": 1.0 / C, "Wp": 1.0 / math.sqrt(C), "bp": 0.1, "Wq": 0.1 / math.sqrt(C),
             "bq": 0.01}
    shapes = param_shapes(C, M, L)
    P = {k: _uniform(shapes[k] or (1,), scale[k], g).reshape(shapes[k]) for k in PARAM_NAMES}
    u = _uniform((B, n, n), 0.9, g)
    target = 0.5 * u + _uniform((B, n, n), 0.1, g)
    r = np.random.default_rng(seed)
    D = [float(d) for d in np.exp(r.uniform(math.log(1e-4), math.log(1e-2), B))]
    return P, u, target, D


def prepare(case, seed):
    if case["kind"] == "plan":
        flin, fcub, flog = _reaction(case)
        plan = Plan(_dims(case), case["D"], case["tau"], scheme=case["scheme"], dtype=case["dtype"], flin=flin,
                    fcub=fcub, flog=flog, bc=case["bc"], route=case["route"])
        if case["source"]:
            amp, rate, gs = _source(case)
            plan.set_source(amp, rate, *gs)
        u0 = _field(case, seed)
        return {"case": case, "plan": plan, "u0": u0, "u": torch.empty_like(u0)}
    if case["kind"] == "batch":
        N, D, flat = _batch_fields(case, seed)
        u = torch.empty_like(flat)
        return {"case": case, "batch": Batch(N, D, case["tau"], scheme=case["scheme"], dtype="f32"), "u0": flat,
                "u": u, "fields": _views(u, N)}
    P, u, target, D = _sno_data(case, seed)
    op = Sno(case["N"], case["C"], case["M"], case["L"], case["batch"])
    op.set_params({k: v.cpu().numpy() for k, v in P.items()})
    return {"case": case, "sno": op, "u": u, "target": target, "D": D, "out": torch.empty_like(u)}


def run(state):
    case = state["case"]
    if case["kind"] == "plan":
        u = state["u"].copy_(state["u0"])
        if case["steps"] == 1 and not case["source"]:
            return state["plan"].step(u)
        return state["plan"].run(u, case["steps"])
    if case["kind"] == "batch":
        state["u"].copy_(state["u0"])
        state["batch"].run(state["fields"], case["steps"])
        return state["u"]
    if case["grad"]:
        loss, grads = state["sno"].gradient(state["u"], state["D"], state["target"])
        return [loss] + [grads[k] for k in PARAM_NAMES]
    return state["sno"].forward(state["u"], state["D"], out=state["out"])


# ---------------------------------------------------------------- work

def _step_flops(N, scheme):
    """Flops of the sine transforms of a time step, 2.5 N log2 N per pencil: per stage an inverse and a
    forward transform along every axis, plus one transform of the state per axis and step kept spectral."""
    unk = math.prod(N)
    per_transform_set = sum(2.5 * math.log2(n) for n in N) * unk
    return 2.0 * scheme * per_transform_set + 20.0 * scheme * unk


def work(case):
    if case["kind"] == "plan":
        N = _dims(case)
        elem = 8 if case["dtype"] == "f64" else 4
        return {"bytes": 2.0 * math.prod(N) * elem, "flops": case["steps"] * _step_flops(N, case["scheme"])}
    if case["kind"] == "batch":
        N, _ = _meshes(case)
        return {"bytes": 8.0 * sum(a * b for a, b in N),
                "flops": case["steps"] * sum(_step_flops(n, case["scheme"]) for n in N)}
    C, M, L, B, n = case["C"], case["M"], case["L"], case["batch"], case["N"] - 1
    nparam = sum(math.prod(s) for s in param_shapes(C, M, L).values())
    layer = B * C * (2 * (2.0 * n * n * M + 2.0 * n * M * M)) + 2.0 * B * C * C * (n * n + M * M)
    fwd = L * layer + B * n * n * (4.0 * C)
    if case["grad"]:
        return {"bytes": 8.0 * B * n * n + 8.0 * nparam, "flops": 3.0 * fwd}
    return {"bytes": 8.0 * B * n * n + 4.0 * nparam, "flops": fwd}


# ---------------------------------------------------------------- values in 64 bits

def _axis(n, h, bc):
    """Orthonormal eigenvectors and eigenvalues of the Q1 stiffness against the mass matrix of one axis."""
    j = torch.arange(0 if bc == "periodic" else 1, n, dtype=torch.float64, device="cuda")
    jk = torch.outer(j, j)
    if bc == "periodic":
        t = 2.0 * math.pi * torch.remainder(jk, n) / n
        S = (torch.cos(t) + torch.sin(t)) / math.sqrt(n)
        th = 2.0 * math.pi * j / n
    else:
        S = math.sqrt(2.0 / n) * torch.sin(math.pi * torch.remainder(jk, 2 * n) / n)
        th = math.pi * j / n
    return S, (12.0 / h ** 2) * torch.sin(0.5 * th) ** 2 / (2.0 + torch.cos(th))


def _phi(z):
    """phi_1(-z), phi_2(-z), z >= 0."""
    s = torch.where(z < 0.5, z, torch.zeros_like(z))
    s1, s2 = torch.zeros_like(z), torch.zeros_like(z)
    for m in range(22, -1, -1):
        s1 = 1.0 / math.factorial(m + 1) - s1 * s
        s2 = 1.0 / math.factorial(m + 2) - s2 * s
    zb = torch.where(z < 0.5, torch.ones_like(z), z)
    p1 = -torch.expm1(-zb) / zb
    p2 = (zb + torch.expm1(-zb)) / zb ** 2
    return torch.where(z < 0.5, s1, p1), torch.where(z < 0.5, s2, p2)


class _Exact:
    def __init__(self, N, D, tau, scheme, bc, reaction, source=None):
        ax = [_axis(n, 1.0 / n, bc) for n in N]
        self.S = [a[0] for a in ax]
        z = tau * D * ax[0][1]
        for a in ax[1:]:
            z = z + (tau * D * a[1]).reshape((-1,) + (1,) * z.dim())
        self.tau, self.scheme, self.f = tau, scheme, reaction
        p1, p2 = _phi(z)
        self.E, self.w1 = torch.exp(-z), tau * p1
        if scheme == 2:
            self.Ec, self.wc = torch.exp(-0.5 * z), 0.5 * tau * _phi(0.5 * z)[0]
            self.wa, self.wb = tau * (p1 - 2.0 * p2), 2.0 * tau * p2
        self.source = None
        if source is not None:
            amp, rate, gs = source
            g = torch.ones((), dtype=torch.float64, device="cuda")
            for v in reversed(gs):
                g = g.unsqueeze(-1) * torch.from_numpy(v).cuda()
            self.source = (amp, rate, g)

    def dst(self, u):
        u = u @ self.S[0]
        u = torch.matmul(self.S[1], u)
        if len(self.S) == 3:
            u = torch.matmul(self.S[2], u.reshape(u.shape[0], -1)).reshape(u.shape)
        return u

    def react(self, u, t):
        flin, fcub, flog = self.f
        r = u * (flin + fcub * u * u)
        if flog:
            r = r + flog * torch.atanh(u)
        if self.source is not None:
            amp, rate, g = self.source
            r = r + amp * math.exp(-rate * t) * g
        return r

    def run(self, u, steps):
        U = self.dst(u)
        for n in range(steps):
            t = n * self.tau
            N0 = self.dst(self.react(self.dst(U), t))
            if self.scheme == 1:
                U = self.E * U + self.w1 * N0
            else:
                N2 = self.dst(self.react(self.dst(self.Ec * U + self.wc * N0), t + 0.5 * self.tau))
                U = self.E * U + self.wa * N0 + self.wb * N2
        return self.dst(U)


def _bf(x):
    return x.float().bfloat16().double()


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _gelu_grad(z):
    return 0.5 * (1.0 + torch.erf(z / math.sqrt(2.0))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)


def _mix(W, h):
    """sum_c W[o, c] h[b, c, y, x]"""
    return torch.matmul(W, h.reshape(h.shape[0], h.shape[1], -1)).reshape(h.shape)


def _sno_exact(case, seed):
    P32, u, target, D = _sno_data(case, seed)
    P = {k: v.double() for k, v in P32.items()}
    u, target = u.double(), target.double()
    C, M, L, N = case["C"], case["M"], case["L"], case["N"]
    a = torch.tensor([(math.log(d) - math.log(1e-3)) / math.log(100.0) for d in D], dtype=torch.float64, device="cuda")
    p = torch.arange(1, M + 1, dtype=torch.float64, device="cuda")
    j = torch.arange(1, N, dtype=torch.float64, device="cuda")
    S = math.sqrt(2.0 / N) * torch.sin(math.pi * torch.remainder(torch.outer(p, j), 2 * N) / N)
    Sb = _bf(S)
    h = P["Wl"][:, 0, None, None] * u[:, None] + (P["Wl"][:, 1] * a[:, None])[..., None, None] + P["bl"][:, None, None]
    hs, zs, hhs = [h], [], []
    for l in range(L):
        hh = _bf(torch.matmul(S, torch.matmul(_bf(h), Sb.T)))
        gh = torch.einsum("pqoc,bcpq->bopq", _bf(P["Wm"][l]), hh)
        z = torch.matmul(Sb.T, _bf(torch.matmul(gh, S))) + _mix(_bf(P["Wp"][l]), _bf(h)) + P["bp"][l][:, None, None]
        h = _gelu(z)
        if case["grad"]:
            hs.append(h)
            zs.append(z)
            hhs.append(hh)
    out = u + torch.einsum("c,bcyx->byx", P["Wq"], h) + P["bq"]
    if not case["grad"]:
        return out
    loss = torch.mean((out - target) ** 2).item()
    du = 2.0 * (out - target) / out.numel()
    G = {"Wq": torch.einsum("byx,bcyx->c", du, hs[-1]), "bq": du.sum(), "Wm": torch.zeros_like(P["Wm"]),
         "Wp": torch.zeros_like(P["Wp"]), "bp": torch.zeros_like(P["bp"]), "Wl": torch.zeros_like(P["Wl"])}
    dh = P["Wq"][:, None, None] * du[:, None]
    for l in reversed(range(L)):
        dz = dh * _gelu_grad(zs[l])
        G["bp"][l] = dz.sum(dim=(0, 2, 3))
        G["Wp"][l] = torch.einsum("boi,bci->oc", dz.flatten(2), hs[l].flatten(2))
        dgh = torch.matmul(torch.matmul(S, dz), S.T)
        G["Wm"][l] = torch.einsum("bopq,bcpq->pqoc", dgh, hhs[l])
        dhh = torch.einsum("pqoc,bopq->bcpq", _bf(P["Wm"][l]), dgh)
        dh = _mix(P["Wp"][l].T, dz) + torch.matmul(S.T, torch.matmul(dhh, S))
    G["Wl"][:, 0] = torch.einsum("bcyx,byx->c", dh, u)
    G["Wl"][:, 1] = torch.einsum("bcyx,b->c", dh, a)
    G["bl"] = dh.sum(dim=(0, 2, 3))
    return [loss] + [G[k].cpu().numpy() for k in PARAM_NAMES]


def exact(case, seed):
    if case["kind"] == "plan":
        ex = _Exact(_dims(case), case["D"], case["tau"], case["scheme"], case["bc"], _reaction(case),
                    _source(case) if case["source"] else None)
        return ex.run(_field(case, seed).double(), case["steps"])
    if case["kind"] == "batch":
        N, D, flat = _batch_fields(case, seed)
        out = torch.empty(flat.shape, dtype=torch.float64, device="cuda")
        for n, d, v, o in zip(N, D, _views(flat, N), _views(out, N)):
            o.copy_(_Exact(n, d, case["tau"], case["scheme"], "dirichlet", (1.0, -1.0, 0.0)).run(v.double(), case["steps"]))
        return out
    return _sno_exact(case, seed)

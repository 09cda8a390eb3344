"""The pass plans chosen by axis length and number of pencils, and the fused operator layers, against the CPU oracle.

Tolerances: those of the other step tests, FP64 1e-12 and FP32 1e-5 in relative L2 and Linf over at most four steps (the
rounding of a step is a few hundred ulp at most: ~1e-13 and ~2e-6 times the number of steps' growth e^{tau L} ~ 1). The
operator's are those of the small operator (2e-4 of the increment, 2e-3 per gradient array), widened to 1e-3 and 5e-3 as at
its full size, for operands whose FP32 and FP64 values straddle a bf16 rounding boundary.
"""
import numpy as np
import pytest

from oracle import etd as oetd
from oracle import sno as osno
from paper_2209_11922_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5}
FH = dict(flin=1.6, fcub=0.0, flog=-0.8)


def _steps(N, scheme, bc, dtype, react, nsteps=3, seed=71, U=None, tau=2e-3, D=None):
    from paper_2209_11922_gb300.etd import Plan
    if D is None:   # the logarithm's argument stays inside (-1, 1) over these steps at 1e-4
        D = 1e-4 if react == "fh" else 1e-2
    if U is None:
        U = inputs.uniform_field(inputs.field_shape(N, bc), -0.9, 0.9, seed)
    if dtype == "f32":
        U = U.astype(np.float32).astype(np.float64)
    kw = FH if react == "fh" else {}
    ref = oetd.run(U, N, tuple(1.0 / n for n in N), D, tau, nsteps, scheme, bc=bc, **kw)
    with Plan(N, D, tau, scheme=scheme, dtype=dtype, bc=bc, **kw) as pl:
        d = torch.from_numpy(np.ascontiguousarray(U.astype(np.float32 if dtype == "f32" else np.float64))).cuda()
        pl.run(d, nsteps)
        got = d.cpu().numpy().astype(np.float64)
    l2, linf = np.linalg.norm(got - ref) / np.linalg.norm(ref), np.abs(got - ref).max() / np.abs(ref).max()
    assert l2 <= TOL[dtype] and linf <= TOL[dtype], (l2, linf)


# few pencils: dense products (FP64 up to 256), the many-thread plans (192 .. 512), whole axes in one CTA; many pencils: the
# plain plans; odd tiles (23, 47, 95 pencils) and lengths at each end of a plan's range
GRIDS = [(64, 64), (24, 192), (192, 24), (48, 256), (384, 32), (512, 48), (512, 512), (96, 768), (1024, 16), (1536, 12),
         (12, 2048), (128, 24, 8), (8, 48, 256), (64, 32, 96), (512, 8, 12)]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("N", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_plans_match_oracle(N, bc, dtype):
    react = "fh" if bc == "periodic" else "ac"   # the logarithmic reaction runs on periodic plans
    for scheme in (1, 2) if max(N) < 768 else (2,):
        _steps(N, scheme, bc, dtype, react)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_weights_over_the_range_of_zeta(bc, dtype):
    """tau D mu from 1e-9 (and 0, the periodic constant mode) to 1e4 in one field, 2D and 3D."""
    for N in ((64, 96), (32, 24, 64)):
        for tau_d in (1e-9, 1e-3, 1.0):
            _steps(N, 2, bc, dtype, "ac", nsteps=2, tau=1e-2, D=tau_d / 1e-2)
    if bc == "periodic":
        _steps((32, 16, 24), 2, bc, dtype, "ac", U=np.full((24, 16, 32), 0.3))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_logarithmic_reaction_near_its_poles(dtype):
    """|u| up to 1 - 1e-3 and down to 1e-7: artanh near its poles and its zero."""
    N = (32, 24, 16)
    u = inputs.uniform_field(inputs.field_shape(N, "periodic"), -1, 1, 5)
    U = np.sign(u) * np.where(np.abs(u) < 0.3, 1e-7 + 1e-3 * np.abs(u), 0.9 + 0.099 * np.abs(u))
    # f = -0.8 artanh u is 3.0 at the largest |u| and its slope 0.8 / (1 - u^2) is 400 there: with tau = 1e-4 a step
    # multiplies a rounding error by 1.04
    _steps(N, 2, "periodic", dtype, "fh", nsteps=2, U=U, tau=1e-4)


@pytest.mark.parametrize("C,M,N,B", [(16, 12, 32, 3), (16, 24, 96, 2), (32, 6, 24, 5), (32, 16, 48, 1), (32, 17, 64, 2)])
def test_operator_layers_match_oracle(C, M, N, B):
    from paper_2209_11922_gb300.sno import Sno
    w = inputs.SnoWorkload("layers", N=N, C=C, M=M, L=3, window=5, tau=1e-2)
    P = w.init_weights()
    P["bl"], P["bp"], P["bq"], P["Wq"] = P["bl"] + 0.05, P["bp"] - 0.02, np.array(0.01), P["Wq"] * 10
    f = lambda i0: np.stack([w.u0(i) for i in range(i0, i0 + B)]).astype(np.float32)
    u, D = f(0), [w.D(i) for i in range(B)]
    tgt = (u + 0.1 * f(10)).astype(np.float32)
    OP = osno.Params(*[np.asarray(P[n], dtype=np.float32).astype(np.float64) for n in osno.Params.NAMES])
    uh, cache = osno.forward(OP, u.astype(np.float64), D, w.N)
    g_ref = osno.backward(OP, cache, uh, tgt.astype(np.float64), w.N)
    s = Sno(N, C, M, 3, B + 1)
    s.set_params(P)
    rel = lambda a, b: float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))
    got = s.forward(torch.from_numpy(u).cuda(), D).cpu().numpy()
    assert rel(got - u, uh - u) <= 1e-3
    loss, g = s.gradient(torch.from_numpy(u).cuda(), D, torch.from_numpy(tgt).cuda())
    assert abs(loss - osno.loss(uh, tgt)) <= 1e-4 * osno.loss(uh, tgt)
    for n in osno.Params.NAMES:
        assert rel(g[n], getattr(g_ref, n)) <= 5e-3, n

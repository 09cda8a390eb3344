"""The kernels on both sides of the lines by number of pencils that the other plan tests do not reach: the plain two-step plans
of axes that take the many-thread, recurrence or dense kernels over few pencils, the tiles of 3 and 12 pairs, and the recurrence
at 96 and 1024. Against the CPU oracle, two ETDRK2 steps, with the step tests' tolerances (FP64 1e-12, FP32 1e-5)."""
import numpy as np
import pytest

from oracle import etd as oetd
from paper_2209_11922_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F64 = [
    (12, 768),                                          # y 768 in tiles of three pairs
    (24, 128, 256),                                     # y 128 in tiles of twelve pairs
    (24, 128, 384),                                     # y in twelve, z 384 in three
    (64, 96, 128), (48, 128, 192), (192, 48, 64),       # 48 to 192, along x and strided
    (32, 128, 192), (128, 32, 192),                     # 32 along x and strided
    (1536, 24, 24), (24, 24, 1536), (2048, 24, 24), (24, 24, 2048),   # 1536 and 2048 over more than 256 pairs
    (96, 24, 96), (1024, 32), (32, 1024),               # the recurrence
]
F32 = [(192, 64, 64), (512, 64, 64), (64, 192, 64), (64, 64, 256), (64, 384, 64), (64, 64, 512), (256, 64, 64), (384, 64, 64)]
F32_PERIODIC = [(96, 64, 64), (192, 64, 64), (256, 64, 64), (384, 64, 64), (512, 64, 64), (64, 512, 64), (64, 64, 512)]


def _check(N, bc, dtype):
    from paper_2209_11922_gb300.etd import Plan
    U = inputs.uniform_field(inputs.field_shape(N, bc), -0.9, 0.9, 97)
    np_t = np.float32 if dtype == "f32" else np.float64
    U = U.astype(np_t).astype(np.float64)
    ref = oetd.run(U, N, tuple(1.0 / n for n in N), 1e-2, 2e-3, 2, 2, bc=bc)
    with Plan(N, 1e-2, 2e-3, scheme=2, dtype=dtype, bc=bc) as pl:
        d = torch.from_numpy(np.ascontiguousarray(U.astype(np_t))).cuda()
        pl.run(d, 2)
        got = d.cpu().numpy().astype(np.float64)
    tol = 1e-5 if dtype == "f32" else 1e-12
    l2, linf = np.linalg.norm(got - ref) / np.linalg.norm(ref), np.abs(got - ref).max() / np.abs(ref).max()
    assert l2 <= tol and linf <= tol, (l2, linf)


@pytest.mark.parametrize("N", F64, ids=lambda n: "x".join(map(str, n)))
def test_fp64_dirichlet(N):
    _check(N, "dirichlet", "f64")


@pytest.mark.parametrize("N", F32, ids=lambda n: "x".join(map(str, n)))
def test_fp32_dirichlet(N):
    _check(N, "dirichlet", "f32")


@pytest.mark.parametrize("N", F32_PERIODIC, ids=lambda n: "x".join(map(str, n)))
def test_fp32_periodic(N):
    _check(N, "periodic", "f32")


@pytest.mark.parametrize("N", [(64, 64), (1024, 1024), (96, 48), (32, 48, 64)], ids=lambda n: "x".join(map(str, n)))
def test_fft_routes_are_one_route_from_length_32(N):
    """ETD_ROUTE_FFT and ETD_ROUTE_FFT_HALF run AUTO's kernels on axes of 32 and more: the same bits, hence AUTO's 1e-5."""
    from paper_2209_11922_gb300.etd import Plan
    U = inputs.uniform_field(inputs.field_shape(N, "dirichlet"), -0.9, 0.9, 77).astype(np.float32)
    got = []
    for route in ("auto", "fft", "fft_half"):
        with Plan(N, 1e-3, 1e-2, scheme=2, dtype="f32", route=route) as pl:
            d = torch.from_numpy(np.ascontiguousarray(U)).cuda()
            pl.run(d, 5)
            got.append(d)
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])

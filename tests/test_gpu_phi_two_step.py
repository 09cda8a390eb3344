"""The phi-function weights as the two-step pass kernels evaluate them: their own device functions (fold_pass.cuh), compiled into
a small program, on zeta = zeta_x + zeta_y + zeta_z from per-axis values zeta_a and m_a = 1 - e^{-zeta_a} as a 3D plan's tables
hold them, against 50-digit values at the exact sum of the held zeta_a.

Bounds, in units u of half an ulp, to first order. m: 1 u per axis value; m + m' - m m' inherits at most the larger (the
weights (1 - m) m'/r and (1 - m') m/r add up to at most 1) and adds one rounding of the sum, at most 2 u of the result, where the inherited part vanishes, or
1 u, and one of the fused product: 3 u, for three axes 5. zeta: two sums, 2 u. 1/zeta: FP32 at most one ulp, 2 u. The product: 1 u. phi_1:
10 u. phi_2 = (1 - phi_1)/zeta at zeta >= 1, where phi_1 <= 0.63 and 1 - phi_1 >= 0.36: 10 u * 0.63 / 0.36 + 1 + 2 + 2 + 1 = 24 u;
below 1 the series, whose alternating terms shrink by 3 and more: 4 u. c2 phi_1(-c2 zeta) as phi_1, with
1 - e^{-c2 zeta_a} in place of m_a. FP64: the same sums."""
import ctypes
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_2209_11922_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

getcontext().prec = 50
C2 = 0.5
SRC = r"""
#include "fold_pass.cuh"
using namespace etd;
// two modes per thread: in [z(3) m(3) mc(3)] per mode, out {phi_1, phi_2, c2 phi_1(c2)}
template <class T> __global__ void run(const T* in, T* out, int pairs, T c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pairs) return;
  const T *a = in + 18 * i, *b = a + 9;
  // the pair shares its y and z values, as two adjacent x modes do
  Cx<T> z{a[0], b[0]}, m{a[3], b[3]}, mc{a[6], b[6]};
  for (int d = 1; d < 3; ++d) {
    z = z + Cx<T>{a[d], a[d]};
    m = join_m(a[3 + d], m);
    mc = join_m(a[6 + d], mc);
  }
  const Cx<T> rz = rcp2(bounded_zeta(z)), p1 = phi1_pair(z, rz, m, T(1)), t1 = phi1_pair(z, rz, mc, c2);
  const Cx<T> p2 = phi2_pair<T>(bounded_zeta(z), rz, p1, __activemask());
  T* o = out + 6 * i;
  o[0] = p1.x; o[1] = p2.x; o[2] = t1.x;
  o[3] = p1.y; o[4] = p2.y; o[5] = t1.y;
}
template <class T> int go(const T* in, T* out, int pairs, T c2) {
  T *d = nullptr, *r = nullptr;
  int e = cudaMalloc(&d, 18 * sizeof(T) * pairs);
  if (!e) e = cudaMalloc(&r, 6 * sizeof(T) * pairs);
  if (!e) e = cudaMemcpy(d, in, 18 * sizeof(T) * pairs, cudaMemcpyHostToDevice);
  if (!e) {
    run<T><<<(pairs + 127) / 128, 128>>>(d, r, pairs, c2);
    e = cudaGetLastError();
  }
  if (!e) e = cudaMemcpy(out, r, 6 * sizeof(T) * pairs, cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(r);
  return e;
}
extern "C" int phi_f32(const float* in, float* out, int pairs) { return go<float>(in, out, pairs, 0.5f); }
extern "C" int phi_f64(const double* in, double* out, int pairs) { return go<double>(in, out, pairs, 0.5); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("phi")
    (d / "phi.cu").write_text(SRC)
    so = d / "libphi.so"
    subprocess.run([build.nvcc(), *build._flags(), "-shared", "-o", str(so), str(d / "phi.cu")], check=True, capture_output=True, text=True)
    return ctypes.CDLL(str(so))


def _exact(zs):
    Z = sum(Decimal(float(v)) for v in zs)
    if Z == 0:
        return 1.0, 0.5, C2
    e, c = (-Z).exp(), (-Decimal(C2) * Z).exp()
    return float((1 - e) / Z), float((e - 1 + Z) / (Z * Z)), float((1 - c) / Z)


def _grid():
    """zeta from 1e-8 to 1e3 (and 0) in pairs of x modes with one split over the axes, both sides of zeta = 1 and the ranges of
    the 3D workloads (3e-4 to 24) among them."""
    rng = np.random.default_rng(5)
    rows = [[(0.0, 0.0, 0.0), (1e-3, 0.0, 0.0)], [(0.0, 0.5, 0.5), (1e-7, 0.5, 0.5)], [(0.3, 0.3, 0.4), (0.3000001, 0.3, 0.4)]]
    for t in np.concatenate([np.logspace(-8, 3, 700), np.linspace(0.9, 1.1, 200), np.logspace(-3.5, 1.4, 600)]):
        f = rng.dirichlet([0.6, 0.6, 0.6])
        rows.append([tuple(t * f), (t * f[0] * rng.uniform(0.5, 2.0), t * f[1], t * f[2])])
    return np.array(rows)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_two_step_weights_match_closed_forms(lib, dtype):
    np_t = np.float32 if dtype == "f32" else np.float64
    z = _grid().astype(np_t)
    z64 = z.astype(np.float64)
    x = np.ascontiguousarray(np.concatenate([z, (-np.expm1(-z64)).astype(np_t), (-np.expm1(-C2 * z64)).astype(np_t)], axis=2))
    out = np.zeros((len(z), 2, 3), np_t)
    fn = lib.phi_f32 if dtype == "f32" else lib.phi_f64
    assert fn(x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), len(z)) == 0
    ref = np.array([[_exact(v) for v in p] for p in z64])
    u = np.finfo(np_t).eps / 2
    worst = (np.abs(out.astype(np.float64) - ref) / ref / u).reshape(-1, 3).max(axis=0)
    print(dtype, "worst, in half ulps:", worst)
    assert worst[0] <= 10 and worst[1] <= 24 and worst[2] <= 10, worst

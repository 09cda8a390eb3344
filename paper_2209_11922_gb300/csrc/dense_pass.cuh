// dense_pass.cuh - the axis passes of FP64 plans over few short pencils, by dense products.
//
// GB300 issues a warp's FP64 instruction over 64 cycles of one of an SM's four schedulers (0.5 lanes per cycle), so an FFT
// pass whose pencils are few is bound by the FP64 instructions of one thread (N = 64 on 4 threads: 1040 of them, 38 us
// for a REACT pass whatever else is idle). The dense product of a folded pencil needs N/2 multiply-adds per output, two to
// three times the FFT's work at N = 64, but one output per thread, or a part of one: the chain is N/(2 KS) instructions
// and every scheduler of the chip takes part.
//
//   Dirichlet: E_j = c_j + c_{N-j}, O_j = c_j - c_{N-j} (E_{N/2} = c_{N/2}); F_q = sum_j M[j][q] (q odd ? E_j : O_j),
//     M[j][q] = sqrt(2/N) sin(pi j q / N), j = 1..N/2.
//   Periodic:  E_j = x_j + x_{N-j} (E_0 = x_0, E_{N/2} = x_{N/2}), O_j = x_j - x_{N-j}; C_q = sum_j M[j][q] E_j for
//     q <= N/2, S_{N-q} = sum_j M[j][q] O_j for q > N/2, M = N^{-1/2} cos, sin; H_q = C_q + S_q, H_{N-q} = C_q - S_q.
// A CTA transforms W pencils (x axis: rows; strided: adjacent columns) with KS threads per output, each summing every
// KS-th j; the partial sums meet in shared memory. Reading M (L2-resident, [j][q], coalesced along q) hides under the
// multiply-adds.
#pragma once
#include "fold_pass.cuh"

namespace etd {

struct DenseArgs {
  PassArgs<double> a;   // a.tw: the matrix M [N/2 + 1][N]; a.P: pencils W per CTA; a.tiles_x: CTAs per row of tiles
  int N, KS, per;
};

// OP: ENTRY, EXIT, REACT, TRANSFORM_X (x axis), TRANSFORM, RK1S, S1S, S2S (strided).
template <int OP>
__global__ void __launch_bounds__(512) dense_kernel(const DenseArgs g) {
  constexpr bool XAX = OP == OP_ENTRY || OP == OP_EXIT || OP == OP_REACT || OP == OP_TRANSFORM_X;
  constexpr bool STAGE = OP == OP_RK1S || OP == OP_S1S || OP == OP_S2S;
  extern __shared__ __align__(16) unsigned char dsm[];
  const PassArgs<double>& A = g.a;
  const int N = g.N, KS = g.KS, W = A.P, NT = blockDim.x, tid = threadIdx.x, J = N / 2 + 1;
  const bool per = g.per != 0;
  double* c = reinterpret_cast<double*>(dsm);   // [W][N]
  double* eo = c + W * N;                        // [W][2][J]
  double* part = eo + W * 2 * J;                 // [KS - 1][W N]
  // thread -> (part ks, pencil w, output q)
  const int out = tid % (W * N), ks = tid / (W * N), w = out / N, q = out - w * N;

  int x0 = 0, o = 0;
  size_t rs = 0;
  long long base = 0;
  if constexpr (!XAX) {
    const int xt = blockIdx.x % A.tiles_x;
    o = blockIdx.x / A.tiles_x;
    x0 = xt * W;
    rs = A.axis == 1 ? (size_t)A.nx : (size_t)A.nx * A.ny;
    base = x0 + (A.axis == 1 ? (long long)o * A.nx * A.ny : (long long)o * A.nx);
    if (!per && o == 0 && A.ndim == 3) {   // boundary plane: stays zero
      count_step(A);
      return;
    }
  }
  const int row0 = blockIdx.x * W;          // x axis: first row (y + ny z)
  const int rows = A.ny * A.nz;
  // row factors of this thread's mode (constants): before the dependency wait
  [[maybe_unused]] double e = 0, ec = 0, zt = 0, m1 = 0, mc = 0, cf0 = 0, cf1 = 0;
  if constexpr (STAGE) {
    const int x = x0 + w;
    const int ax = A.axis;
    const double* gz = ax == 1 ? A.zeta[1] : A.zeta[2];
    const double* ge = ax == 1 ? A.ex[1] : A.ex[2];
    const double* gc = ax == 1 ? A.ec[1] : A.ec[2];
    const double* gm = ax == 1 ? A.em[1] : A.em[2];
    const double* gcm = ax == 1 ? A.cm[1] : A.cm[2];
    if (ks == 0) {
      double pe = A.ex[0][x], pc = A.ec[0][x], pz = A.zeta[0][x], pm = A.em[0][x], pcm = A.cm[0][x];
      if (ax == 2) {
        pe *= A.ex[1][o];
        pc *= A.ec[1][o];
        pz += A.zeta[1][o];
        pm = fma(-A.em[1][o], pm, pm + A.em[1][o]);
        pcm = fma(-A.cm[1][o], pcm, pcm + A.cm[1][o]);
      }
      e = pe * ge[q];
      ec = pc * gc[q];
      if (A.coef) {
        const size_t mode = (size_t)q * A.nx + x;
        cf0 = OP == OP_S1S ? A.coef[2 * mode] : A.coef[mode];
        if (OP == OP_S1S) cf1 = A.coef[2 * mode + 1];
      } else {
        // phi_1 = m / zeta, phi_2 = (1 - phi_1) / zeta or its series below 1 (see fold_pass.cuh); phi_1 -> 1, phi_2 -> 1/2
        zt = pz + gz[q];
        m1 = fma(-gm[q], pm, pm + gm[q]);
        mc = fma(-gcm[q], pcm, pcm + gcm[q]);
        const double z = fmin(fmax(zt, 1e-290), 1e290), rz = 1.0 / z;
        const double p1 = zt > 1e-290 ? m1 * rz : 1.0;
        double p2 = (1.0 - p1) * rz;
        if (zt < 1.0) p2 = phi2_series<double>(-zt);
        if (OP == OP_S1S) {
          cf0 = A.tau * (zt > 1e-290 ? mc * rz : A.c2);
          cf1 = A.tau * (p1 - p2 / A.c2);
        } else if (OP == OP_RK1S) {
          cf0 = A.tau * p1;
        } else {
          cf0 = A.tau * p2 / A.c2;
        }
      }
    }
  }
  griddep_wait();
  if (A.step_inc && blockIdx.x == 0 && tid == 0) atomicAdd(A.step_inc, 1ULL);

  const int cut = per ? 0 : 1;
  auto dense_row = [&](int r) -> long long {   // row r's index 0 in the user's dense field, -2: no row there
    const int z = r / A.ny, y = r - z * A.ny;
    if (r >= rows || y < cut || (A.ndim == 3 && z < cut)) return -2;
    return ((A.ndim == 3 ? (long long)(z - cut) * (A.ny - cut) : 0LL) + (y - cut)) * (A.nx - cut) - cut;
  };
  // ---- load W pencils
  for (int i = tid; i < W * N; i += NT) {
    double v = 0.0;
    if constexpr (XAX) {
      const int ww = i / N, x = i - ww * N, r = row0 + ww;
      if constexpr (OP == OP_ENTRY) {
        const long long d = dense_row(r);
        if (d > -2 && x >= cut) v = A.in0[d + x];
      } else {
        if (r < rows) v = A.in0[(size_t)r * A.nx + x];
      }
      c[i] = v;
    } else {   // consecutive threads on consecutive columns
      const int j = i / W, ww = i - j * W;
      const double* src = OP == OP_S1S || OP == OP_RK1S ? A.in1 : A.in0;
      c[ww * N + j] = src[base + ww + (size_t)j * rs];
    }
  }
  [[maybe_unused]] double u = 0.0;   // the stage pass's second operand at this thread's mode
  if constexpr (STAGE) {
    if (ks == 0) u = (OP == OP_S2S ? A.in1 : A.in0)[base + w + (size_t)q * rs];
  }
  __syncthreads();

  // one transform of the pencils in c; the result of (w, q) in the thread with ks = 0
  auto transform = [&]() -> double {
    for (int i = tid; i < W * J; i += NT) {
      const int ww = i / J, j = i - ww * J;
      const double* cw = c + ww * N;
      const double a = (j == 0 && !per) ? 0.0 : cw[j];
      const double b = j == 0 || j == N / 2 ? 0.0 : cw[N - j];
      eo[(ww * 2) * J + j] = a + b;
      eo[(ww * 2 + 1) * J + j] = j == 0 || j == N / 2 ? 0.0 : a - b;
    }
    __syncthreads();
    const bool odd = per ? q > N / 2 : (q & 1) == 0;   // which fold this output takes
    const double* v = eo + (w * 2 + (odd ? 1 : 0)) * J;
    const double* M = A.tw + q;
    double acc = 0.0;
#pragma unroll 8
    for (int j = ks; j < J; j += KS) acc = fma(M[(size_t)j * N], v[j], acc);
    if (ks > 0) part[(ks - 1) * W * N + out] = acc;
    if (KS > 1) {
      __syncthreads();
      if (ks == 0)
        for (int k = 1; k < KS; ++k) acc += part[(k - 1) * W * N + out];
    }
    if (per) {   // H_q = C_q + S_q, H_{N-q} = C_q - S_q
      __syncthreads();
      if (ks == 0) c[out] = acc;
      __syncthreads();
      if (ks == 0 && q != 0 && q != N / 2) {
        const double other = c[w * N + N - q];
        acc = q < N / 2 ? acc + other : other - acc;
      }
    }
    return !per && q == 0 ? 0.0 : acc;
  };
  double r = transform();
  if constexpr (OP == OP_REACT || STAGE) {
    if constexpr (OP == OP_REACT) {
      double f = r * (A.flin + A.fcub * r * r);
      if (A.flog != 0.0 && ks == 0) f += A.flog * atanh(r);
      r = f;
    } else if (ks == 0) {
      double r1;
      if constexpr (OP == OP_S1S) {
        r1 = e * u + cf1 * r;
        r = ec * u + cf0 * r;
      } else if constexpr (OP == OP_RK1S) {
        r = r1 = e * u + cf0 * r;
      } else {
        r = r1 = u + cf0 * r;
      }
      A.out1[base + w + (size_t)q * rs] = r1;
    }
    __syncthreads();
    if (ks == 0) c[out] = r;
    __syncthreads();
    r = transform();
  }
  griddep_launch_dependents();
  if (ks != 0) return;
  if constexpr (XAX) {
    const int rr = row0 + w;
    if (rr >= rows) return;
    if constexpr (OP == OP_EXIT) {
      const long long d = dense_row(rr);
      if (d > -2 && q >= cut) A.out0[d + q] = r;
    } else {
      if (OP == OP_REACT && A.src_gx) {
        const double t = *A.src_t0 + ((double)*A.step_ctr + A.src_c) * A.tau;
        const double ga = A.src_amp * exp(-A.src_rate * t) * A.src_gy[rr % A.ny] * (A.src_gz ? A.src_gz[rr / A.ny] : 1.0);
        r += ga * A.src_gx[q];
      }
      A.out0[(size_t)rr * A.nx + q] = r;
    }
  } else {
    A.out0[base + w + (size_t)q * rs] = r;
  }
}

inline size_t dense_smem_bytes(int N, int W, int KS) {
  return ((size_t)W * N + (size_t)W * 2 * (N / 2 + 1) + (size_t)(KS - 1) * W * N) * sizeof(double);
}

inline const void* find_dense_kernel(int op) {
  switch (op) {
    case OP_ENTRY: return reinterpret_cast<const void*>(&dense_kernel<OP_ENTRY>);
    case OP_EXIT: return reinterpret_cast<const void*>(&dense_kernel<OP_EXIT>);
    case OP_REACT: return reinterpret_cast<const void*>(&dense_kernel<OP_REACT>);
    case OP_TRANSFORM: return reinterpret_cast<const void*>(&dense_kernel<OP_TRANSFORM>);
    case OP_TRANSFORM_X: return reinterpret_cast<const void*>(&dense_kernel<OP_TRANSFORM_X>);
    case OP_RK1S: return reinterpret_cast<const void*>(&dense_kernel<OP_RK1S>);
    case OP_S1S: return reinterpret_cast<const void*>(&dense_kernel<OP_S1S>);
    case OP_S2S: return reinterpret_cast<const void*>(&dense_kernel<OP_S2S>);
  }
  return nullptr;
}

}  // namespace etd

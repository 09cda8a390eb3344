// sno_grad.cuh - kernels of the spectral neural operator's gradient (FP32, fields [b][c][y][x], C = 16 or 32 channels,
// M <= 24 modes). Every sum runs in the order of the general kernels (sno_kernels.cuh: serial fused multiply-adds over the
// contracted index, pixels in 16 pieces per field), so a gradient has the same bits by either route.
//
// Per layer, from the loss down:
//   grad_point_kernel    dz_l = (Wp^T dz_{l+1} + field) gelu'(z_l); at the top Wq du in place of the bracket, below layer 0
//                        without gelu'. One pass over four fields where a GEMM, an accumulating GEMM and a GELU pass ran.
//   grad_weight_kernel   dWp over one piece of one field
//   grad_modes_x_kernel  first contraction of the truncated transform of dz (along x)
//   grad_field_kernel    inverse truncated transform of the mode gradient, both contractions
#pragma once
#include "sno_layer.cuh"

namespace etd {
namespace sno {

struct GradPointArgs {
  int B;
  long long np;          // pixels per field
  const float* du;       // top: [B][np]
  const float* Wq;       // top: [C]
  const float* Wp;       // others: the layer above's mix [o][c]
  const float* dzin;     // others: [B][C][np]
  const float* field;    // others: spectral part [B][C][np]
  const float* z;        // [B][C][np]; out may be z itself (each element is read before it is written, by one thread)
  float* out;
};

enum { GRAD_TOP = 0, GRAD_LAYER = 1, GRAD_LIFT = 2 };

// One pixel per lane, four channels at a time in packed pairs, the weights broadcast from shared memory (one 16-byte read
// per two packed operations), the next channels' loads in flight: 262 us where memory alone (four fields of B C np floats, 32 of 255^2 x 32) takes 160;
// two pixels per lane at two CTAs per SM 313; as separate GEMM, accumulation and GELU passes about 900.
template <int C, int KIND>
__global__ void __launch_bounds__(256, 3) grad_point_kernel(const GradPointArgs g) {
  __shared__ __align__(16) float W[C * C];   // [o][c]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int i = tid; i < (KIND == GRAD_TOP ? C : C * C); i += 256) W[i] = KIND == GRAD_TOP ? g.Wq[i] : g.Wp[i];
  __syncthreads();
  const long long chunks = (g.np + 31) / 32, total = chunks * g.B;
  for (long long t = (long long)blockIdx.x * 8 + w; t < total; t += (long long)gridDim.x * 8) {
    const int b = (int)(t / chunks);
    long long p = (t - b * chunks) * 32 + lane;
    const bool on = p < g.np;
    if (!on) p = g.np - 1;
    long long e = (long long)b * C * g.np + p;
    float f[4], z[4];
    auto load = [&](long long q) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (KIND != GRAD_TOP) f[k] = g.field[q + k * g.np];
        if (KIND != GRAD_LIFT) z[k] = g.z[q + k * g.np];
      }
    };
    float d[KIND == GRAD_TOP ? 1 : C];
    if constexpr (KIND == GRAD_TOP) {
      d[0] = g.du[(long long)b * g.np + p];
    } else {
#pragma unroll
      for (int o = 0; o < C; ++o) d[o] = g.dzin[e + o * g.np];
    }
    load(e);
#pragma unroll 1
    for (int c0 = 0; c0 < C; c0 += 4) {
      float fc[4], zc[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        fc[k] = f[k];
        zc[k] = z[k];
      }
      if (c0 + 4 < C) load(e + 4 * g.np);
      float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
      for (int o = 0; o < (KIND == GRAD_TOP ? 1 : C); ++o) {
        const float4 r = *reinterpret_cast<const float4*>(W + o * C + c0);
        const float2 v = make_float2(d[o], d[o]);
        a0 = fma2f(make_float2(r.x, r.y), v, a0);
        a1 = fma2f(make_float2(r.z, r.w), v, a1);
      }
      float h[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (KIND != GRAD_TOP) h[k] += fc[k];
        if (KIND != GRAD_LIFT) h[k] *= gelu_grad(zc[k]);
        if (on) g.out[e + k * g.np] = h[k];
      }
      e += 4 * g.np;
    }
  }
}

// part[b][s][o][c] = sum over the pixels of piece s (kc of them, of field b) of dz[b][o][i] h[b][c][i], in order. One CTA per
// piece, 4 o x 2 c sums per thread; 32 pixels at a time through shared memory as [pixel][channel], the next ones' loads in
// flight. A warp loads 8 pixels x 4 channels (32-byte sectors; distinct banks on the transposed store). As a general GEMM
// with 2 x 2 sums per thread this took 1142 us for 32 fields of 255^2 and 32 channels, here 285; 4 x 4 sums on 64 threads 312 and dz stored
// twice for the packed operations 320: shared-memory reads and their latency bound it (memory alone: 80).
template <int C>
__global__ void __launch_bounds__(C * C / 8) grad_weight_kernel(const float* __restrict__ dz, const float* __restrict__ h, float* __restrict__ part,
                                                                long long np, int ks) {
  constexpr int T = C * C / 8, PX = 32, PITCH = 2 * C + 4, WARPS = T / 32;
  constexpr int RG = 2 * C / 4, PER = RG * (PX / 8) / WARPS;   // groups of 4 rows (C of dz, C of h) x 8 pixels, per warp
  __shared__ __align__(16) float sm[2][PX * PITCH];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int b = blockIdx.x / ks, sk = blockIdx.x % ks;
  const long long kc = ((np + ks - 1) / ks + 15) / 16 * 16, beg = sk * kc, end = beg + kc < np ? beg + kc : np;
  const float* A = dz + (long long)b * C * np;
  const float* H = h + (long long)b * C * np;
  const int lp = lane >> 2, lr = lane & 3;
  float v[PER];
  auto load = [&](long long p0) {
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int u = w * PER + k, row = (u / (PX / 8)) * 4 + lr;
      const long long p = p0 + (u % (PX / 8)) * 8 + lp;
      v[k] = p < end ? (row < C ? A[row * np + p] : H[(row - C) * np + p]) : 0.f;
    }
  };
  const int ob = 4 * (tid / (C / 2)), cb = 2 * (tid % (C / 2));
  float2 acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = make_float2(0.f, 0.f);
  if (beg < end) load(beg);
  int buf = 0;
  for (long long p0 = beg; p0 < end; p0 += PX, buf ^= 1) {
    float* s = sm[buf];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int u = w * PER + k;
      s[((u % (PX / 8)) * 8 + lp) * PITCH + (u / (PX / 8)) * 4 + lr] = v[k];
    }
    __syncthreads();   // one per 32 pixels: the buffer written next was last read before this barrier
    if (p0 + PX < end) load(p0 + PX);
#pragma unroll 8
    for (int i = 0; i < PX; ++i) {
      const float4 d = *reinterpret_cast<const float4*>(s + i * PITCH + ob);
      const float2 x = *reinterpret_cast<const float2*>(s + i * PITCH + C + cb);
      acc[0] = fma2f(make_float2(d.x, d.x), x, acc[0]);
      acc[1] = fma2f(make_float2(d.y, d.y), x, acc[1]);
      acc[2] = fma2f(make_float2(d.z, d.z), x, acc[2]);
      acc[3] = fma2f(make_float2(d.w, d.w), x, acc[3]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) *reinterpret_cast<float2*>(part + ((long long)blockIdx.x * C + ob + i) * C + cb) = acc[i];
}

// First contraction of the truncated transform: T[img][m][y] = sum_x X[img][y][x] S[m][x] (FP32, x in order). One CTA of 128
// threads per image, two rows y per thread, X staged in 32-column tiles (transposed reads on distinct banks), S as [x][MP]
// read as broadcasts, two modes per packed instruction: 175 us for 1024 images of 255^2 and 24 modes (general GEMM 227; memory 42:
// bound by the shared-memory reads, one broadcast of 16 bytes per four packed operations).
template <int MP>
__global__ void __launch_bounds__(128) grad_modes_x_kernel(const float* __restrict__ X, const float* __restrict__ S, float* __restrict__ T,
                                                           int n, int M) {
  __shared__ __align__(16) float ss[32][MP];
  __shared__ float xs[256][33];
  const int tid = threadIdx.x;
  const float* Xi = X + (size_t)blockIdx.x * n * n;
  for (int y0 = 0; y0 < n; y0 += 256) {
    float2 a0[MP / 2], a1[MP / 2];
#pragma unroll
    for (int i = 0; i < MP / 2; ++i) a0[i] = a1[i] = make_float2(0.f, 0.f);
    for (int x0 = 0; x0 < n; x0 += 32) {
      __syncthreads();
      {
        const int xx = tid & 31, yy = tid >> 5;
#pragma unroll 16
        for (int k = 0; k < 64; ++k) {
          const int y = yy + 4 * k;
          xs[y][xx] = y0 + y < n && x0 + xx < n ? Xi[(size_t)(y0 + y) * n + x0 + xx] : 0.f;
        }
        for (int i = tid; i < 32 * MP; i += 128) {
          const int m = i / 32, x = i % 32;
          ss[x][m] = m < M && x0 + x < n ? S[(size_t)m * n + x0 + x] : 0.f;
        }
      }
      __syncthreads();
#pragma unroll 4
      for (int x = 0; x < 32; ++x) {
        const float v0 = xs[tid][x], v1 = xs[tid + 128][x];
        const float4* s = reinterpret_cast<const float4*>(ss[x]);
#pragma unroll
        for (int q = 0; q < MP / 4; ++q) {
          const float4 f = s[q];
          a0[2 * q] = fma2f(make_float2(f.x, f.y), make_float2(v0, v0), a0[2 * q]);
          a0[2 * q + 1] = fma2f(make_float2(f.z, f.w), make_float2(v0, v0), a0[2 * q + 1]);
          a1[2 * q] = fma2f(make_float2(f.x, f.y), make_float2(v1, v1), a1[2 * q]);
          a1[2 * q + 1] = fma2f(make_float2(f.z, f.w), make_float2(v1, v1), a1[2 * q + 1]);
        }
      }
    }
    float* Ti = T + (size_t)blockIdx.x * M * n + y0 + tid;
#pragma unroll
    for (int i = 0; i < MP / 2; ++i) {
      if (2 * i < M) {
        if (y0 + tid < n) Ti[(size_t)(2 * i) * n] = a0[i].x;
        if (y0 + tid + 128 < n) Ti[(size_t)(2 * i) * n + 128] = a1[i].x;
      }
      if (2 * i + 1 < M) {
        if (y0 + tid < n) Ti[(size_t)(2 * i + 1) * n] = a0[i].y;
        if (y0 + tid + 128 < n) Ti[(size_t)(2 * i + 1) * n + 128] = a1[i].y;
      }
    }
  }
}

// Inverse truncated transform of an image's modes: out[y][x] = sum_p S[p][y] (sum_q Y[p][q] S[q][x]) (FP32). One CTA of 256
// threads per image and 256 columns; a thread forms its column's 24 inner sums, then 32 rows y at a time in packed pairs,
// S as [p][y] read as broadcasts: 189 us for 1024 images of 255^2 and 24 modes, 520 as two GEMM launches (memory 40; bound by
// the packed operations and their broadcast reads).
template <int MP>
__global__ void __launch_bounds__(256, 2) grad_field_kernel(const float* __restrict__ Y, const float* __restrict__ S, float* __restrict__ out,
                                                            int n, int M) {
  extern __shared__ __align__(16) float gsm[];
  const int np = (n + 31) / 32 * 32;
  float* sp = gsm;             // [MP][np]
  float* ys = gsm + MP * np;   // [MP][MP]
  const int tid = threadIdx.x;
  for (int i = tid; i < MP * np; i += 256) {
    const int p = i / np, y = i - p * np;
    sp[i] = p < M && y < n ? S[(size_t)p * n + y] : 0.f;
  }
  const float* Yi = Y + (size_t)blockIdx.x * M * M;
  for (int i = tid; i < MP * MP; i += 256) {
    const int p = i / MP, q = i - p * MP;
    ys[i] = p < M && q < M ? Yi[p * M + q] : 0.f;
  }
  __syncthreads();
  for (int x = tid; x < n; x += 256) {
    float s[MP], v[MP];
#pragma unroll
    for (int q = 0; q < MP; ++q) s[q] = q < M ? S[(size_t)q * n + x] : 0.f;
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      const float4* r = reinterpret_cast<const float4*>(ys + p * MP);
      float a = 0.f;
#pragma unroll
      for (int q = 0; q < MP / 4; ++q) {
        const float4 f = r[q];
        a = fmaf(f.x, s[4 * q], a);
        a = fmaf(f.y, s[4 * q + 1], a);
        a = fmaf(f.z, s[4 * q + 2], a);
        a = fmaf(f.w, s[4 * q + 3], a);
      }
      v[p] = a;
    }
    float* o = out + (size_t)blockIdx.x * n * n + x;
#pragma unroll 1
    for (int y0 = 0; y0 < n; y0 += 32) {
      float2 acc[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        const float4* r = reinterpret_cast<const float4*>(sp + p * np + y0);
        const float2 vv = make_float2(v[p], v[p]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 f = r[i];
          acc[2 * i] = fma2f(make_float2(f.x, f.y), vv, acc[2 * i]);
          acc[2 * i + 1] = fma2f(make_float2(f.z, f.w), vv, acc[2 * i + 1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (y0 + 2 * i < n) o[(size_t)(y0 + 2 * i) * n] = acc[i].x;
        if (y0 + 2 * i + 1 < n) o[(size_t)(y0 + 2 * i + 1) * n] = acc[i].y;
      }
    }
  }
}

}  // namespace sno
}  // namespace etd

// sno_layer.cuh - fused inference layers of the spectral neural operator (channels last).
//
// One layer (Section "operator" of sno_kernels.cuh) reads h_l once and writes h_{l+1} once: the inverse truncated
// transform's second contraction, the pointwise channel mix, bias and GELU, and the next layer's first contraction
// run on the same registers. What bounds it is the traffic of h (B C n^2 floats, 0.53 GB at 64 fields of 255^2 and 32
// channels); unfused, a layer moved 3.2 GB (h read twice, z written and read twice, h' written).
//
// Layout h[b][y][x][c]: a pixel's channels are one 64- or 128-byte line. Fragments (mma.m16n8k16, bf16 operands, FP32
// accumulators; rows g = lane/4 and g + 8, columns 2t, 2t+1 with t = lane%4):
//   inverse transform at one x:  D[y][o] += sum_p bf(S[p][y]) bf(Tf[o][p][x])   A: S (constant), B: Tf[x][o][p]
//   channel mix at one x:        D[y][o] += sum_c bf(h[y][x][c]) bf(Wp[o][c])   A: the tile of h, B: Wp (constant)
// accumulate into the same fragment, so z needs no exchange; the warp-level instruction is used because its fragment
// layout makes these two contractions (and the pointwise epilogue) share registers, where tcgen05's tile of 128 rows
// by whole accumulators in tensor memory would need both products materialised; at 2-10 flops per byte the tensor
// rate does not matter. h' goes through a bf16 tile in shared memory to the next layer's first contraction
//   T[y][c][m] = sum_x bf(h'[y][x][c]) bf(S[m][x])                              A: the tile transposed, B: S
// whose accumulators a warp keeps for its 2 rows y over the whole loop along x. The operands rounded to bf16, and the
// FP32 ones, are those of the unfused kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstring>
#include <vector>

#include "sno_kernels.cuh"

namespace etd {
namespace sno {

__device__ __forceinline__ uint32_t bf2(float lo, float hi) {   // two bf16, round to nearest even; lo in the low half
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the same with the accumulator's initial value in other registers: columns c0, c1 of every row
__device__ __forceinline__ void mma16816_init(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, float c0, float c1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
}

union F2 {
  float2 f;
  unsigned long long u;
};
__device__ __forceinline__ float2 fma2f(float2 a, float2 b, float2 c) {
  F2 x, y, z, r;
  x.f = a;
  y.f = b;
  z.f = c;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(x.u), "l"(y.u), "l"(z.u));
  return r.f;
}
// gelu(z) = z/2 (1 + erf(z/sqrt2)) = max(z, 0) - (|z|/2) erfc(|z|/sqrt2) with
// erfc(t/sqrt2) = 2^{-q(t)}, q(t)/t a degree-9 polynomial fitted on [0, 6.5] (minimax in the error of the result; beyond,
// q keeps growing and the term vanishes). Over N(0, 2^2) and [-9, 9] its error against 64 bits is 3.6e-8 and 4.9e-8 rms,
// 2.4e-7 at most; z/2 (1 + erff(z/sqrt2)) in FP32 gives 5.1e-8, 6.7e-8 and 4.9e-7.
// (Scalar instructions: packed ones cost more register moves around the MMA fragments than they saved.)
// SAFE: gelu(+inf) = +inf, as in the training forward; without, NaN (the vanishing term is inf * 0). The last layer, whose
// values the projection adds up, takes it; in the others, whose infinities the next transform turns into NaN all over the field
// either way, the one instruction more was 1.8 % of a forward pass (1356 -> 1380 us at 64 fields of 255^2 and 32 channels).
template <bool SAFE> __device__ __forceinline__ float gelu_erfc(float z) {
  const float t = fabsf(SAFE ? fminf(z, 3.4028235e38f) : z);
  float p = 2.7615620012966247e-08f;
  p = fmaf(p, t, -8.48519789542479e-07f);
  p = fmaf(p, t, 1.105071078200126e-05f);
  p = fmaf(p, t, -7.781414751661941e-05f);
  p = fmaf(p, t, 0.00028622374520637095f);
  p = fmaf(p, t, -1.5051219634187873e-05f);
  p = fmaf(p, t, -0.0069295442663133144f);
  p = fmaf(p, t, 0.052432045340538025f);
  p = fmaf(p, t, 0.4592224359512329f);
  p = fmaf(p, t, 1.151104211807251f);
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(p * -t));
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(z));
  return fmaf(-0.5f * t, e, r);
}
template <bool SAFE> __device__ __forceinline__ void gelu4(float2 (&z)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) z[k] = make_float2(gelu_erfc<SAFE>(z[k].x), gelu_erfc<SAFE>(z[k].y));
}

struct LayerArgs {
  int B, n, M;
  const float* u;       // [B][n][n]
  const float* a;       // [B] input feature
  const float* Wl;      // lift weights [C][2], bias [C]
  const float* bl;
  const float* S;       // S_M [M][n]
  const uint2* Sf;      // S_M as fragments (s_fragments)
  const float* h;       // [B][n][n][C] (not read by the first layer: the lift of u)
  float* hn;            // [B][n][n][C] (not written by the last layer)
  const float* Tf;      // [B][n x][C / 8][MP / 8][32 lanes][2]: the inverse transform's first contraction, as fragments
  float* T;             // [B][n y][C][MP]: the next layer's first contraction (NULL output for the last)
  const float* Wp;      // [C][C]
  const float* bp;      // [C]
  const float* Wq;      // [C], bias: projection (last layer)
  const float* bq;
  float* out;           // [B][n][n] (last layer)
};

constexpr int LY = 16, LX = 8;   // rows y per CTA, columns x per step

// Row pitches of the shared-memory tiles, so that a fragment's accesses hit distinct banks.
template <int C> __host__ __device__ constexpr int layer_row_bytes() { return LX * C * 4 + 64; }   // staged row of h
template <int C> __host__ __device__ constexpr int tile_x_bytes() { return C * 2 + 16; }            // bf16 tile: one x
template <int C> __host__ __device__ constexpr int tile_y_bytes() { return 2 * LX * tile_x_bytes<C>() + 32; }
// Channel of column n of the fragments' 8-column block j: a thread's columns 2t, 2t + 1 of blocks 2i, 2i + 1 are then the
// four consecutive channels 16 i + 4 t .., loaded and stored as 16 bytes.
__host__ __device__ constexpr int frag_ch(int j, int n) { return 16 * (j >> 1) + 4 * (n >> 1) + 2 * (j & 1) + (n & 1); }
template <int C, bool FIRST> __host__ __device__ constexpr size_t layer_h_bytes() {
  return FIRST ? (size_t)LY * (LX + 1) * 4 : (size_t)LY * layer_row_bytes<C>();
}
template <int C, int MP> __host__ __device__ constexpr size_t layer_t_bytes() { return (size_t)LX * C * MP * 4; }
template <int C, int MP, bool FIRST, bool LAST> size_t layer_smem() {
  return 2 * layer_h_bytes<C, FIRST>() + 2 * layer_t_bytes<C, MP>() + (LAST ? 0 : (size_t)LY * tile_y_bytes<C>());
}

// S_M as B fragments of the contraction along x: for 16 columns x0 and 8 modes 8 j, lane (g, t) holds bf16 pairs
// S[8j + g][x0 + 2t ..] and S[8j + g][x0 + 8 + 2t ..]; zero outside M x n. [x0 / 16][MP / 8][32] (built on the host).
inline uint32_t bf16_bits(float f) {   // round to nearest even
  uint32_t b;
  memcpy(&b, &f, 4);
  return (b + 0x7FFFu + ((b >> 16) & 1u)) >> 16;
}
inline std::vector<uint2> s_fragments(const std::vector<float>& S, int M, int MP, int n) {
  std::vector<uint2> f;
  for (int x0 = 0; x0 < n; x0 += 16)
    for (int j = 0; j < MP / 8; ++j)
      for (int lane = 0; lane < 32; ++lane) {
        auto at = [&](int x) -> uint32_t {
          const int m = 8 * j + (lane >> 2);
          return m < M && x < n ? bf16_bits(S[(size_t)m * n + x]) : 0u;
        };
        const int x = x0 + 2 * (lane & 3);
        f.push_back(make_uint2(at(x) | at(x + 1) << 16, at(x + 8) | at(x + 9) << 16));
      }
  return f;
}

// First contraction of the first layer, straight from u: T[b][y][c][m] = sum_x bf(h0[c]) bf(S[m][x]),
// h0[c] = Wl[c][0] u + (Wl[c][1] a + bl[c]). One warp per row y, a CTA looping over groups of 8 rows.
template <int C, int MP>
__global__ void __launch_bounds__(256) lift_modes_kernel(const LayerArgs g) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gr = lane >> 2, t = lane & 3;
  const int n = g.n, b = blockIdx.y;
  const float af = g.a[b];
  float w0[C / 8], of[C / 8];
#pragma unroll
  for (int i = 0; i < C / 8; ++i) {
    const int c = 8 * i + gr;
    w0[i] = g.Wl[2 * c];
    of[i] = g.Wl[2 * c + 1] * af + g.bl[c];
  }
  for (int y = blockIdx.x * 8 + w; y < n; y += 8 * gridDim.x) {
  const float* u = g.u + ((size_t)b * n + y) * n;
  float acc[C / 16][MP / 8][4] = {};
#pragma unroll 2
  for (int x0 = 0; x0 < n; x0 += 16) {
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int x = x0 + 2 * t + (e & 1) + 8 * (e >> 1);
      v[e] = x < n ? u[x] : 0.f;
    }
    uint2 bS[MP / 8];
#pragma unroll
    for (int j = 0; j < MP / 8; ++j) bS[j] = g.Sf[((x0 >> 4) * (MP / 8) + j) * 32 + lane];
#pragma unroll
    for (int i = 0; i < C / 16; ++i) {
      uint32_t a[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {   // register e: row half e & 1, k half e >> 1
        const int hc = 2 * i + (e & 1);
        a[e] = bf2(w0[hc] * v[2 * (e >> 1)] + of[hc], w0[hc] * v[2 * (e >> 1) + 1] + of[hc]);
      }
#pragma unroll
      for (int j = 0; j < MP / 8; ++j) mma16816(acc[i][j], a, bS[j].x, bS[j].y);
    }
  }
  float* T = g.T + ((size_t)b * n + y) * C * MP;
#pragma unroll
  for (int i = 0; i < C / 16; ++i)
#pragma unroll
    for (int j = 0; j < MP / 8; ++j) {
      *reinterpret_cast<float2*>(T + (16 * i + gr) * MP + 8 * j + 2 * t) = make_float2(acc[i][j][0], acc[i][j][1]);
      *reinterpret_cast<float2*>(T + (16 * i + gr + 8) * MP + 8 * j + 2 * t) = make_float2(acc[i][j][2], acc[i][j][3]);
    }
  }
}

// One layer: CTA = 16 rows y of one field, 8 warps, steps of 8 columns x; warp w handles column w of the step for all
// 16 rows, and after every second step rows 2w, 2w + 1 of the contraction along x. The tiles of h (from HBM) and Tf (from
// L2) arrive by cp.async one step ahead in two stages; what hides the rest of their latency is the second CTA of the SM.
// 251 us for an inner layer of 64 fields of 255^2 and 32 channels (0.67 of the copy bandwidth), 256 for the first, which
// reads only u: the instruction stream (GELU, conversions, fragment moves) bounds both.
template <int C, int MP, bool FIRST, bool LAST>
__global__ void __launch_bounds__(256, 2) layer_kernel(const LayerArgs g) {
  constexpr int NJ = C / 8, KC = C / 16, KS = (MP + 15) / 16, MJ = MP / 8, NT = 256;
  constexpr int ROWB = layer_row_bytes<C>(), TX = tile_x_bytes<C>(), TY = tile_y_bytes<C>();
  constexpr unsigned HB = (unsigned)layer_h_bytes<C, FIRST>(), TB = (unsigned)layer_t_bytes<C, MP>();
  extern __shared__ __align__(16) unsigned char lsm[];
  unsigned char* stage = lsm;                                  // [2] tiles of h (first layer: of u), [2] of Tf
  unsigned char* tile = lsm + 2 * HB + 2 * TB;                 // bf16 h' [y][16 x][c]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gr = lane >> 2, t = lane & 3;
  const int n = g.n, b = blockIdx.y, y0 = blockIdx.x * LY;
  const int ny = min(LY, n - y0), steps = (n + 2 * LX - 1) / (2 * LX) * 2;

  // this thread's share of a stage: rows tid / CH + k NT / CH of the tile of h, 16-byte chunk tid % CH of them; chunks
  // tid + k NT of Tf
  constexpr int CH = LX * C / 4, HR = NT / CH, TC = LX * C * MP / 4;
  const int hy = FIRST ? tid / LX : tid / CH, hq = FIRST ? tid % LX : tid % CH;
  const float* hsrc = FIRST ? g.u + ((size_t)b * n + y0 + hy) * n + hq : g.h + ((size_t)b * n + y0 + hy) * n * C + hq * 4;
  const unsigned hdst = (unsigned)__cvta_generic_to_shared(stage) + (FIRST ? (hy * (LX + 1) + hq) * 4 : hy * ROWB + hq * 16);
  const float* tsrc = g.Tf + (size_t)b * n * C * MP + tid * 4;
  const unsigned tdst = (unsigned)__cvta_generic_to_shared(stage) + 2 * HB + tid * 16;
  auto load_h = [&](int step, unsigned so) {
    const int nx = min(LX, n - step * LX);   // <= 0 past the row: nothing to load
    if constexpr (FIRST) {
      if (tid < LY * LX && hy < ny && hq < nx)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(hdst + so), "l"(hsrc + step * LX) : "memory");
    } else {
      const float* src = hsrc + (size_t)step * (LX * C);
#pragma unroll
      for (int k = 0; k < LY / HR; ++k)
        if (hy + k * HR < ny && hq < nx * (C / 4))
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(hdst + so + k * HR * ROWB),
                       "l"(src + (size_t)(k * HR) * n * C) : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  auto load_t = [&](int step) {
    const int nx = min(LX, n - step * LX);
    const float* tf = tsrc + (size_t)step * (LX * C * MP);
#pragma unroll
    for (int k = 0; k < (TC + NT - 1) / NT; ++k)
      if (tid + k * NT < nx * (C * MP / 4))
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tdst + (step & 1) * TB + k * NT * 16), "l"(tf + k * NT * 4)
                     : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  load_h(0, 0);
  load_t(0);

  // constant operands
  uint32_t aS[KS][4];   // S^T: rows y, columns p
#pragma unroll
  for (int ks = 0; ks < KS; ++ks)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int y = y0 + gr + 8 * (e & 1), p = 16 * ks + 2 * t + 8 * (e >> 1);
      const float s0 = y < n && p < g.M ? g.S[(size_t)p * n + y] : 0.f;
      const float s1 = y < n && p + 1 < g.M ? g.S[(size_t)(p + 1) * n + y] : 0.f;
      aS[ks][e] = bf2(s0, s1);
    }
  uint32_t bW[NJ][KC][2];   // Wp: columns o, rows c (row 2t + 8 e + r: channel 16 kc + 4 t + 2 e + r)
  float bias[NJ][2];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
#pragma unroll
    for (int kc = 0; kc < KC; ++kc)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float* p = g.Wp + frag_ch(j, gr) * C + 16 * kc + 4 * t + 2 * e;
        bW[j][kc][e] = bf2(p[0], p[1]);
      }
    bias[j][0] = g.bp[frag_ch(j, 2 * t)];
    bias[j][1] = g.bp[frag_ch(j, 2 * t + 1)];
  }
  float lw[FIRST ? 4 * KC : 1], lo[FIRST ? 4 * KC : 1];   // lift of the channels this thread feeds
  if constexpr (FIRST) {
    const float af = g.a[b];
#pragma unroll
    for (int i = 0; i < 4 * KC; ++i) {
      const int c = 16 * (i >> 2) + 4 * t + (i & 3);
      lw[i] = g.Wl[2 * c];
      lo[i] = g.Wl[2 * c + 1] * af + g.bl[c];
    }
  }
  float wq[LAST ? NJ : 1][2];
  float bqv = 0.f;
  if constexpr (LAST) {
    bqv = g.bq[0];
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      wq[j][0] = g.Wq[frag_ch(j, 2 * t)];
      wq[j][1] = g.Wq[frag_ch(j, 2 * t + 1)];
    }
  }
  float accF[LAST ? 1 : 2][LAST ? 1 : KC][LAST ? 1 : MJ][4] = {};
  const int xl = w, ya = gr, yb = ya + 8;

  const bool vya = y0 + ya < n, vyb = y0 + yb < n;
  [[maybe_unused]] float* oa = g.hn + (((size_t)b * n + y0 + ya) * n + xl) * C + 4 * t;
  [[maybe_unused]] float* ob = oa + 8 * (size_t)n * C;
  [[maybe_unused]] const uint2* sf = g.Sf + lane;
  // transposed 8 x 8 matrices (rows x, columns c): lanes 8i .. 8i + 7 address matrix i = (k half, row half)
  [[maybe_unused]] const unsigned tl = (unsigned)__cvta_generic_to_shared(tile) + 2 * w * TY + ((lane & 7) + 8 * (lane >> 4)) * TX +
                                       16 * ((lane >> 3) & 1);

#pragma unroll 1
  for (int step0 = 0; step0 < steps; step0 += 2) {
#pragma unroll
  for (int odd = 0; odd < 2; ++odd) {
    const int step = step0 + odd, x = step * LX + xl;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // the tiles of this step are there; those of the last step (and before even steps the bf16 tile) are free
    load_t(step + 1);
    load_h(step + 1, (1 - odd) * HB);
    const unsigned char* d = stage + odd * HB;
    const unsigned char* dt = stage + 2 * HB + odd * TB;
    float acc[NJ][4];
    {
      const float2* tf = reinterpret_cast<const float2*>(dt) + xl * (C * MP / 2) + lane;
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        uint32_t bT[2 * KS];
#pragma unroll
        for (int e = 0; e < 2 * KS; ++e) {
          bT[e] = 0u;
          if (8 * e < MP) {
            const float2 v = tf[(j * MJ + e) * 32];
            bT[e] = bf2(v.x, v.y);
          }
        }
        mma16816_init(acc[j], aS[0], bT[0], bT[1], bias[j][0], bias[j][1]);
#pragma unroll
        for (int ks = 1; ks < KS; ++ks) mma16816(acc[j], aS[ks], bT[2 * ks], bT[2 * ks + 1]);
      }
    }
    [[maybe_unused]] float ua = 0.f, ub = 0.f;
    if constexpr (FIRST) {
      ua = reinterpret_cast<const float*>(d)[ya * (LX + 1) + xl];
      ub = reinterpret_cast<const float*>(d)[yb * (LX + 1) + xl];
    }
#pragma unroll
    for (int kc = 0; kc < KC; ++kc) {
      uint32_t a[4];
      if constexpr (FIRST) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {   // register e: row half e & 1, k half e >> 1
          const float v = (e & 1) ? ub : ua;
          const int i = 4 * kc + 2 * (e >> 1);
          a[e] = bf2(lw[i] * v + lo[i], lw[i + 1] * v + lo[i + 1]);
        }
      } else {
        const float4 va = *reinterpret_cast<const float4*>(d + ya * ROWB + (xl * C + 16 * kc + 4 * t) * 4);
        const float4 vb = *reinterpret_cast<const float4*>(d + yb * ROWB + (xl * C + 16 * kc + 4 * t) * 4);
        a[0] = bf2(va.x, va.y);
        a[1] = bf2(vb.x, vb.y);
        a[2] = bf2(va.z, va.w);
        a[3] = bf2(vb.z, vb.w);
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) mma16816(acc[j], a, bW[j][kc][0], bW[j][kc][1]);
    }
    const bool va = x < n && vya, vb = x < n && vyb;
    if constexpr (LAST) {
      float sa = 0.f, sb = 0.f;
#pragma unroll
      for (int i = 0; i < NJ / 2; ++i) {
        float2 z[4] = {make_float2(acc[2 * i][0], acc[2 * i][1]), make_float2(acc[2 * i + 1][0], acc[2 * i + 1][1]),
                       make_float2(acc[2 * i][2], acc[2 * i][3]), make_float2(acc[2 * i + 1][2], acc[2 * i + 1][3])};
        gelu4<LAST>(z);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          sa = fmaf(wq[2 * i + h][1], z[h].y, fmaf(wq[2 * i + h][0], z[h].x, sa));
          sb = fmaf(wq[2 * i + h][1], z[2 + h].y, fmaf(wq[2 * i + h][0], z[2 + h].x, sb));
        }
      }
#pragma unroll
      for (int m = 1; m < 4; m <<= 1) {
        sa += __shfl_xor_sync(0xffffffffu, sa, m);
        sb += __shfl_xor_sync(0xffffffffu, sb, m);
      }
      if (t == 0) {
        const size_t ia = ((size_t)b * n + y0 + ya) * n + x, ib = ia + 8 * (size_t)n;
        if (va) g.out[ia] = sa + (g.u[ia] + bqv);
        if (vb) g.out[ib] = sb + (g.u[ib] + bqv);
      }
    } else {
      unsigned char* ta = tile + ya * TY + (odd * LX + xl) * TX + 8 * t;
#pragma unroll
      for (int i = 0; i < NJ / 2; ++i) {
        float2 z[4] = {make_float2(acc[2 * i][0], acc[2 * i][1]), make_float2(acc[2 * i + 1][0], acc[2 * i + 1][1]),
                       make_float2(acc[2 * i][2], acc[2 * i][3]), make_float2(acc[2 * i + 1][2], acc[2 * i + 1][3])};
        gelu4<LAST>(z);
        if (va) *reinterpret_cast<float4*>(oa + odd * LX * C + 16 * i) = make_float4(z[0].x, z[0].y, z[1].x, z[1].y);
        if (vb) *reinterpret_cast<float4*>(ob + odd * LX * C + 16 * i) = make_float4(z[2].x, z[2].y, z[3].x, z[3].y);
        *reinterpret_cast<uint2*>(ta + 32 * i) = va ? make_uint2(bf2(z[0].x, z[0].y), bf2(z[1].x, z[1].y)) : make_uint2(0u, 0u);
        *reinterpret_cast<uint2*>(ta + 8 * TY + 32 * i) = vb ? make_uint2(bf2(z[2].x, z[2].y), bf2(z[3].x, z[3].y)) : make_uint2(0u, 0u);
      }
    }
  }
  if constexpr (!LAST) {
    oa += 2 * LX * C;
    ob += 2 * LX * C;
    __syncthreads();
    uint2 bS[MJ];
#pragma unroll
    for (int j = 0; j < MJ; ++j) bS[j] = sf[j * 32];
    sf += MJ * 32;
#pragma unroll
    for (int yy = 0; yy < 2; ++yy)
#pragma unroll
      for (int i = 0; i < KC; ++i) {
        uint32_t a[4];
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(tl + yy * TY + 32 * i) : "memory");
#pragma unroll
        for (int j = 0; j < MJ; ++j) mma16816(accF[yy][i][j], a, bS[j].x, bS[j].y);
      }
  }
  }
  if constexpr (!LAST) {
#pragma unroll
    for (int yy = 0; yy < 2; ++yy) {
      const int y = y0 + 2 * w + yy;
      if (y >= n) continue;
      float* T = g.T + ((size_t)b * n + y) * C * MP;
#pragma unroll
      for (int i = 0; i < KC; ++i)
#pragma unroll
        for (int j = 0; j < MJ; ++j) {
          *reinterpret_cast<float2*>(T + (16 * i + gr) * MP + 8 * j + 2 * t) = make_float2(accF[yy][i][j][0], accF[yy][i][j][1]);
          *reinterpret_cast<float2*>(T + (16 * i + gr + 8) * MP + 8 * j + 2 * t) = make_float2(accF[yy][i][j][2], accF[yy][i][j][3]);
        }
    }
  }
}

// Second contraction of the truncated transform: hh[p M + q][b][c] = bf(sum_y S[p][y] T[b][y][c][q]) in FP32. One thread
// per (c, q) column and half of the rows y (its loads coalesce; the halves add up in shared memory), S in shared memory
// as [y][MP], read as broadcasts, two p per packed instruction, the next U rows' loads in flight.
template <int MP>
__global__ void __launch_bounds__(256) modes_y_kernel(const float* __restrict__ S, const float* __restrict__ T, float* __restrict__ hh,
                                                      int B, int n, int M, int C) {
  extern __shared__ __align__(16) float lsy[];
  for (int p = threadIdx.x / 32; p < MP; p += 8)
    for (int y = threadIdx.x % 32; y < n; y += 32) lsy[y * MP + p] = p < M ? S[(size_t)p * n + y] : 0.f;
  __syncthreads();
  const int half = threadIdx.x >> 7, ct = threadIdx.x & 127;
  const int b = blockIdx.y, col = blockIdx.x * 128 + ct;
  const bool on = col < C * MP;
  const int ybeg = half ? (n + 1) / 2 : 0, yend = half ? n : (n + 1) / 2;
  const float* Tb = T + (size_t)b * n * C * MP + (on ? col : 0);
  const size_t st = (size_t)C * MP;
  float2 acc[MP / 2];
#pragma unroll
  for (int i = 0; i < MP / 2; ++i) acc[i] = make_float2(0.f, 0.f);
  constexpr int U = 8;
  float v[U], vn[U];
#pragma unroll
  for (int k = 0; k < U; ++k) v[k] = ybeg + k < yend ? Tb[(ybeg + k) * st] : 0.f;
  for (int y0 = ybeg; y0 < yend; y0 += U) {
#pragma unroll
    for (int k = 0; k < U; ++k) vn[k] = y0 + U + k < yend ? Tb[(y0 + U + k) * st] : 0.f;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (y0 + k >= yend) break;
      const float4* s = reinterpret_cast<const float4*>(lsy + (y0 + k) * MP);
      const float2 vv = make_float2(v[k], v[k]);
#pragma unroll
      for (int q = 0; q < MP / 4; ++q) {
        const float4 f = s[q];
        acc[2 * q] = fma2f(make_float2(f.x, f.y), vv, acc[2 * q]);
        acc[2 * q + 1] = fma2f(make_float2(f.z, f.w), vv, acc[2 * q + 1]);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) v[k] = vn[k];
  }
  __syncthreads();   // S is no longer read: its space takes the second half's sums
  float2* part = reinterpret_cast<float2*>(lsy);
  if (half)
#pragma unroll
    for (int i = 0; i < MP / 2; ++i) part[i * 128 + ct] = acc[i];
  __syncthreads();
  const int c = col / MP, q = col - c * MP;
  if (half || !on || q >= M) return;
#pragma unroll
  for (int i = 0; i < MP / 2; ++i) {
    const float2 o = part[i * 128 + ct];
    if (2 * i < M) hh[((size_t)(2 * i * M + q) * B + b) * C + c] = bf16_round(acc[i].x + o.x);
    if (2 * i + 1 < M) hh[((size_t)((2 * i + 1) * M + q) * B + b) * C + c] = bf16_round(acc[i].y + o.y);
  }
}
constexpr size_t modes_y_smem(int n, int MP) { return (size_t)(n * MP > 128 * MP ? n * MP : 128 * MP) * sizeof(float); }

// Per-mode channel mix: gh[mode][b][o] = sum_c bf(Wm[mode][o][c]) hh[mode][b][c] (FP32, channels in order). One CTA per
// mode, o = tid % C.
template <int C>
__global__ void __launch_bounds__(256) mode_mix_kernel(const float* __restrict__ Wm, const float* __restrict__ hh,
                                                       float* __restrict__ gh, int B) {
  __shared__ float W[C][C + 1];
  __shared__ float hs[64 * C];   // 64 fields at a time
  const float* w = Wm + (size_t)blockIdx.x * C * C;
  for (int i = threadIdx.x; i < C * C; i += 256) W[i / C][i % C] = bf16_round(w[i]);
  __syncthreads();
  const int o = threadIdx.x % C;
  float wr[C];
#pragma unroll
  for (int c = 0; c < C; ++c) wr[c] = W[o][c];
  for (int b0 = 0; b0 < B; b0 += 64) {
    const int nb = min(64, B - b0);
    const size_t base = ((size_t)blockIdx.x * B + b0) * C;
    for (int i = threadIdx.x; i < nb * C; i += 256) hs[i] = hh[base + i];
    __syncthreads();
    for (int b = threadIdx.x / C; b < nb; b += 256 / C) {
      float acc = 0.f;
#pragma unroll
      for (int c = 0; c < C; ++c) acc = fmaf(hs[b * C + c], wr[c], acc);
      gh[base + (size_t)b * C + o] = acc;
    }
    __syncthreads();
  }
}

// First contraction of the inverse transform: Tf[b][x](o, p) = sum_q gh[p M + q][b][o] S[q][x] (FP32, q in order), 0 for
// p >= M, in the order of the layer kernel's fragments. One thread per (o, p) column, 64 values of x per CTA, four x per round in two packed accumulators, S in shared
// memory as [q][x], read as broadcasts.
template <int MP>
__global__ void __launch_bounds__(256) modes_x_kernel(const float* __restrict__ S, const float* __restrict__ gh, float* __restrict__ Tf,
                                                      int B, int n, int M, int C) {
  __shared__ __align__(16) float sx[MP][64];
  const int x0 = blockIdx.z * 64, nx = min(64, n - x0);
  for (int q = threadIdx.x / 64; q < MP; q += 4) {
    const int x = threadIdx.x % 64;
    sx[q][x] = q < M && x < nx ? S[(size_t)q * n + x0 + x] : 0.f;
  }
  __syncthreads();
  const int b = blockIdx.y, col = blockIdx.x * 256 + threadIdx.x;
  if (col >= C * MP) return;
  // column in fragment order: block j, p group e, lane (row of the block's columns, pair of p)
  const int lane = (col >> 1) & 31, je = col >> 6, j = je / (MP / 8);
  const int o = frag_ch(j, lane >> 2), p = 8 * (je - j * (MP / 8)) + 2 * (lane & 3) + (col & 1);
  float v[MP];
#pragma unroll
  for (int q = 0; q < MP; ++q) v[q] = p < M && q < M ? gh[((size_t)(p * M + q) * B + b) * C + o] : 0.f;
  float* out = Tf + ((size_t)b * n + x0) * C * MP + col;
  const size_t st = (size_t)C * MP;
  for (int x = 0; x < nx; x += 4) {
    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      const float4 f = *reinterpret_cast<const float4*>(&sx[q][x]);
      const float2 vv = make_float2(v[q], v[q]);
      a0 = fma2f(vv, make_float2(f.x, f.y), a0);
      a1 = fma2f(vv, make_float2(f.z, f.w), a1);
    }
    out[x * st] = a0.x;
    if (x + 1 < nx) out[(x + 1) * st] = a0.y;
    if (x + 2 < nx) out[(x + 2) * st] = a1.x;
    if (x + 3 < nx) out[(x + 3) * st] = a1.y;
  }
}

}  // namespace sno
}  // namespace etd

// fold_dst.cuh - orthonormal DST-I by a folded odd extension: the transform of the Dirichlet axes.
//
// As in dst_engine.cuh two real pencils are packed as one complex sequence c_j (j = 1..N-1) and the DST-I is
// read off the odd extension of length M = 2N: F_k = -i sc Z_k, Z = DFT_M (kernel exp(+2 pi i j k / M)),
// sc = sqrt(2/N)/2. Only the half of that DFT which the symmetry leaves is computed. With M = R L:
//
//   A   butterfly jj (radix R) reads the extension at jj + r L. Butterfly L - jj holds the same values
//       reversed and negated, so its outputs are -w_R^{-k} X_{-k} of butterfly jj's outputs X_k: the
//       butterflies jj = 0..L/2 suffice. jj reads c at r L + jj and r L + L - jj (r < R/2): every value once.
//       With tau_k = -i sc w_M^{jj k} the sub-sequences of the second step are
//         y_k[jj] = tau_k X_k,  y_k[L-jj] = conj(tau_k) X_{R-k}      (1 <= k < R/2).
//   B   the DFT of length L of y_k gives F at R m + k (m < L/2) and, negated, at R m + R - k: unit k and unit
//       R - k are the same numbers, so k < R/2 suffices.
//   Unit 0 stands for k = 0 and k = R/2 together, whose outputs are F at the multiples of R/2: the DST-I of
//   length L of the folded sequence d_jj = (X_0 + X_{R/2})/2, d_{L-jj} = (X_{R/2} - X_0)/2. It is computed by
//   a DFT of the same length L (the half-length recurrence of dst_engine.cuh: y_jj = sin(pi jj/L) X_{R/2} +
//   X_0/2, y_{L-jj} = sin(pi jj/L) X_{R/2} - X_0/2, even outputs as differences, odd ones as running sums of
//   at most L/2 = 16 terms held by one thread), or for L >= 64 by this scheme itself (R' = 2 UT, L' = L/UT below).
//   Butterflies 0 and L/2 (self-symmetric, half the data each) share one radix-R DFT: C = X^{(0)} + X^{(L/2)},
//   from which y_k[0] = (-i sc/2)(C_k - C_{-k}) - (sc/2) cot(pi k/R)(C_k + C_{-k}) and
//   y_k[L/2] = sc/(2 sin(pi k/R)) (C_k + C_{-k}).
//
// The transform is symmetric, so the transposed graph (B^T then A^T, the same DFTs and twiddles) is the same
// transform. A pass that transforms, works pointwise and transforms back runs A B | pointwise | B^T A^T: the
// thread that holds F at R m + k, R m + R - k after B holds what B^T starts from, and nothing is exchanged
// between them. Both steps are in place: A leaves y_k[jj], y_k[L-jj] in the R slots it read (slot k L + j).
//
// What it replaces, per complex value of a transform: the odd extension (radix passes over 2N points) made
// 11 shared-memory accesses and the recurrence 7; here a lone transform makes 2 (A and B sit in registers at
// both ends where the axis is strided) and the arithmetic is that of a length-N FFT.
#pragma once
#include <type_traits>

#include "dst_engine.cuh"

namespace etd {

// Plans: radix R, sub-length L (R L = 2N), threads per pencil pair, values per thread at most R or L.
// L <= 32: step B is one register DFT per unit. L = 64, 128: units of UT = 8 threads, L/8 values each (L/8 x 8);
// L = 256: units of 16 threads (16 x 16).
// G: one padding slot every G positions (G divides L, so slot offsets are compile-time constants).
template <class T, int N, bool MANY = false> struct FoldPlan { static constexpr int R = 0, L = 0, TPP = 1, G = 1; };
#define ETD_FOLD(NN, R_, L_, TPP_, G_)                                             \
  template <class T> struct FoldPlan<T, NN, false> {                               \
    static_assert(R_ * L_ == 2 * NN, "R L = 2N");                                  \
    static constexpr int R = R_, L = L_, TPP = TPP_, G = G_;                       \
  };
ETD_FOLD(32, 8, 8, 4, 4)
ETD_FOLD(48, 12, 8, 4, 4)
ETD_FOLD(64, 16, 8, 4, 4)
ETD_FOLD(96, 24, 8, 4, 4)
ETD_FOLD(128, 16, 16, 8, 16)
ETD_FOLD(192, 24, 16, 8, 16)
ETD_FOLD(256, 32, 16, 8, 16)
ETD_FOLD(384, 24, 32, 16, 16)
ETD_FOLD(512, 32, 32, 16, 16)
ETD_FOLD(768, 12, 128, 64, 8)
ETD_FOLD(1024, 16, 128, 64, 8)
ETD_FOLD(1536, 24, 128, 64, 8)
ETD_FOLD(2048, 16, 256, 128, 16)
#undef ETD_FOLD
// FP64, 192..512: GB300 issues a warp's FP64 instruction over 64 cycles of one of the SM's four schedulers, whatever
// lanes it has, so a pass over few pencils costs its longest thread: fewer values per thread and more threads
// (L = 64: eight values) than FP32 (256^2 ETDRK2 326 -> 158 us per step against R = 32, L = 16). Shorter axes keep
// the plans that leave no lane idle in step B (64^3: 233 us; R = 8, L = 16 idles half of them there, 350 us).
#define ETD_FOLD64(NN, R_, L_, TPP_, G_)                                           \
  template <> struct FoldPlan<double, NN, false> {                                 \
    static_assert(R_ * L_ == 2 * NN, "R L = 2N");                                  \
    static constexpr int R = R_, L = L_, TPP = TPP_, G = G_;                       \
  };
// MANY: FP32 plans over few pencils, the same many-threads form (an FP32 pass over few pencils costs its longest chain).
#define ETD_FOLDM(NN, R_, L_, TPP_, G_)                                            \
  template <> struct FoldPlan<float, NN, true> {                                   \
    static_assert(R_ * L_ == 2 * NN, "R L = 2N");                                  \
    static constexpr int R = R_, L = L_, TPP = TPP_, G = G_;                       \
  };
ETD_FOLDM(192, 6, 64, 32, 8)
ETD_FOLDM(256, 8, 64, 32, 8)
ETD_FOLDM(384, 12, 64, 32, 8)
ETD_FOLDM(512, 16, 64, 32, 8)
#undef ETD_FOLDM
ETD_FOLD64(192, 6, 64, 32, 8)
ETD_FOLD64(256, 8, 64, 32, 8)
ETD_FOLD64(384, 12, 64, 32, 8)
ETD_FOLD64(512, 16, 64, 32, 8)
ETD_FOLD64(2048, 32, 128, 64, 8)   // R = 16, L = 256 on 128 threads: 2048 x 1024 ETDRK2 1016 us per step against 891
#undef ETD_FOLD64

constexpr bool foldm_has(int n) { return n == 192 || n == 256 || n == 384 || n == 512; }   // FP32
constexpr bool fold_has(int n) {
  return n == 32 || n == 48 || n == 64 || n == 96 || n == 128 || n == 192 || n == 256 || n == 384 || n == 512 ||
         n == 768 || n == 1024 || n == 1536 || n == 2048;
}

constexpr unsigned long long FOLD_MAX_STRIDE = 2048ULL * 2048ULL;   // largest row stride: the z axis behind two axes of 2048

template <class T> __device__ __forceinline__ Cx<T> cmulc(Cx<T> a, Cx<T> b) {   // conj(a) b
  return {a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x};
}

// Radix-R step A of one unit: a[r] = c at r L + jj, b[r] = c at r L + L - jj (unit 0: r L + L/2), r < H = R/2;
// on return a[k] = y_k[jj], b[k] = y_k[L-jj] (unit 0: y_k[L/2]). tw is the axis's table, [k][jj] with row
// length TS: entry (k >= 1, jj >= 1) tau_k, entry (0, jj) (sc sin(pi jj/L), sc/2), entry (k, 0)
// (sc/2 cot(pi k/R), sc/(2 sin(pi k/R))), entry (0, 0) (0, sc). REC: unit 0 of step B takes the recurrence's
// input, else the folded sequence d.
template <class T, int R, bool REC, int TS>
__device__ __forceinline__ void fold_a(Cx<T> (&a)[R / 2], Cx<T> (&b)[R / 2], int jj, const Cx<T>* __restrict__ tw) {
  constexpr int H = R / 2;
  Cx<T> x[R];
  if (jj == 0) {
    a[0] = Cx<T>{T(0), T(0)};   // the boundary position
#pragma unroll
    for (int r = 0; r < H; ++r) {
      x[r] = a[r] + b[r];
      x[R - 1 - r] = r + 1 < H ? b[r] + a[r + 1 < H ? r + 1 : 0] : b[r];   // negated: second half
    }
  } else {
#pragma unroll
    for (int r = 0; r < H; ++r) {
      x[r] = a[r];
      x[R - 1 - r] = b[r];   // negated: second half
    }
  }
  Dft<T, R, true, false>::run(x);
  if (jj == 0) {
    const T sc = tw[0].y, hsc = T(0.5) * sc;
    a[0] = Cx<T>{T(0), T(0)};
    b[0] = REC ? sc * x[H] : T(0.5) * x[H];
#pragma unroll
    for (int k = 1; k < H; ++k) {
      const Cx<T> w = tw[k * TS], s = x[k] + x[R - k], d = x[k] - x[R - k];
      a[k] = Cx<T>{hsc * d.y - w.x * s.x, -hsc * d.x - w.x * s.y};
      b[k] = w.y * s;
    }
  } else {
    if constexpr (REC) {
      const Cx<T> w = tw[jj];
      const Cx<T> p = w.x * x[H], q = w.y * x[0];
      a[0] = p + q;
      b[0] = p - q;
    } else {
      a[0] = T(0.5) * (x[H] + x[0]);
      b[0] = T(0.5) * (x[H] - x[0]);
    }
#pragma unroll
    for (int k = 1; k < H; ++k) {
      const Cx<T> w = tw[k * TS + jj];
      a[k] = cmul(w, x[k]);
      b[k] = cmulc(w, x[R - k]);
    }
  }
}

// Transpose of fold_a.
template <class T, int R, bool REC, int TS>
__device__ __forceinline__ void fold_at(Cx<T> (&a)[R / 2], Cx<T> (&b)[R / 2], int jj, const Cx<T>* __restrict__ tw) {
  constexpr int H = R / 2;
  Cx<T> x[R];
  if (jj == 0) {
    const T sc = tw[0].y, hsc = T(0.5) * sc;
    x[0] = Cx<T>{T(0), T(0)};
    x[H] = REC ? sc * b[0] : T(0.5) * b[0];
#pragma unroll
    for (int k = 1; k < H; ++k) {
      const Cx<T> w = tw[k * TS];
      const Cx<T> q = Cx<T>{w.y * b[k].x - w.x * a[k].x, w.y * b[k].y - w.x * a[k].y};
      const Cx<T> g = Cx<T>{hsc * a[k].y, -hsc * a[k].x};   // (-i sc/2) a
      x[k] = q + g;
      x[R - k] = q - g;
    }
  } else {
    if constexpr (REC) {
      const Cx<T> w = tw[jj];
      x[H] = w.x * (a[0] + b[0]);
      x[0] = w.y * (a[0] - b[0]);
    } else {
      x[H] = T(0.5) * (a[0] + b[0]);
      x[0] = T(0.5) * (a[0] - b[0]);
    }
#pragma unroll
    for (int k = 1; k < H; ++k) {
      const Cx<T> w = tw[k * TS + jj];
      x[k] = cmul(w, a[k]);
      x[R - k] = cmulc(w, b[k]);
    }
  }
  Dft<T, R, false, true>::run(x);   // second half negated
  if (jj == 0) {
#pragma unroll
    for (int r = 0; r < H; ++r) {
      a[r] = r == 0 ? Cx<T>{T(0), T(0)} : x[r] + x[(R - r) % R];
      b[r] = x[r] + x[R - 1 - r];
    }
  } else {
#pragma unroll
    for (int r = 0; r < H; ++r) {
      a[r] = x[r];
      b[r] = x[R - 1 - r];
    }
  }
}

// Step B of one unit, L <= 32 values in registers: z[j] = y_k[j] in; out z[m] = F at R m + k and z[L/2 + m] =
// F at R m + R - k (special: at R m and R m + R/2), m < L/2.
template <class T, int L>
__device__ __forceinline__ void fold_b(Cx<T> (&z)[L], bool special) {
  constexpr int H = L / 2;
  Dft<T, L, false, true>::run(z);   // second half negated
  Cx<T> v2[H];
  if (special) {
    Cx<T> acc = z[0];
    v2[0] = acc;
    z[0] = Cx<T>{T(0), T(0)};
#pragma unroll
    for (int m = 1; m < H; ++m) {
      const Cx<T> u = z[m], w = z[L - m];   // w negated
      acc = acc + (u - w);
      v2[m] = acc;
      z[m] = Cx<T>{u.y + w.y, -u.x - w.x};   // -i (Z_m - Z_{L-m})
    }
  } else {
#pragma unroll
    for (int m = 0; m < H; ++m) v2[m] = z[L - 1 - m];
  }
#pragma unroll
  for (int m = 0; m < H; ++m) z[H + m] = v2[m];
}
// Transpose of fold_b.
template <class T, int L>
__device__ __forceinline__ void fold_bt(Cx<T> (&z)[L], bool special) {
  constexpr int H = L / 2;
  Cx<T> y[L];
  if (special) {
    Cx<T> s{T(0), T(0)};
    y[H] = s;
#pragma unroll
    for (int q = H - 1; q >= 1; --q) {
      s = s + z[H + q];
      y[q] = sub_i(s, z[q]);
      y[L - q] = Cx<T>{z[q].y - s.x, -s.y - z[q].x};   // -(s + i z): second half negated
    }
    y[0] = s + z[H];
  } else {
#pragma unroll
    for (int m = 0; m < H; ++m) {
      y[m] = z[m];
      y[L - 1 - m] = z[H + m];   // negated: second half
    }
  }
  Dft<T, L, true, false>::run(y);
#pragma unroll
  for (int j = 0; j < L; ++j) z[j] = y[j];
}

// Geometry and the two steps of one axis transform for a thread (pair buffer bp, thread l of the pair).
template <class T, int N, bool MANY = false> struct Fold {
  using Plan = FoldPlan<T, N, MANY>;
  using C = Cx<T>;
  static constexpr int R = Plan::R, L = Plan::L, TPP = Plan::TPP, G = Plan::G;
  static constexpr int H = R / 2;                       // units of step B
  static constexpr int UA = L / 2;                      // units of step A
  static constexpr bool BIG = L >= 64;                  // step B across UT threads per unit
  static constexpr int UT = L == 256 ? 16 : 8;
  static constexpr int QA = (UA + TPP - 1) / TPP;       // A units per thread
  static constexpr int SLOTS = BIG ? UT * H : H;         // thread slots of step B
  static constexpr int QB = (SLOTS + TPP - 1) / TPP;    // B slots per thread
  static constexpr int VB = BIG ? L / UT : L;               // values per B slot
  static constexpr int LP = N + N / G;                  // complex slots per pair
  static constexpr int UI = BIG ? VB / 2 : 1;           // A units of unit 0's inner transform (R' = 2 UT, L' = VB)
  // tables: A twiddles [H][UA]; BIG: exp(2 pi i t i / L) [VB][UT], then unit 0's A twiddles [UT][UI]
  static constexpr int TW_A = H * UA, TW_B = BIG ? UT * VB : 0, TW_S = BIG ? UT * UI : 0;
  static constexpr int TWN = TW_A + TW_B + TW_S;
  static_assert(L % G == 0, "padding group divides L");
  static __device__ __forceinline__ int at(int j) { return j + j / G; }
  static constexpr int LS = L + L / G;                  // slots from position j to j + L

  static __device__ __forceinline__ bool a_on(int jj) { return UA % TPP == 0 || jj < UA; }
  static __device__ __forceinline__ bool b_on(int s) { return SLOTS % TPP == 0 || s < SLOTS; }
  static constexpr __host__ __device__ __forceinline__ int partner(int jj) { return jj == 0 ? L / 2 : L - jj; }
  // Rows of step A's inputs: a[r] at jj + r L, b[r] at partner_row(jj) + (PARTNER_STEPS + r) L, where the multiples of L are
  // the same for every thread.
  static constexpr int PARTNER_STEPS = 0;
  static constexpr __host__ __device__ __forceinline__ int partner_row(int jj) { return partner(jj); }

  static __device__ __forceinline__ void a(C (&va)[H], C (&vb)[H], int jj, const C* __restrict__ tw) {
    fold_a<T, R, !BIG, UA>(va, vb, jj, tw);
  }
  static __device__ __forceinline__ void at_(C (&va)[H], C (&vb)[H], int jj, const C* __restrict__ tw) {
    fold_at<T, R, !BIG, UA>(va, vb, jj, tw);
  }
  static __device__ __forceinline__ void a_get(const C* __restrict__ bp, int jj, C (&va)[H], C (&vb)[H]) {
    const C* pa = bp + at(jj);
    const C* pb = bp + at(partner(jj));
#pragma unroll
    for (int r = 0; r < H; ++r) {
      va[r] = pa[r * LS];
      vb[r] = pb[r * LS];
    }
  }
  static __device__ __forceinline__ void a_put(C* __restrict__ bp, int jj, const C (&va)[H], const C (&vb)[H]) {
    C* pa = bp + at(jj);
    C* pb = bp + at(partner(jj));
#pragma unroll
    for (int r = 0; r < H; ++r) {
      pa[r * LS] = va[r];
      pb[r * LS] = vb[r];
    }
  }

  // Rows (output positions) of the values of B slot s: value i < HV at row1(s) + i STEP, value HV + i at
  // row2(s) + i STEP.
  static constexpr int HV = VB / 2, STEP = BIG ? UT * R : R;
  static constexpr __host__ __device__ __forceinline__ int row1(int s) {
    if constexpr (!BIG) return s;
    const int k = s / UT, t = s % UT;
    return k == 0 ? H * t : R * t + k;
  }
  static constexpr __host__ __device__ __forceinline__ int row2(int s) {
    if constexpr (!BIG) return s == 0 ? H : R - s;
    const int k = s / UT, t = s % UT;
    return k == 0 ? H * (t == 0 ? UT : 2 * UT - t) : R * (UT - 1 - t) + R - k;   // unit 0: the inner transform's rows
  }

  // The slots b_end reads and bt_begin writes for value i: own_base(s) + own_off(i).
  static __device__ __forceinline__ int own_base(int s) {
    if constexpr (!BIG) return s * LS;
    else return (s / UT) == 0 ? at(VB * (s % UT)) : (s / UT) * LS + at(UT * (s % UT));
  }
  static __device__ __forceinline__ int own_off(int s, int i) {
    if constexpr (!BIG) return i + i / G;
    else return (s / UT) == 0 ? i + i / G : (i % UT) + (i / UT) * (UT * UT + UT * UT / G);
  }

  // Step B: slot s of the pair, values to registers in the order of row1 / row2. The BIG form has an exchange
  // inside its unit: mid() is the part before it.
  static __device__ __forceinline__ void b_mid(C* __restrict__ bp, int s, const C* __restrict__ tw) {
    if constexpr (BIG) {
      const int k = s / UT, t = s % UT;
      if (k == 0) {
        if (t < UI) {
          C va[UT], vb[UT];
          const int part = t == 0 ? VB / 2 : VB - t;
#pragma unroll
          for (int r = 0; r < UT; ++r) {
            va[r] = bp[at(VB * r + t)];
            vb[r] = bp[at(VB * r + part)];
          }
          fold_a<T, 2 * UT, true, UI>(va, vb, t, tw + TW_A + TW_B);
#pragma unroll
          for (int r = 0; r < UT; ++r) {
            bp[at(VB * r + t)] = va[r];
            bp[at(VB * r + part)] = vb[r];
          }
        }
      } else {
        C* p = bp + k * LS + at(t);
        C x[VB];
#pragma unroll
        for (int i = 0; i < VB; ++i) x[i] = p[i * (UT + UT / G)];
        Dft<T, VB>::run(x);
        const C* w = tw + TW_A + t;
#pragma unroll
        for (int i = 0; i < VB; ++i) p[i * (UT + UT / G)] = i == 0 ? x[0] : cmul(w[UT * i], x[i]);
      }
    }
  }
  static __device__ __forceinline__ void b_end(const C* __restrict__ bp, int s, C (&z)[VB], const C* __restrict__) {
    if constexpr (!BIG) {
      const C* p = bp + s * LS;
#pragma unroll
      for (int j = 0; j < L; ++j) z[j] = p[j + j / G];
      fold_b<T, L>(z, s == 0);
    } else {
      const int k = s / UT, t = s % UT;
      if (k == 0) {
        const C* p = bp + at(VB * t);
#pragma unroll
        for (int j = 0; j < VB; ++j) z[j] = p[j + j / G];
        fold_b<T, VB>(z, t == 0);
      } else {
#pragma unroll
        for (int h = 0; h < VB / UT; ++h) {
          const C* p = bp + k * LS + at(UT * (t + UT * h));
          C x[UT];
#pragma unroll
          for (int j = 0; j < UT; ++j) x[j] = p[j];
          Dft<T, UT, false, true>::run(x);   // Z_m, m = t + UT h + VB q; rows R m + k, and R (L - 1 - m) + R - k negated
#pragma unroll
          for (int q = 0; q < UT / 2; ++q) {
            z[h + VB / UT * q] = x[q];
            z[HV + HV - 1 - (h + VB / UT * q)] = x[UT / 2 + q];
          }
        }
      }
    }
  }
  // Transposes, in the slots that b_end / b_mid read.
  static __device__ __forceinline__ void bt_begin(C* __restrict__ bp, int s, C (&z)[VB], const C* __restrict__) {
    if constexpr (!BIG) {
      fold_bt<T, L>(z, s == 0);
      C* p = bp + s * LS;
#pragma unroll
      for (int j = 0; j < L; ++j) p[j + j / G] = z[j];
    } else {
      const int k = s / UT, t = s % UT;
      if (k == 0) {
        fold_bt<T, VB>(z, t == 0);
        C* p = bp + at(VB * t);
#pragma unroll
        for (int j = 0; j < VB; ++j) p[j + j / G] = z[j];
      } else {
#pragma unroll
        for (int h = 0; h < VB / UT; ++h) {
          C x[UT];
#pragma unroll
          for (int q = 0; q < UT / 2; ++q) {
            x[q] = z[h + VB / UT * q];
            x[UT / 2 + q] = z[HV + HV - 1 - (h + VB / UT * q)];
          }
          Dft<T, UT, true, false>::run(x);
          C* p = bp + k * LS + at(UT * (t + UT * h));
#pragma unroll
          for (int j = 0; j < UT; ++j) p[j] = x[j];
        }
      }
    }
  }
  static __device__ __forceinline__ void bt_mid(C* __restrict__ bp, int s, const C* __restrict__ tw) {
    if constexpr (BIG) {
      const int k = s / UT, t = s % UT;
      if (k == 0) {
        if (t < UI) {
          C va[UT], vb[UT];
          const int part = t == 0 ? VB / 2 : VB - t;
#pragma unroll
          for (int r = 0; r < UT; ++r) {
            va[r] = bp[at(VB * r + t)];
            vb[r] = bp[at(VB * r + part)];
          }
          fold_at<T, 2 * UT, true, UI>(va, vb, t, tw + TW_A + TW_B);
#pragma unroll
          for (int r = 0; r < UT; ++r) {
            bp[at(VB * r + t)] = va[r];
            bp[at(VB * r + part)] = vb[r];
          }
        }
      } else {
        C* p = bp + k * LS + at(t);
        const C* w = tw + TW_A + t;
        C x[VB];
#pragma unroll
        for (int i = 0; i < VB; ++i) x[i] = i == 0 ? p[0] : cmul(w[UT * i], p[i * (UT + UT / G)]);
        Dft<T, VB>::run(x);
#pragma unroll
        for (int i = 0; i < VB; ++i) p[i * (UT + UT / G)] = x[i];
      }
    }
  }
};

// ---------------------------------------------------------------------------------------------
// Periodic axes: the Hartley transform of dst_engine.cuh in the same two steps (N = R L). A: radix-R butterflies
// jj = 0..L-1 over z[jj + r L], y_k[jj] = w_N^{jj k} X_k left in the slots it read (k L + jj). B: the DFT of length L of
// y_k gives Z at R m + k; H needs Z_n and Z_{N-n} together, which units k and R - k hold, so a thread runs both (unit 0
// with unit R/2, each paired with itself), 2 L values. The transform is symmetric, so its transpose is the same
// transform: the combination's transpose, then B and A with the conjugate kernel, which is the same kernel between two
// swaps of the components.
template <class T, int N> struct FoldHPlan { static constexpr int R = 0, L = 0, TPP = 1, G = 1; };
#define ETD_FOLDH(NN, R_, L_, G_)                                                  \
  template <class T> struct FoldHPlan<T, NN> {                                     \
    static_assert(R_ * L_ == NN, "R L = N");                                       \
    static constexpr int R = R_, L = L_, TPP = L_, G = G_;                         \
  };
ETD_FOLDH(32, 8, 4, 4)
ETD_FOLDH(48, 12, 4, 4)
ETD_FOLDH(64, 16, 4, 4)
ETD_FOLDH(96, 24, 4, 4)
ETD_FOLDH(128, 16, 8, 8)
ETD_FOLDH(192, 24, 8, 8)
ETD_FOLDH(256, 32, 8, 8)
ETD_FOLDH(384, 24, 16, 16)
ETD_FOLDH(512, 32, 16, 16)
#undef ETD_FOLDH

// FP32 only: FP64 passes cost their longest thread (see the plans above), and the general Hartley kernels hold half the
// values per thread up to 128 (64^2 ETDRK2: 159 us per step against 204); at 128^3, where every thread is busy, the two
// are equal (1378 and 1404). N = 512 (32 values per thread) needs enough pairs to fill the SMs: 512^2 with 256 pairs
// takes 28.9 us against 26.5.
constexpr bool foldh_has(int elem, int n, long long pairs) {
  return elem == 4 && (n == 32 || n == 48 || n == 64 || n == 96 || n == 128 || n == 192 || n == 256 || n == 384 ||
                       (n == 512 && pairs >= 1024));
}

template <class T> __device__ __forceinline__ Cx<T> swp(Cx<T> a) { return {a.y, a.x}; }

template <class T, int N> struct FoldH {
  using Plan = FoldHPlan<T, N>;
  using C = Cx<T>;
  static constexpr int R = Plan::R, L = Plan::L, TPP = Plan::TPP, G = Plan::G;
  static constexpr int H = R / 2;
  static constexpr int UA = L;
  static constexpr bool BIG = false;
  static constexpr int SLOTS = H, QB = (SLOTS + TPP - 1) / TPP;
  static constexpr int VB = 2 * L, HV = L, STEP = R;
  static constexpr int LP = N + N / G;
  static constexpr int TWN = R * L;   // w_N^{jj k} at [k][jj]; entry (0, 0) holds sc = 1/(2 sqrt N) in its imaginary part
  static_assert(L % G == 0 || G % L == 0, "padding group");
  static __device__ __forceinline__ int at(int j) { return j + j / G; }
  static constexpr int LS = L + L / G;
  static_assert(L % G == 0, "slot offsets are compile-time constants");
  static __device__ __forceinline__ bool b_on(int s) { return SLOTS % TPP == 0 || s < SLOTS; }
  // b's rows lie N/2 beyond a's: part of the thread's offset (128^3 751 us per 16 steps; as uniform steps 764, 64 x 384 x 384
  // 570 and 589), but at N = 512, where 32 bits would not hold it behind two axes of 2048, uniform steps.
  static constexpr bool FAR = (unsigned long long)(H * L + L - 1) * FOLD_MAX_STRIDE * sizeof(T) > 0xffffffffULL;
  static constexpr int PARTNER_STEPS = FAR ? H : 0;
  static constexpr __host__ __device__ __forceinline__ int partner_row(int jj) { return FAR ? jj : jj + H * L; }
  static constexpr __host__ __device__ __forceinline__ int unit2(int s) { return s == 0 ? H : R - s; }
  static constexpr __host__ __device__ __forceinline__ int row1(int s) { return s; }
  static constexpr __host__ __device__ __forceinline__ int row2(int s) { return unit2(s); }
  static __device__ __forceinline__ int own_base(int) { return 0; }
  static __device__ __forceinline__ int own_off(int s, int i) { return i < L ? s * LS + i + i / G : unit2(s) * LS + (i - L) + (i - L) / G; }

  // a[r] = z at jj + r L, b[r] = z at jj + (r + R/2) L; on return y_k[jj] in the same order
  static __device__ __forceinline__ void a(C (&va)[H], C (&vb)[H], int jj, const C* __restrict__ tw) {
    C x[R];
#pragma unroll
    for (int r = 0; r < H; ++r) {
      x[r] = va[r];
      x[H + r] = vb[r];
    }
    Dft<T, R>::run(x);
    va[0] = x[0];
#pragma unroll
    for (int k = 1; k < R; ++k) (k < H ? va[k < H ? k : 0] : vb[k < H ? 0 : k - H]) = cmul(tw[k * L + jj], x[k]);
  }
  static __device__ __forceinline__ void at_(C (&va)[H], C (&vb)[H], int jj, const C* __restrict__ tw) {
    C x[R];
    x[0] = va[0];
#pragma unroll
    for (int k = 1; k < R; ++k) x[k] = cmul(tw[k * L + jj], k < H ? va[k < H ? k : 0] : vb[k < H ? 0 : k - H]);
    Dft<T, R>::run(x);
#pragma unroll
    for (int r = 0; r < H; ++r) {
      va[r] = swp(x[r]);
      vb[r] = swp(x[H + r]);
    }
  }
  static __device__ __forceinline__ void a_get(const C* __restrict__ bp, int jj, C (&va)[H], C (&vb)[H]) {
    const C* pa = bp + at(jj);
#pragma unroll
    for (int r = 0; r < H; ++r) {
      va[r] = pa[r * LS];
      vb[r] = pa[(r + H) * LS];
    }
  }
  static __device__ __forceinline__ void a_put(C* __restrict__ bp, int jj, const C (&va)[H], const C (&vb)[H]) {
    C* pa = bp + at(jj);
#pragma unroll
    for (int r = 0; r < H; ++r) {
      pa[r * LS] = va[r];
      pa[(r + H) * LS] = vb[r];
    }
  }
  static __device__ __forceinline__ void b_mid(C* __restrict__, int, const C* __restrict__) {}
  static __device__ __forceinline__ void bt_mid(C* __restrict__, int, const C* __restrict__) {}
  // H at n and N - n from z = Z_n, w = Z_{N-n}
  static __device__ __forceinline__ void comb(C& z, C& w, T sc) {
    const C s = z + w, d = z - w;   // H_n = (s.x + d.y, s.y - d.x), H_{N-n} = (s.x - d.y, s.y + d.x)
    z = sc * sub_i(s, d);
    w = sc * add_i(s, d);
  }
  // transpose, components swapped
  static __device__ __forceinline__ void comb_t(C& p, C& r, T sc) {
    const C s = p + r, d = p - r;   // z = (s.x - d.y, s.y + d.x), w = (s.x + d.y, s.y - d.x)
    p = sc * swp(add_i(s, d));
    r = sc * swp(sub_i(s, d));
  }
  static __device__ __forceinline__ void b_end(const C* __restrict__ bp, int s, C (&z)[VB], const C* __restrict__ tw) {
    const T sc = tw[0].y;
    C u[L], v[L];
    const C *pu = bp + s * LS, *pv = bp + unit2(s) * LS;
#pragma unroll
    for (int j = 0; j < L; ++j) {
      u[j] = pu[j + j / G];
      v[j] = pv[j + j / G];
    }
    Dft<T, L>::run(u);
    Dft<T, L>::run(v);
    if (s == 0) {
      u[0] = (sc + sc) * u[0];
      u[L / 2] = (sc + sc) * u[L / 2];
#pragma unroll
      for (int m = 1; m < L / 2; ++m) comb(u[m], u[L - m], sc);
#pragma unroll
      for (int m = 0; m < L / 2; ++m) comb(v[m], v[L - 1 - m], sc);
    } else {
#pragma unroll
      for (int m = 0; m < L; ++m) comb(u[m], v[L - 1 - m], sc);
    }
#pragma unroll
    for (int j = 0; j < L; ++j) {
      z[j] = u[j];
      z[L + j] = v[j];
    }
  }
  static __device__ __forceinline__ void bt_begin(C* __restrict__ bp, int s, C (&z)[VB], const C* __restrict__ tw) {
    const T sc = tw[0].y;
    C u[L], v[L];
#pragma unroll
    for (int j = 0; j < L; ++j) {
      u[j] = z[j];
      v[j] = z[L + j];
    }
    if (s == 0) {
      u[0] = (sc + sc) * swp(u[0]);
      u[L / 2] = (sc + sc) * swp(u[L / 2]);
#pragma unroll
      for (int m = 1; m < L / 2; ++m) comb_t(u[m], u[L - m], sc);
#pragma unroll
      for (int m = 0; m < L / 2; ++m) comb_t(v[m], v[L - 1 - m], sc);
    } else {
#pragma unroll
      for (int m = 0; m < L; ++m) comb_t(u[m], v[L - 1 - m], sc);
    }
    Dft<T, L>::run(u);
    Dft<T, L>::run(v);
    C *pu = bp + s * LS, *pv = bp + unit2(s) * LS;
#pragma unroll
    for (int j = 0; j < L; ++j) {
      pu[j + j / G] = u[j];
      pv[j + j / G] = v[j];
    }
  }
};

// ---------------------------------------------------------------------------------------------
// Offsets of strided rows. A row's address is a base and a row multiple that are the same for the whole CTA (uniform
// registers) plus the thread's own part, (row * row stride + column) values with row at most fold_max_row: 32 bits where
// that fits at the largest row stride, else 64 bits. Only
// the FP64 plans of N = 1536 and 2048 (rows up to 191 and 255) need 64: 1536 x 1536 x 2048 reaches 4.8e9 bytes, and its six
// fields (232 GB) fit the card.
template <class F> __host__ __device__ constexpr int fold_max_row() {
  int m = 0;
  for (int s = 0; s < F::SLOTS; ++s) {
    if (F::row1(s) > m) m = F::row1(s);
    if (F::row2(s) > m) m = F::row2(s);
  }
  for (int jj = 0; jj < F::UA; ++jj) {
    if (jj > m) m = jj;
    if (F::partner_row(jj) > m) m = F::partner_row(jj);
  }
  return m;
}
constexpr int FOLD_MAX_COLUMN = 32;   // columns of a tile: 2 P, P <= 16
template <class F, class T>
using FoldOffset =
    typename std::conditional<((unsigned long long)fold_max_row<F>() * FOLD_MAX_STRIDE + FOLD_MAX_COLUMN) * sizeof(T) <= 0xffffffffULL,
                              unsigned, unsigned long long>::type;
template <class F, class T>
__host__ __device__ __forceinline__ FoldOffset<F, T> fold_offset(int row, size_t stride, int column) {
  using O = FoldOffset<F, T>;
  return ((O)row * (O)stride + (O)column) * (O)sizeof(T);
}

}  // namespace etd

// fold_pass.cuh - the axis passes of plans and batches on the two-step transforms of fold_dst.cuh: the folded DST-I of
// Dirichlet axes and the Hartley transform of periodic ones.
//
// A CTA owns P pencil pairs of one axis; thread tid works for pair tid % P as thread tid / P of
// it. What bounds these passes is the chain load - A - exchange - B - store and, at 3D sizes, HBM; so data
// stays in registers wherever the next step starts from what the thread holds:
//   strided axes (y, z; pair = two adjacent x columns): step A reads its rows straight from global memory
//     (P lanes on adjacent 2-element columns: full 32-byte sectors from P = 4, 128-byte lines at P = 16) and the
//     last step writes them straight back: a lone transform (TRANSFORM) crosses shared memory once, a stage
//     pass (A B | combination | B^T A^T) twice;
//   the x axis (pair = two adjacent rows): the tile is staged through shared memory with 16-byte row accesses,
//     because a thread's positions lie R or L apart along the row.
// A REACT pass runs A B | f(u) | B^T A^T in place with three barriers between the steps.
// The second operand of a stage pass (U~ or P, read at the rows a thread holds after B) and the per-mode weights
// of 2D plans come by cp.async into slots only their own thread reads, so they need no barrier, and the weights
// (constant) are requested before the dependency wait.
#pragma once
#include "fold_dst.cuh"
#include "pass_kernel.cuh"

namespace etd {

// Register budgets: FP32 plans with at most 16 values per thread take 3 CTAs of 256 threads per SM, those with up
// to 32 two (128 registers); FP64 plans run CTAs of at most 128 threads, up to 16 values 3 per SM and 32 values 2,
// and from N = 768 CTAs of 256 threads with the full register file; N = 2048 CTAs of 512 (FP64 256) threads.
// The stage kernels with weight tables (TAB: 2D plans, whose few tiles give an SM one or two CTAs) take one fewer.
// KIND: V_FOLD, V_FOLDM (Dirichlet) or V_FOLDH (periodic).
template <class T, int N, int KIND>
using FoldOf = typename std::conditional<KIND == V_FOLDH, FoldH<T, N>, Fold<T, N, KIND == V_FOLDM>>::type;
template <class T, int N, int KIND, bool TAB = false> struct FoldBudget {
  using F = FoldOf<T, N, KIND>;
  static constexpr int VALS = F::L == 256 ? 32 : (F::R > F::VB ? F::R : F::VB);   // (L = 256: unit 0's inner radix)
  static constexpr int THREADS = F::L == 256 && sizeof(T) == 4 ? 512 : sizeof(T) == 4 || F::L >= 128 ? 256 : 128;
  static constexpr int BLOCKS = F::L == 256 || (sizeof(T) == 8 && F::L == 128) ? 1 : (VALS <= 16 ? 3 : 2) - (TAB ? 1 : 0);
};

// Operations of a fold kernel: PassOp, and the transform along x.
constexpr int OP_TRANSFORM_X = OP_COUNT;

template <class T, int N, int OP> constexpr bool fold_is_x() {
  return OP == OP_ENTRY || OP == OP_EXIT || OP == OP_REACT || OP == OP_TRANSFORM_X;
}
constexpr bool fold_is_stage(int op) { return op == OP_RK1S || op == OP_S1S || op == OP_S2S; }

// 8- and 16-byte copies of one complex value / weight group
template <class T> __device__ __forceinline__ Cx<T> ld_pair(const T* p) {
  const typename V2<T>::type v = *reinterpret_cast<const typename V2<T>::type*>(p);
  return Cx<T>{v.x, v.y};
}
template <class T> __device__ __forceinline__ void st_pair(T* p, Cx<T> c) {
  *reinterpret_cast<typename V2<T>::type*>(p) = typename V2<T>::type{c.x, c.y};
}

// Address of a row-segment element: the base and the row step are the same for the whole CTA (uniform registers), the
// thread's part is fold_offset's.
template <class T, class O> __device__ __forceinline__ T* at_byte(T* base, size_t uniform, O off) {
  return reinterpret_cast<T*>(const_cast<char*>(reinterpret_cast<const char*>(base)) + uniform + off);
}

// Reciprocals of two adjacent modes' zeta. FP32: the hardware approximation and one Newton step (1 ulp), both modes in
// packed instructions, where it applies (finite normal results).
__device__ __forceinline__ Cx<double> rcp2(Cx<double> z) { return Cx<double>{rcp_rn(z.x), rcp_rn(z.y)}; }
__device__ __forceinline__ Cx<float> rcp2(Cx<float> z) {
  const Cx<float> r{rcp_approx(z.x), rcp_approx(z.y)};
  const Cx<float> e = fma2(Cx<float>{-z.x, -z.y}, r, Cx<float>{1.f, 1.f});
  return fma2(r, e, r);
}
// phi_2(-zeta) by its series (etd_coeffs.cuh), two modes.
template <class T> __device__ __forceinline__ Cx<T> phi2_series2(Cx<T> z) {
  constexpr int M = sizeof(T) == 4 ? 10 : 18;
  constexpr T c0 = (T)inv_factorial(M + 1);
  Cx<T> p{c0, c0};
  const Cx<T> nz{-z.x, -z.y};
  static_for<0, M - 1>([&](auto mc) {
    constexpr T c = (T)inv_factorial(M - decltype(mc)::value);
    p = fma2(p, nz, Cx<T>{c, c});
  });
  return p;
}
// phi_1(-zeta) = m / zeta and phi_2(-zeta) of two adjacent modes, m = 1 - e^{-zeta}: m comes from the per-axis values
// m_a = 1 - e^{-zeta_a} by 1 - (1-m)(1-m') = m + m' - m m' (no cancellation), so phi_1 needs no series at any zeta;
// phi_2 = (1 - phi_1)/zeta, below zeta = 1 its series, evaluated only in warps holding such a mode. What bounds the
// stage passes of 3D plans and batches is this evaluation's instruction count: against phi_1 and phi_1(c2) by
// series and an IEEE reciprocal per mode it is a third.
// 1 - e^{-(zeta + zeta')} of two modes from p = 1 - e^{-zeta} and m = 1 - e^{-zeta'}.
template <class T> __device__ __forceinline__ Cx<T> join_m(T m, Cx<T> p) { return fma2(Cx<T>{-m, -m}, p, p + Cx<T>{m, m}); }
// phi_1 -> 1 as zeta -> 0 (periodic mode 0; the Dirichlet boundary slot, whose values are zero); the bounds keep the
// reciprocal finite.
template <class T> constexpr T zeta_lo() { return sizeof(T) == 4 ? T(1e-30) : T(1e-290); }
template <class T> __device__ __forceinline__ Cx<T> bounded_zeta(Cx<T> zt) {
  constexpr T lo = zeta_lo<T>(), hi = T(1) / lo;
  return Cx<T>{fmin(fmax(zt.x, lo), hi), fmin(fmax(zt.y, lo), hi)};
}
// m / zeta, rz = 1 / bounded_zeta(zt); at0: the value at zeta = 0.
template <class T> __device__ __forceinline__ Cx<T> phi1_pair(Cx<T> zt, Cx<T> rz, Cx<T> m, T at0) {
  constexpr T lo = zeta_lo<T>();
  const Cx<T> q = mul2(m, rz);
  return Cx<T>{zt.x > lo ? q.x : at0, zt.y > lo ? q.y : at0};
}
template <class T> __device__ __forceinline__ Cx<T> phi2_pair(Cx<T> zeta, Cx<T> rz, Cx<T> p1, unsigned act) {
  const Cx<T> one{T(1), T(1)};
  Cx<T> p2 = mul2(one - p1, rz);
  if (__any_sync(act, zeta.x < T(1) || zeta.y < T(1))) {
    const Cx<T> s{zeta.x < T(1) ? zeta.x : T(0), zeta.y < T(1) ? zeta.y : T(0)};
    const Cx<T> q = phi2_series2<T>(s);
    p2 = Cx<T>{zeta.x < T(1) ? q.x : p2.x, zeta.y < T(1) ? q.y : p2.y};
  }
  return p2;
}

// artanh of two values. FP32: artanh x = (k/2) ln 2 + artanh s with s = (a - 2^k b)/(a + 2^k b), a = 1 + x, b = 1 - x and
// 2^k next to a/b, so that |s| <= 1/5 and the odd series up to s^11 suffices; s = x where k = 0. Component-wise packed;
// over (-1, 1) its relative error is 5.0e-8 rms and 3.6e-7 (3 ulp, the documented bound of atanhf) at most. Not finite for
// |x| >= 1.
__device__ __forceinline__ Cx<double> artanh2(Cx<double> x) { return Cx<double>{atanh(x.x), atanh(x.y)}; }
__device__ __forceinline__ Cx<float> artanh2(Cx<float> x) {
  const Cx<float> one{1.f, 1.f}, a = one + x, b = one - x;
  // k from the exponent of a / b against 3/4 (the quotient's approximation moves the line by an ulp, which the series
  // absorbs); |x| >= 1 gives a NaN below
  const float qx = a.x * rcp_approx(b.x), qy = a.y * rcp_approx(b.y);
  const int kx = (__float_as_int(qx) - 0x3f400000) >> 23, ky = (__float_as_int(qy) - 0x3f400000) >> 23;
  const Cx<float> K{__int_as_float((kx + 127) << 23), __int_as_float((ky + 127) << 23)};
  const Cx<float> kb = mul2(K, b), num = a - kb, den = a + kb;   // K b is exact
  const Cx<float> q = mul2(num, rcp2(den));
  const Cx<float> s{kx == 0 ? x.x : q.x, ky == 0 ? x.y : q.y}, s2 = mul2(s, s);
  Cx<float> p{1.f / 11, 1.f / 11};
  p = fma2(p, s2, Cx<float>{1.f / 9, 1.f / 9});
  p = fma2(p, s2, Cx<float>{1.f / 7, 1.f / 7});
  p = fma2(p, s2, Cx<float>{1.f / 5, 1.f / 5});
  p = fma2(p, s2, Cx<float>{1.f / 3, 1.f / 3});
  const Cx<float> t = fma2(mul2(s, s2), p, s);
  const Cx<float> r = fma2(Cx<float>{(float)kx, (float)ky}, Cx<float>{0.34657359027997264f, 0.34657359027997264f}, t);
  const float nan = __int_as_float(0x7fffffff);
  return Cx<float>{fabsf(x.x) < 1.f ? r.x : nan, fabsf(x.y) < 1.f ? r.y : nan};
}

// TAB: the stage weights come from the plan's per-mode tables (2D plans), else from phi evaluated per mode.
// dense: the caller's field (ENTRY source, EXIT destination).
template <class T, int N, int KIND, int OP, bool TAB>
__device__ __forceinline__ void fold_body(const PassArgs<T>& A, const int tile, T* dense) {
  using F = FoldOf<T, N, KIND>;
  constexpr bool PER = KIND == V_FOLDH;
  using C = Cx<T>;
  using VT = typename V2<T>::type;
  constexpr int H = F::H, QB = F::QB, VB = F::VB, HV = F::HV, TPP = F::TPP;
  constexpr bool XAX = fold_is_x<T, N, OP>();
  constexpr bool STAGE = fold_is_stage(OP);
  static_assert(F::UA == TPP, "one A unit per thread");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, NT = blockDim.x, P = A.P, LP = A.lp;
  int p, l;
  if (P & (P - 1)) {   // 12, 6 or 3 pairs: x extents that are odd multiples of 8 or less
    l = tid / P;
    p = tid - l * P;
  } else {
    p = tid & (P - 1);
    l = tid >> (31 - __clz(P));
  }
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + F::TWN;
  C* const bp = buf + p * LP;
  // stage passes: second operand [QB VB][NT], then the row factors e, ec (S1S), zeta (no tables), then weights
  C* own = reinterpret_cast<C*>(smem_raw + (((size_t)((unsigned char*)(buf + P * LP) - smem_raw) + 15) & ~(size_t)15));
  T* te = reinterpret_cast<T*>(own + (TAB ? QB * VB * NT : 0));
  T* tcs = te + N;
  T* tz = tcs + N;
  T* tem = tz + N;      // without tables: zeta, 1 - e, 1 - ec
  T* tcm = tem + N;
  T* wgt = tcs + N;     // with tables

  // ---- tile geometry
  int x0 = 0, o = 0;
  size_t rs = 0;        // elements between rows of the axis
  long long base = 0;
  const int q0 = tile * P;
  if constexpr (!XAX) {
    const int xt = tile % A.tiles_x;
    o = tile / A.tiles_x;
    x0 = xt * 2 * P;
    if (A.axis == 1) {
      rs = A.nx;
      base = x0 + (long long)o * A.nx * A.ny;
    } else {
      rs = (size_t)A.nx * A.ny;
      base = x0 + (long long)o * A.nx;
    }
    if (!PER && o == 0 && A.ndim == 3) {   // boundary plane z = 0 (axis y) or row y = 0 (axis z): stays zero
      count_step(A);
      return;
    }
  }
  [[maybe_unused]] auto row_off = [&](int row) { return fold_offset<F, T>(row, rs, 2 * p); };   // this thread's columns of a row
  // ---- constant tables, before the dependency wait
  {
    const C* gtw = reinterpret_cast<const C*>(A.tw);
    for (int i = tid; i < F::TWN; i += NT) cp_async<2 * sizeof(T)>(&tw[i], &gtw[i]);
  }
  constexpr int FPM = OP == OP_S1S ? 2 : 1;                 // weights per mode
  constexpr int WB = 2 * FPM * sizeof(T);                   // bytes of a pair's weights
  if constexpr (STAGE) {
    const T* gz = A.axis == 1 ? A.zeta[1] : A.zeta[2];
    const T* ge = A.axis == 1 ? A.ex[1] : A.ex[2];
    const T* gc = A.axis == 1 ? A.ec[1] : A.ec[2];
    [[maybe_unused]] const T* gem = A.axis == 1 ? A.em[1] : A.em[2];
    [[maybe_unused]] const T* gcm = A.axis == 1 ? A.cm[1] : A.cm[2];
    for (int i = tid; i < N; i += NT) {
      if (OP != OP_S2S || !TAB) cp_async<sizeof(T)>(&te[i], &ge[i]);
      if (OP == OP_S1S) cp_async<sizeof(T)>(&tcs[i], &gc[i]);
      if (!TAB) {
        cp_async<sizeof(T)>(&tz[i], &gz[i]);
        cp_async<sizeof(T)>(&tem[i], &gem[i]);
        if (OP == OP_S1S) cp_async<sizeof(T)>(&tcm[i], &gcm[i]);
      }
    }
    if constexpr (TAB) {
      if (A.coef_smem) {
#pragma unroll 1
        for (int q = 0; q < QB; ++q) {
          const int s = l + TPP * q;
          if (F::b_on(s)) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const unsigned off = ((unsigned)(h ? F::row2(s) : F::row1(s)) * A.nx + 2 * p) * (unsigned)(FPM * sizeof(T));
              unsigned char* dst = reinterpret_cast<unsigned char*>(wgt) + (size_t)((q * VB + h * HV) * NT + tid) * WB;
#pragma unroll
              for (int i = 0; i < HV; ++i) {
                const T* src = at_byte(A.coef + (size_t)x0 * FPM, (size_t)(F::STEP * i) * A.nx * (FPM * sizeof(T)), off);
                cp_async<WB < 16 ? 8 : 16>(dst + (size_t)(i * NT) * WB, src);
                if constexpr (WB == 32) cp_async<16>(dst + (size_t)(i * NT) * WB + 16, src + 16 / sizeof(T));
              }
            }
          }
        }
      }
    }
  }
  griddep_wait();
  if (A.step_inc && blockIdx.x == 0 && tid == 0) atomicAdd(A.step_inc, 1ULL);

  // ---- x axis: staged rows
  constexpr int V = sizeof(T) == 4 && (N / 4) % TPP == 0 ? 4 : 2;   // elements per vector access
  using VL = typename std::conditional<V == 4, float4, VT>::type;
  constexpr int RV = N / V;                                  // vectors per row
  constexpr int CNT = RV / TPP;                              // per thread and row
  static_assert(CNT * TPP == RV, "rows split evenly");
  auto stage_in = [&](const T* __restrict__ src) {
    constexpr int U = CNT % 4 == 0 ? 4 : (CNT % 3 == 0 ? 3 : CNT);
#pragma unroll 1
    for (int c0 = 0; c0 < CNT; c0 += U) {
      VL va[U], vb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = tid + (c0 + u) * NT, pp = i / RV, k = i - pp * RV;
        va[u] = VL{};
        vb[u] = VL{};
        if (q0 + pp < A.npairs) {
          const T* ra = src + (size_t)(2 * (q0 + pp)) * A.nx;
          va[u] = reinterpret_cast<const VL*>(ra)[k];
          vb[u] = reinterpret_cast<const VL*>(ra + A.nx)[k];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = tid + (c0 + u) * NT, pp = i / RV, k = i - pp * RV;
        C* d = buf + pp * LP;
        const T* a = reinterpret_cast<const T*>(&va[u]);
        const T* b = reinterpret_cast<const T*>(&vb[u]);
#pragma unroll
        for (int e = 0; e < V; ++e) d[F::at(V * k + e)] = C{a[e], b[e]};
      }
    }
  };
  auto stage_out = [&](T* __restrict__ dst) {
    double amp = 0;
    if (OP == OP_REACT && A.src_gx) {
      // separable source, already in the x-spectral form the pass stores (rare path)
      const double t = *A.src_t0 + ((double)*A.step_ctr + A.src_c) * (double)A.tau;
      amp = A.src_amp * exp(-A.src_rate * t);
    }
#pragma unroll 2
    for (int c = 0; c < CNT; ++c) {
      const int i = tid + c * NT, pp = i / RV, k = i - pp * RV;
      if (q0 + pp >= A.npairs) continue;
      const C* s = buf + pp * LP;
      VL va, vb;
      T* a = reinterpret_cast<T*>(&va);
      T* b = reinterpret_cast<T*>(&vb);
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const C w = s[F::at(V * k + e)];
        a[e] = w.x;
        b[e] = w.y;
      }
      const int ra = 2 * (q0 + pp), rb = ra + 1;
      if (OP == OP_REACT && A.src_gx) {
        const double ga = amp * (double)A.src_gy[ra % A.ny] * (A.src_gz ? (double)A.src_gz[ra / A.ny] : 1.0);
        const double gb = amp * (double)A.src_gy[rb % A.ny] * (A.src_gz ? (double)A.src_gz[rb / A.ny] : 1.0);
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const double g = (double)A.src_gx[V * k + e];
          a[e] += (T)(ga * g);
          b[e] += (T)(gb * g);
        }
      }
      reinterpret_cast<VL*>(dst + (size_t)ra * A.nx)[k] = va;
      reinterpret_cast<VL*>(dst + (size_t)rb * A.nx)[k] = vb;
    }
  };
  // index 0 of a row in the dense user field: nx - 1 interior values of the rows with y >= 1 (and z >= 1); periodic: the
  // pitched rows
  auto dense_row = [&](int r) -> long long {
    if constexpr (PER) return (long long)r * A.nx;
    const int y = r % A.ny, z = r / A.ny;
    if (y == 0 || (A.ndim == 3 && z == 0)) return -2;
    return ((A.ndim == 3 ? (long long)(z - 1) * (A.ny - 1) : 0LL) + (y - 1)) * (A.nx - 1) - 1;
  };
  long long* drow = reinterpret_cast<long long*>(own);   // ENTRY, EXIT: [2 P]

  constexpr int X0 = PER ? 0 : 1;   // first index with a value
  C va[H], vb[H];
  const size_t ostep = (size_t)F::STEP * rs * sizeof(T);   // bytes between a thread's consecutive rows after step B
  if constexpr (XAX) {
    if constexpr (OP == OP_ENTRY) {
      // dense starts of the tile's rows (index 0), -2 for boundary rows and rows past the end, once per row
      for (int i = tid; i < 2 * P; i += NT) drow[i] = q0 + (i >> 1) < A.npairs ? dense_row(2 * q0 + i) : -2;
      __syncthreads();
#pragma unroll 8
      for (int i = tid; i < P * N; i += NT) {
        const int pp = i / N, x = i - pp * N;
        const long long da = drow[2 * pp], db = drow[2 * pp + 1];
        C c{T(0), T(0)};
        if (x >= X0 && da > -2) c.x = dense[da + x];
        if (x >= X0 && db > -2) c.y = dense[db + x];
        buf[pp * LP + F::at(x)] = c;
      }
    } else {
      stage_in(A.in0);
    }
    cp_async_wait_all();
    __syncthreads();
    F::a_get(bp, l, va, vb);
  } else {
    // step A's rows, and the stage pass's second operand, in flight together
    const T* src = (OP == OP_S1S || OP == OP_RK1S) ? A.in1 : A.in0;
    const auto oa = row_off(l), ob = row_off(F::partner_row(l));
    const size_t step = (size_t)F::L * rs * sizeof(T);
#pragma unroll
    for (int r = 0; r < H; ++r) {
      va[r] = ld_pair(at_byte(src + base, r * step, oa));
      vb[r] = ld_pair(at_byte(src + base, (F::PARTNER_STEPS + r) * step, ob));
    }
    if constexpr (STAGE && TAB) {
      const T* g = ((OP == OP_S1S || OP == OP_RK1S) ? A.in0 : A.in1) + base;
#pragma unroll 1
      for (int q = 0; q < QB; ++q) {
        const int s = l + TPP * q;
        if (F::b_on(s)) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const auto off = row_off(h ? F::row2(s) : F::row1(s));
#pragma unroll
            for (int i = 0; i < HV; ++i)
              cp_async<2 * sizeof(T)>(&own[(q * VB + h * HV + i) * NT + tid], at_byte(g, i * ostep, off));
          }
        }
      }
    }
    if constexpr (!STAGE) cp_async_wait_all();
    else asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();   // the twiddle table
  }
  F::a(va, vb, l, tw);
  F::a_put(bp, l, va, vb);
  __syncthreads();
  // exchange inside the units of step B: the threads of a unit lie in one warp where P divides a warp's share of them
  auto unit_sync = [&]() {
    if constexpr (F::BIG) {
      if (P * F::UT <= 32 && (P & (P - 1)) == 0) __syncwarp();
      else __syncthreads();
    }
  };
  if constexpr (F::BIG) {
#pragma unroll 1
    for (int q = 0; q < QB; ++q)
      if (F::b_on(l + TPP * q)) F::b_mid(bp, l + TPP * q, tw);
    unit_sync();
  }

  if constexpr (OP == OP_TRANSFORM) {
    T* g = A.out0 + base;
    griddep_launch_dependents();
#pragma unroll 1
    for (int q = 0; q < QB; ++q) {
      const int s = l + TPP * q;
      if (F::b_on(s)) {
        C z[VB];
        F::b_end(bp, s, z, tw);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const auto off = row_off(h ? F::row2(s) : F::row1(s));
#pragma unroll
          for (int i = 0; i < HV; ++i) st_pair(at_byte(g, i * ostep, off), z[h * HV + i]);
        }
      }
    }
    return;
  } else if constexpr (OP == OP_ENTRY || OP == OP_EXIT || OP == OP_TRANSFORM_X) {
    C z[QB][VB];
#pragma unroll
    for (int q = 0; q < QB; ++q)
      if (F::b_on(l + TPP * q)) F::b_end(bp, l + TPP * q, z[q], tw);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < QB; ++q)
      if (F::b_on(l + TPP * q)) {
#pragma unroll
        for (int i = 0; i < VB; ++i)
          bp[F::at((i < HV ? F::row1(l + TPP * q) : F::row2(l + TPP * q)) + F::STEP * (i % HV))] = z[q][i];
      }
    __syncthreads();
    griddep_launch_dependents();
    if constexpr (OP == OP_EXIT) {
      for (int i = tid; i < 2 * P; i += NT) drow[i] = q0 + (i >> 1) < A.npairs ? dense_row(2 * q0 + i) : -2;
      __syncthreads();
#pragma unroll 8
      for (int i = tid; i < P * N; i += NT) {
        const int pp = i / N, x = i - pp * N;
        const long long da = drow[2 * pp], db = drow[2 * pp + 1];
        const C c = buf[pp * LP + F::at(x)];
        if (x >= X0 && da > -2) dense[da + x] = c.x;
        if (x >= X0 && db > -2) dense[db + x] = c.y;
      }
    } else {
      stage_out(A.out0);
    }
    return;
  } else {
    // pointwise work between the transform and its transpose
    [[maybe_unused]] C pz, pe, pc, pm, pcm;   // the pair's factors over the other axes
    if constexpr (STAGE) {
      const int x = x0 + 2 * p;
      pe = ld_pair(A.ex[0] + x);
      pc = ld_pair(A.ec[0] + x);
      if constexpr (!TAB) {
        pz = ld_pair(A.zeta[0] + x);
        pm = ld_pair(A.em[0] + x);
        pcm = ld_pair(A.cm[0] + x);
      }
      if (A.ndim == 3) {
        pe = A.ex[1][o] * pe;
        pc = A.ec[1][o] * pc;
        if constexpr (!TAB) {
          const T z = A.zeta[1][o], m = A.em[1][o], cm = A.cm[1][o];
          pz = pz + C{z, z};
          pm = join_m(m, pm);
          pcm = join_m(cm, pcm);
        }
      }
    }
    // Stage passes that evaluate their weights take the second operand straight from global memory, CH values
    // ahead of the arithmetic (shared memory for it would cost a CTA per SM).
    constexpr int CH = HV < 8 ? HV : 8, NCH = VB / CH;
    static_assert(HV % CH == 0, "chunks within a half");
    [[maybe_unused]] const T* gu = ((OP == OP_S1S || OP == OP_RK1S) ? A.in0 : A.in1) + base;
    [[maybe_unused]] auto load_u = [&](int s, int c, C (&u)[CH]) {
      const int h = c * CH / HV, i0 = c * CH % HV;
      const T* g = at_byte(gu, i0 * ostep, row_off(h ? F::row2(s) : F::row1(s)));
#pragma unroll
      for (int i = 0; i < CH; ++i) u[i] = ld_pair(at_byte(g, i * ostep, 0u));
    };
#pragma unroll 1
    for (int q = 0; q < QB; ++q) {
      const int s = l + TPP * q;
      if (!F::b_on(s)) continue;
      C z[VB];
      [[maybe_unused]] C un[CH];
      if constexpr (STAGE && !TAB) load_u(s, 0, un);
      F::b_end(bp, s, z, tw);
      if constexpr (OP == OP_REACT) {
        const T fl = A.flin, fc = A.fcub;
#pragma unroll
        for (int i = 0; i < VB; ++i) {
          const C r = mul2(z[i], fma2(mul2(C{fc, fc}, z[i]), z[i], C{fl, fl}));
          if constexpr (PER) {
            // the logarithmic term of the Flory-Huggins reaction (periodic plans): through the thread's own slots below
            if (A.flog != T(0)) bp[F::own_off(s, i)] = z[i];
          }
          z[i] = r;
        }
        if constexpr (PER) {
          if (A.flog != T(0)) {
            const T fg = A.flog;
#pragma unroll 4
            for (int i = 0; i < VB; ++i) {   // a loop: artanh's code once
              bp[F::own_off(s, i)] = fg * artanh2(bp[F::own_off(s, i)]);
            }
#pragma unroll
            for (int i = 0; i < VB; ++i) z[i] = z[i] + bp[F::own_off(s, i)];
          }
        }
      } else if constexpr (TAB) {
        T* g1 = A.out1 + base;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row = h ? F::row2(s) : F::row1(s);
          const auto off = row_off(row);
          const unsigned coff = ((unsigned)row * A.nx + 2 * p) * (unsigned)(FPM * sizeof(T));
          const C* uo = own + (q * VB + h * HV) * NT + tid;
          const unsigned char* wo = reinterpret_cast<const unsigned char*>(wgt) + (size_t)((q * VB + h * HV) * NT + tid) * WB;
#pragma unroll
          for (int i = 0; i < HV; ++i) {
            const C u = uo[i * NT], w = z[h * HV + i];
            const VT* src = A.coef_smem ? reinterpret_cast<const VT*>(wo + (size_t)(i * NT) * WB)
                                        : reinterpret_cast<const VT*>(at_byte(A.coef + (size_t)x0 * FPM,
                                                                              (size_t)(F::STEP * i) * A.nx * (FPM * sizeof(T)), coff));
            T cf[2 * FPM];
#pragma unroll
            for (int e = 0; e < FPM; ++e) {
              const VT v = src[e];
              cf[2 * e] = v.x;
              cf[2 * e + 1] = v.y;
            }
            C r1;
            if constexpr (OP == OP_S1S) {          // {c2 tau phi1(-c2 z), tau (phi1 - phi2/c2)(-z)} per mode
              const T e = te[row + F::STEP * i], ec = tcs[row + F::STEP * i];
              z[h * HV + i] = C{pc.x * ec * u.x + cf[0] * w.x, pc.y * ec * u.y + cf[2] * w.y};
              r1 = C{pe.x * e * u.x + cf[1] * w.x, pe.y * e * u.y + cf[3] * w.y};
            } else if constexpr (OP == OP_RK1S) {  // tau phi1(-z) per mode
              const T e = te[row + F::STEP * i];
              z[h * HV + i] = r1 = C{pe.x * e * u.x + cf[0] * w.x, pe.y * e * u.y + cf[1] * w.y};
            } else {                               // S2S: tau phi2(-z)/c2 per mode; u is P
              z[h * HV + i] = r1 = C{u.x + cf[0] * w.x, u.y + cf[1] * w.y};
            }
            st_pair(at_byte(g1, i * ostep, off), r1);
          }
        }
      } else {
        // weights evaluated per mode: through the thread's own slots, so that the evaluation's code is a loop
        [[maybe_unused]] const T tau = A.tau, inv_c2 = T(1) / A.c2;
        C* zs = bp + F::own_base(s);
#pragma unroll
        for (int i = 0; i < VB; ++i) zs[F::own_off(s, i)] = z[i];
#pragma unroll 1
        for (int c = 0; c < NCH; ++c) {
          C uc[CH];
#pragma unroll
          for (int i = 0; i < CH; ++i) uc[i] = un[i];
          if (c + 1 < NCH) load_u(s, c + 1, un);
          const int h = c * CH / HV, i0 = c * CH % HV;
          const int row = (h ? F::row2(s) : F::row1(s));
          T* g1 = at_byte(A.out1 + base, i0 * ostep, row_off(row));
          C* zo = zs + F::own_off(s, c * CH);
          const int r0 = row + F::STEP * i0;
          const T *tzr = tz + r0, *ter = te + r0, *tcr = tcs + r0, *tmr = tem + r0, *tcmr = tcm + r0;
#pragma unroll
          for (int i = 0; i < CH; ++i) {
            const C u = uc[i], w = zo[i];
            const T zj = tzr[F::STEP * i], mj = tmr[F::STEP * i];
            const C zt = pz + C{zj, zj}, zeta = bounded_zeta(zt), rz = rcp2(zeta);
            const C p1 = phi1_pair(zt, rz, join_m(mj, pm), T(1));
            const unsigned act = __activemask();
            C o0, o1;
            if constexpr (OP == OP_S1S) {
              const T ej = ter[F::STEP * i], cj = tcr[F::STEP * i], cmj = tcmr[F::STEP * i];
              const C p2 = phi2_pair<T>(zeta, rz, p1, act);
              // c2 phi_1(-c2 zeta) = (1 - e^{-c2 zeta}) / zeta
              const C t1 = phi1_pair(zt, rz, join_m(cmj, pcm), A.c2);
              o0 = fma2(mul2(C{tau, tau}, t1), w, mul2(mul2(pc, C{cj, cj}), u));
              o1 = fma2(mul2(C{tau, tau}, fma2(C{-inv_c2, -inv_c2}, p2, p1)), w, mul2(mul2(pe, C{ej, ej}), u));
            } else if constexpr (OP == OP_RK1S) {
              const T ej = ter[F::STEP * i];
              o0 = o1 = fma2(mul2(C{tau, tau}, p1), w, mul2(mul2(pe, C{ej, ej}), u));
            } else {
              const T ti = tau * inv_c2;
              o0 = o1 = fma2(mul2(C{ti, ti}, phi2_pair<T>(zeta, rz, p1, act)), w, u);
            }
            zo[i] = o0;
            st_pair(at_byte(g1, i * ostep, 0u), o1);
          }
        }
#pragma unroll
        for (int i = 0; i < VB; ++i) z[i] = zs[F::own_off(s, i)];
      }
      F::bt_begin(bp, s, z, tw);
    }
    unit_sync();
    if constexpr (F::BIG) {
#pragma unroll 1
      for (int q = 0; q < QB; ++q)
        if (F::b_on(l + TPP * q)) F::bt_mid(bp, l + TPP * q, tw);
    }
    __syncthreads();
    F::a_get(bp, l, va, vb);
    F::at_(va, vb, l, tw);
    if constexpr (XAX) {
      F::a_put(bp, l, va, vb);
      __syncthreads();
      griddep_launch_dependents();
      stage_out(A.out0);
    } else {
      griddep_launch_dependents();
      const auto oa = row_off(l), ob = row_off(F::partner_row(l));
      const size_t step = (size_t)F::L * rs * sizeof(T);
      T* g = A.out0 + base;
#pragma unroll
      for (int r = 0; r < H; ++r) {
        st_pair(at_byte(g, r * step, oa), va[r]);
        st_pair(at_byte(g, (F::PARTNER_STEPS + r) * step, ob), vb[r]);
      }
    }
  }
}

template <class T, int N, int KIND, int OP, bool TAB>
__global__ void __launch_bounds__(FoldBudget<T, N, KIND>::THREADS, FoldBudget<T, N, KIND, TAB>::BLOCKS)
    fold_kernel(const PassArgs<T> A) {
  fold_body<T, N, KIND, OP, TAB>(A, (int)blockIdx.x, OP == OP_ENTRY ? const_cast<T*>(A.in0) : A.out0);
}

// Batches: CTA b works on tile map[b].y of problem descs[map[b].x]; entry and exit passes take the caller's field
// from user[].
template <class T, int N, int KIND, int OP>
__global__ void __launch_bounds__(FoldBudget<T, N, KIND>::THREADS, FoldBudget<T, N, KIND>::BLOCKS)
    fold_kernel_batched(const PassArgs<T>* __restrict__ descs, const int2* __restrict__ map, T* const* __restrict__ user) {
  const int2 m = map[blockIdx.x];
  const PassArgs<T>& A = descs[m.x];   // read in place
  T* dense = nullptr;
  if (OP == OP_ENTRY || OP == OP_EXIT) dense = user[A.user_slot];
  fold_body<T, N, KIND, OP, false>(A, m.y, dense);
}

// Shared memory of a launch: op, pairs per CTA, pair stride, tables / staged weights.
inline size_t fold_smem_bytes(const KernelInfo& k, int op, int P, int lp, bool tab, bool staged) {
  const size_t c = 2 * (size_t)k.elem;
  size_t b = ((size_t)k.twn + (size_t)P * lp) * c;
  b = (b + 15) & ~(size_t)15;
  if (!fold_is_stage(op)) return b + (op == OP_ENTRY || op == OP_EXIT ? 2 * (size_t)P * sizeof(long long) : 0);
  const size_t own = tab ? (size_t)k.own_vals * P * k.tpp : 0;
  b += own * c + (tab ? 2 : 5) * (size_t)k.N * k.elem;
  if (tab && staged) b += own * 2 * k.elem * (op == OP_S1S ? 2 : 1);
  return b;
}

template <class T, int N, int KIND> KernelInfo fold_info() {
  using F = FoldOf<T, N, KIND>;
  KernelInfo k{};
  k.N = N;
  k.tpp = F::TPP;
  k.lp = F::LP;
  k.elem = (int)sizeof(T);
  k.fft_len = KIND == V_FOLDH ? N : 2 * N;
  k.odd = KIND;
  k.padg = F::G;
  k.twn = F::TWN;
  k.radix[0] = F::R;
  k.radix[1] = F::L;
  k.min_blocks = FoldBudget<T, N, KIND>::BLOCKS;
  k.max_threads = FoldBudget<T, N, KIND>::THREADS;
  k.own_vals = F::QB * F::VB;
#define ETD_FOLD_OP(OP)                                                                   \
  k.fn_op[OP] = reinterpret_cast<const void*>(&fold_kernel<T, N, KIND, OP, false>);             \
  k.fn_batched_op[OP] = reinterpret_cast<const void*>(&fold_kernel_batched<T, N, KIND, OP>);
  ETD_FOLD_OP(OP_ENTRY)
  ETD_FOLD_OP(OP_EXIT)
  ETD_FOLD_OP(OP_REACT)
  ETD_FOLD_OP(OP_TRANSFORM)
  ETD_FOLD_OP(OP_RK1S)
  ETD_FOLD_OP(OP_S1S)
  ETD_FOLD_OP(OP_S2S)
#undef ETD_FOLD_OP
  k.fn_tab[OP_RK1S] = reinterpret_cast<const void*>(&fold_kernel<T, N, KIND, OP_RK1S, true>);
  k.fn_tab[OP_S1S] = reinterpret_cast<const void*>(&fold_kernel<T, N, KIND, OP_S1S, true>);
  k.fn_tab[OP_S2S] = reinterpret_cast<const void*>(&fold_kernel<T, N, KIND, OP_S2S, true>);
  k.fn_x = reinterpret_cast<const void*>(&fold_kernel<T, N, KIND, OP_TRANSFORM_X, false>);
  return k;
}

}  // namespace etd

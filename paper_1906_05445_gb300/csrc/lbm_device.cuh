// lbm_device.cuh -- device building blocks of the fused collide-stream sweep
// (Peng, Ayala & Wang, arXiv 1906.05445, Eqs. 1-3 with Guo forcing).
//
// Storage holds deviations d_i = f_i - w_i (optionally scaled for FP16), SoA
// [Q][z][y][x].  The compute type T is double for the FP64 build and float
// otherwise.  Everything that depends on the lattice is a compile-time
// constant so that the unrolled loops fold to straight-line arithmetic.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

namespace lbm {

// Compile-time loop: f(std::integral_constant<int, I>) for I = 0..N-1, so
// that lattice tables indexed by I are constant expressions, not run-time
// lookups, whatever the unroller decides.
template <typename F, int... I>
__host__ __device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__host__ __device__ __forceinline__ void static_for(F &&f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// ---------------------------------------------------------------- lattices
// direction order: see include/lbm.h
template <int LAT> struct Lat;

template <> struct Lat<0> {  // D2Q9
  static constexpr int Q = 9, D = 2;
  __host__ __device__ static constexpr int ex(int i) {
    return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
  }
  __host__ __device__ static constexpr int ey(int i) {
    return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
  }
  __host__ __device__ static constexpr int ez(int) { return 0; }
  __host__ __device__ static constexpr int opp(int i) {
    return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4 + 1) : ((i - 5 + 2) % 4 + 5));
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
};

template <> struct Lat<1> {  // D3Q19
  static constexpr int Q = 19, D = 3;
  __host__ __device__ static constexpr int ex(int i) {
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
           : ((i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0);
  }
  __host__ __device__ static constexpr int ey(int i) {
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
           : ((i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0);
  }
  __host__ __device__ static constexpr int ez(int i) {
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
           : ((i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0);
  }
  __host__ __device__ static constexpr int opp(int i) {
    return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1);
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
};

// component a of e_i
template <int LAT> __host__ __device__ constexpr int ecomp(int a, int i) {
  return a == 0 ? Lat<LAT>::ex(i) : (a == 1 ? Lat<LAT>::ey(i) : Lat<LAT>::ez(i));
}
template <int LAT> __host__ __device__ constexpr int enorm2(int i) {
  return ecomp<LAT>(0, i) * ecomp<LAT>(0, i) + ecomp<LAT>(1, i) * ecomp<LAT>(1, i) +
         ecomp<LAT>(2, i) * ecomp<LAT>(2, i);
}

// Gram-Schmidt moment rows (Lallemand-Luo for D2Q9, d'Humieres et al. for
// D3Q19) as polynomials of e; row order matches lbm_lattice_desc.mrt_rates.
template <int LAT>
__host__ __device__ constexpr int mrow(int k, int i) {
  using L = Lat<LAT>;
  const int x = L::ex(i), y = L::ey(i), z = L::ez(i);
  const int e2 = x * x + y * y + z * z;
  if (LAT == 0) {
    return k == 0 ? 1
         : k == 1 ? -4 + 3 * e2
         : k == 2 ? (8 - 21 * e2 + 9 * e2 * e2) / 2
         : k == 3 ? x
         : k == 4 ? (-5 + 3 * e2) * x
         : k == 5 ? y
         : k == 6 ? (-5 + 3 * e2) * y
         : k == 7 ? x * x - y * y
                  : x * y;
  }
  return k == 0 ? 1
       : k == 1 ? 19 * e2 - 30
       : k == 2 ? (21 * e2 * e2 - 53 * e2 + 24) / 2
       : k == 3 ? x
       : k == 4 ? (5 * e2 - 9) * x
       : k == 5 ? y
       : k == 6 ? (5 * e2 - 9) * y
       : k == 7 ? z
       : k == 8 ? (5 * e2 - 9) * z
       : k == 9 ? 3 * x * x - e2
       : k == 10 ? (3 * e2 - 5) * (3 * x * x - e2)
       : k == 11 ? y * y - z * z
       : k == 12 ? (3 * e2 - 5) * (y * y - z * z)
       : k == 13 ? x * y
       : k == 14 ? y * z
       : k == 15 ? x * z
       : k == 16 ? (y * y - z * z) * x
       : k == 17 ? (z * z - x * x) * y
                 : (x * x - y * y) * z;
}

template <int LAT>
__host__ __device__ constexpr int mnorm(int k) {
  int s = 0;
  for (int i = 0; i < Lat<LAT>::Q; i++) s += mrow<LAT>(k, i) * mrow<LAT>(k, i);
  return s;
}

// moments whose rate is irrelevant (density and momentum)
template <int LAT>
__host__ __device__ constexpr bool conserved(int k) {
  return k == 0 || k == 3 || k == 5 || (LAT == 1 && k == 7);
}

// ---------------------------------------------------------------- storage
// How a kernel reads populations:
//   LD_NC   read-only path: nothing writes the array while the kernel runs;
//   LD_ONCE evict-first (the line is not needed again before it is rewritten);
//   LD_L2   from L2: a kernel of several steps reads what other SMs wrote
//           earlier in the same launch, which the read-only path and L1 may
//           hold stale.
enum : int { LD_NC = 0, LD_ONCE = 1, LD_L2 = 2 };
template <int POL, typename P> __device__ __forceinline__ P ld_pol(const P *p) {
  if constexpr (POL == LD_NC) return __ldg(p);
  else if constexpr (POL == LD_ONCE) return __ldcs(p);
  else return __ldcg(p);
}
template <typename S> struct Store;
// st_stream: evict-first stores
template <> struct Store<double> {
  template <int POL = LD_NC, typename T> __device__ static T ld(const double *p, T) {
    return (T)ld_pol<POL>(p);
  }
  template <typename T> __device__ static void st(double *p, T v, T) { *p = (double)v; }
  template <typename T> __device__ static void st_stream(double *p, T v, T) { __stcs(p, (double)v); }
};
template <> struct Store<float> {
  template <int POL = LD_NC, typename T> __device__ static T ld(const float *p, T) {
    return (T)ld_pol<POL>(p);
  }
  template <typename T> __device__ static void st(float *p, T v, T) { *p = (float)v; }
  template <typename T> __device__ static void st_stream(float *p, T v, T) { __stcs(p, (float)v); }
};
template <> struct Store<__nv_bfloat16> {
  template <int POL = LD_NC, typename T> __device__ static T ld(const __nv_bfloat16 *p, T) {
    return (T)__bfloat162float(ld_pol<POL>(p));
  }
  template <typename T> __device__ static void st(__nv_bfloat16 *p, T v, T) {
    *p = __float2bfloat16_rn((float)v);
  }
  template <typename T> __device__ static void st_stream(__nv_bfloat16 *p, T v, T s) { st(p, v, s); }
};
// FP16 keeps d_i * scale (scale = 2^k) so that deviations stay in the normal
// range; the scale is exact in binary, so it only shifts the exponent.
template <> struct Store<__half> {
  template <int POL = LD_NC, typename T> __device__ static T ld(const __half *p, T inv_scale) {
    return (T)__half2float(ld_pol<POL>(p)) * inv_scale;
  }
  template <typename T> __device__ static void st(__half *p, T v, T inv_scale) {
    *p = __float2half_rn((float)(v / inv_scale));
  }
  template <typename T> __device__ static void st_stream(__half *p, T v, T s) { st(p, v, s); }
};

// ---------------------------------------------------------------- collision
template <typename T> struct Coll {
  T omega;      // 1/tau: rate of the stress moments (and of BGK)
  T omc;        // 1 - omega
  T cforce;     // 1 - omega/2
  T ds[19];     // omega - s_k per moment (0: same as BGK)
};

// Incompressible equilibrium deviation w_i[drho + 3 e.u + 4.5 (e.u)^2 - 1.5 u^2]
template <int LAT, typename T>
__device__ __forceinline__ T feq_dev(int i, T drho, T ux, T uy, T uz, T uu) {
  using L = Lat<LAT>;
  const T eu = (T)L::ex(i) * ux + (T)L::ey(i) * uy + (T)L::ez(i) * uz;
  return (T)L::w(i) * (drho + (T)3 * eu + (T)4.5 * eu * eu - (T)1.5 * uu);
}

// e_i . v with the lattice velocity folded at compile time
template <int LAT, int I, typename T>
__device__ __forceinline__ T edot(T vx, T vy, T vz) {
  using L = Lat<LAT>;
  T r = (T)0;
  if constexpr (L::ex(I) == 1) r += vx;
  if constexpr (L::ex(I) == -1) r -= vx;
  if constexpr (L::ey(I) == 1) r += vy;
  if constexpr (L::ey(I) == -1) r -= vy;
  if constexpr (L::ez(I) == 1) r += vz;
  if constexpr (L::ez(I) == -1) r -= vz;
  return r;
}

// collision modes of the kernels
enum : int { CM_BGK = 0, CM_MRT = 1, CM_MRT_Q = 2 };

// q-moment rows (energy flux, odd in e): (5|e|^2 - 9) e_a on D3Q19,
// (3|e|^2 - 5) e_a on D2Q9 (rows 4, 6, 8 / 4, 6 of the basis)
template <int LAT> __host__ __device__ constexpr int qrow(int a, int i) {
  return mrow<LAT>(4 + 2 * a, i);
}

// ---------------------------------------------------------------- arithmetic
// The collision below is written once for one node (float, double) and for a
// node pair in packed FP32x2 arithmetic (float2: one instruction for two
// nodes; lane x and lane y of every float2).  Each operation is rounded by
// itself (nothing is contracted), so that the packed and the node-by-node
// kernels give the same bits.
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b, exactly as a scalar subtraction (b * -1 is exact)
__device__ __forceinline__ float2 vsub(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
template <typename V, typename C> __device__ __forceinline__ V vbc(C s) {
  if constexpr (std::is_same<V, float2>::value) return make_float2((float)s, (float)s);
  else return (V)s;
}

// e_I . v for the first direction of an opposite pair, which has a positive
// component on both lattices' orderings (no addition to a zero: the compiler
// may not drop those)
template <int LAT, int I, typename V>
__device__ __forceinline__ V edot_lead(V vx, V vy, V vz) {
  using L = Lat<LAT>;
  constexpr int a = L::ex(I), b = L::ey(I), c = L::ez(I);
  static_assert(a == 1 || b == 1 || c == 1, "pair leader without a positive component");
  constexpr int first = a == 1 ? 0 : (b == 1 ? 1 : 2);
  V r = first == 0 ? vx : (first == 1 ? vy : vz);
  if constexpr (first < 1 && b == 1) r = vadd(r, vy);
  if constexpr (first < 2 && c == 1) r = vadd(r, vz);
  if constexpr (a == -1) r = vsub(r, vx);
  if constexpr (b == -1) r = vsub(r, vy);
  if constexpr (c == -1) r = vsub(r, vz);
  return r;
}

// The weights of the collision: w0, the diagonal weight wb (an axis pair has
// r wb, r = 2 on D3Q19, 4 on D2Q9, exactly), and 3 w1 and 3 wb of the terms
// linear in e.  In FP32 they are the neighbours of the printed fractions that
// add up exactly, w0 + 6 r wb + 12 wb = 1 and 2 (3 w1) + 8 (3 wb) = 1 on D3Q19
// (w0 + 4 r wb + 4 wb = 1 and 2 (3 w1) + 4 (3 wb) = 1 on D2Q9): rounded one by
// one (1/6 and 1/12 are both 3e-8 high) they scale the momentum by 1 + 3e-8 omega
// every step.
template <int LAT, typename C> struct CollW {
  static constexpr bool f32 = sizeof(C) == 4;
  static constexpr double p25 = 1.0 / 33554432.0, p26 = p25 / 2, p27 = p25 / 4, p29 = p25 / 16;
  static constexpr C w0 = (C)(f32 ? (LAT == 0 ? 14913082 * p25 : 11184812 * p25) : Lat<LAT>::w(0));
  static constexpr C wb = (C)(f32 ? 14913080 * p29 : 1.0 / 36.0);
  static constexpr C w1x3 = (C)(f32 ? (LAT == 0 ? 11184811 * p25 : 11184810 * p26)
                                    : 3.0 * Lat<LAT>::w(1));
  static constexpr C wbx3 = (C)(f32 ? (LAT == 0 ? 11184810 * p27 : 11184811 * p27) : 1.0 / 12.0);
};

// BGK, or MRT whose only non-BGK rates are those of the q moments, in place.
// Both lattices have one weight for the axis pairs (r wb) and one for the
// diagonal pairs (wb), diagonal directions have exactly two components, and
// the q rows are e_a times -(c - 1) on an axis pair and +1 on a diagonal one
// (c = 5 on D3Q19, 3 on D2Q9).  So every term of the pair form above is a
// linear or bilinear form of a few vectors, shared by all pairs:
//   j_a  = sum over the pairs of e_a (f_i - f_j), u = j + F/2;
//   odd  : omega A + cforce AF = 3 w e.v, v = omega u + cforce F = omega j + F
//          (one rounding: the force of a slow flow is a small fraction of an
//          ulp of j, and adding it twice rounds it twice);
//   even : w [omega (drho - 1.5 u^2) - 3 cforce u.F + (e.u)(4.5 omega e.u + 9 cforce e.F)];
//          with h = wb (4.5 omega u + 9 cforce F), X_a = u_a h_a and S = sum X,
//          Bb = wb omega drho - S/3 is the part without e (its quadratic terms
//          are a third of S), an axis pair has r (Bb + X_a), a diagonal pair
//          Bb + X_a + X_b +- (u_a h_b + u_b h_a), the rest node the w0 part of Bb;
//   q    : m_a = sum_i q_a,i (f_i - f_j) + K (F_a - 2 u_a), K = -1/3 (D3Q19) or
//          -1/2 (D2Q9); the sum is j_a - c d_a (d_a: the axis pair's
//          difference) and F - 2u = -2j, so m_a = c (6 w1 j_a - d_a): the force
//          cancels; the correction k m_a q_a,i joins the odd part.
// That is 135 operations per D3Q19 node (about 250 when every pair forms its
// own e.u, e.F and q sums), which bounds FP64 (GB300 issues about 2 FP64
// operations per SM and cycle; a 96^3 lattice without solids 415.7 -> 258
// us per step) and most of the 16-bit kernels (FP16 160^3: 58.0 -> 51.5 us).
// With SL > 0 the populations and the force come in units of 2^-SL (FP16
// storage's scaled deviations) and the results go out in them: everything
// but h is linear, and h takes the factor 2^-SL.  Power-of-two scaling
// commutes with rounding, so the stored values equal those of colliding the
// unscaled deviations.
// EVEN_FIRST adds the small even part to the old value before the larger odd
// one, so that the odd part is rounded once (half the stress noise of adding the
// parts first).  BF16 storage is also faster with it (160^3 51.7 us per step
// against 53.3); FP16 storage, whose rounding hides the difference, is not
// (53.4 / 53.3) and adds the parts first.
template <typename ST> __host__ __device__ constexpr bool even_first() {
  return !std::is_same<ST, __half>::value;
}
template <int LAT, int CM, int SL, bool EVEN_FIRST, typename V, typename C>
__device__ __forceinline__ void collide_two_rate(V (&f)[Lat<LAT>::Q], V Fx, V Fy, V Fz,
                                                 const Coll<C> &c) {
  using L = Lat<LAT>;
  using CW = CollW<LAT, C>;
  constexpr int Q = L::Q, D = L::D;
  static_assert(CM != CM_MRT, "general MRT rates: collide");
  constexpr C kInv = (C)1 / (C)(1 << SL);  // exact
  constexpr double wb = L::w(Q - 1);
  constexpr double rw = L::w(1) / L::w(Q - 1), r0 = L::w(0) / L::w(Q - 1);
  constexpr int qc = D == 3 ? 5 : 3;  // c
  static_assert(qrow<LAT>(0, 1) == 1 - qc, "axis q row");
  // density, and the momentum from the pairs' differences
  V drho = f[0];
  V j[3];
  V dax[3];
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (i > 0 && L::opp(i) > i) {
      constexpr int o = L::opp(i);
      constexpr bool axis = enorm2<LAT>(i) == 1;
      drho = vadd(drho, vadd(f[i], f[o]));
      const V d = vsub(f[i], f[o]);
      static_for<D>([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        constexpr int ea = ecomp<LAT>(a, i);
        if constexpr (ea != 0) {
          // the axis pairs come first and start each sum
          if constexpr (axis) {
            static_assert(ea == 1, "axis leader");
            dax[a] = d;
            j[a] = d;
          } else if constexpr (ea == 1) {
            j[a] = vadd(j[a], d);
          } else {
            j[a] = vsub(j[a], d);
          }
        }
      });
    }
  });
  const V F[3] = {Fx, Fy, Fz};
  const V half = vbc<V>((C)0.5);
  const V om = vbc<V>(c.omega), omc = vbc<V>(c.omc);
  const V h_u = vbc<V>(c.omega * (C)(4.5 * wb) * kInv);
  const V h_f = vbc<V>(c.cforce * (C)(9.0 * wb) * kInv);
  V u[D], h[D], X[D];
  static_for<D>([&](auto ac) {
    constexpr int a = decltype(ac)::value;
    u[a] = vfma(half, F[a], j[a]);
    h[a] = vfma(h_u, u[a], vmul(h_f, F[a]));
    X[a] = vmul(u[a], h[a]);
  });
  V S = vadd(X[0], X[1]);
  if constexpr (D == 3) S = vadd(S, X[2]);
  const V orho = vmul(om, drho);
  const V Bb = vfma(vbc<V>((C)(-1.0 / 3.0)), S, vmul(vbc<V>(CW::wb), orho));
  const V Ba = vmul(vbc<V>((C)rw), Bb);
  const V Bd = vadd(Bb, S);  // Bb + X_a + X_b + X_c
  f[0] = vfma(omc, f[0], vfma(vbc<V>((C)(-r0 / 3.0)), S, vmul(vbc<V>(CW::w0), orho)));
  // odd part: 3 w e.v plus the q correction; g for the diagonal pairs, ga for
  // the axis pairs
  V g[3], ga[D];
  static_for<D>([&](auto ac) {
    constexpr int a = decltype(ac)::value;
    const V v = vfma(om, j[a], F[a]);
    if constexpr (CM == CM_MRT_Q) {
      // one rate for all q rows: c (omega - s_q) / |M_q|^2, negative
      const C k = c.ds[4] * (C)(-(double)qc / mnorm<LAT>(4));
      const V aq = vmul(vbc<V>(k), vfma(vbc<V>((C)-2 * CW::w1x3), j[a], dax[a]));
      g[a] = vfma(vbc<V>(CW::wbx3), v, aq);
      ga[a] = vfma(vbc<V>((C)(1 - qc)), aq, vmul(vbc<V>(CW::w1x3), v));
    } else {
      g[a] = vmul(vbc<V>(CW::wbx3), v);
      ga[a] = vmul(vbc<V>(CW::w1x3), v);
    }
  });
  if constexpr (D == 2) g[2] = g[0];  // not read
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (i > 0 && L::opp(i) > i) {
      constexpr int o = L::opp(i);
      constexpr bool axis = enorm2<LAT>(i) == 1;
      V P, O;
      if constexpr (axis) {
        constexpr int a = L::ex(i) ? 0 : (L::ey(i) ? 1 : 2);
        P = vfma(vbc<V>((C)rw), X[a], Ba);
        O = ga[a];
      } else {
        constexpr int a = L::ex(i) ? 0 : 1, b = L::ez(i) ? 2 : 1;
        static_assert(enorm2<LAT>(i) == 2 && a < b, "two components");
        V base = Bd;
        if constexpr (D == 3) base = vsub(Bd, X[3 - a - b]);
        const V X2 = vfma(u[a], h[b], vmul(u[b], h[a]));
        P = ecomp<LAT>(a, i) * ecomp<LAT>(b, i) > 0 ? vadd(base, X2) : vsub(base, X2);
        O = edot_lead<LAT, i>(g[0], g[1], g[2]);
      }
      if constexpr (EVEN_FIRST) {
        f[i] = vadd(vfma(omc, f[i], P), O);
        f[o] = vsub(vfma(omc, f[o], P), O);
      } else {
        f[i] = vfma(omc, f[i], vadd(P, O));
        f[o] = vfma(omc, f[o], vsub(P, O));
      }
    }
  });
}

// Sum over the pair leaders i of q_a,i 3 w_i e_i,b: the q moments of the
// pairs' terms -2 A_i + AF_i (A_i = 3 w_i e_i.u, AF_i = 3 w_i e_i.F) are
// sum_b K_ab (F_b - 2 u_b).
template <int LAT> __host__ __device__ constexpr double qk(int a, int b) {
  using L = Lat<LAT>;
  double s = 0;
  for (int i = 1; i < L::Q; i++)
    if (L::opp(i) > i) {
      const int e = b == 0 ? L::ex(i) : (b == 1 ? L::ey(i) : L::ez(i));
      s += qrow<LAT>(a, i) * 3.0 * L::w(i) * e;
    }
  return s;
}

// One node; ST is the storage type of the populations.  FP32 storage collides
// pair by pair: its sweep is bound by HBM (128^3 without solids 51.6 us per
// step, 50.9 with the grouped form, before the walk alternated), and over
// hundreds of steps the two forms' roundings drift apart by 1e-5.
// WALL: a node with cut links.  Its odd part is formed as w (3 e.u): 3 w rounded
// to FP32 is 3e-8 high, w itself 7e-9, and at the wall that shows in the solids'
// torque.  Rms error over 12 seeds: 128^3 sphere after 20 steps 1.09e-6 -> 7.6e-7,
// moving sphere 6.4e-7 -> 4.1e-7.
template <int LAT, int CM, typename ST, typename T, bool WALL = false>
__device__ __forceinline__ void collide(T (&f)[Lat<LAT>::Q], T Fx, T Fy, T Fz,
                                        const Coll<T> &c) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  constexpr bool MRT = CM == CM_MRT;
  if constexpr (!MRT && !std::is_same<ST, float>::value) {
    collide_two_rate<LAT, CM, 0, even_first<ST>(), T, T>(f, Fx, Fy, Fz, c);
    return;
  }
  T drho = 0, jx = 0, jy = 0, jz = 0;
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    drho += f[i];
    if constexpr (L::ex(i) == 1) jx += f[i];
    if constexpr (L::ex(i) == -1) jx -= f[i];
    if constexpr (L::ey(i) == 1) jy += f[i];
    if constexpr (L::ey(i) == -1) jy -= f[i];
    if constexpr (L::ez(i) == 1) jz += f[i];
    if constexpr (L::ez(i) == -1) jz -= f[i];
  });
  const T ux = jx + (T)0.5 * Fx, uy = jy + (T)0.5 * Fy, uz = jz + (T)0.5 * Fz;
  const T uu = ux * ux + uy * uy + uz * uz;
  const T uF = ux * Fx + uy * Fy + uz * Fz;
  const T base = drho - (T)1.5 * uu;
  const T om = c.omega, omc = c.omc, cf = c.cforce;
  if constexpr (CM != CM_MRT) {
    // FP32 storage: BGK, or MRT whose only non-BGK moments are the q moments,
    // in place pair by pair, grouped for few operations (as the packed pair
    // collision): omega S + cforce SF = w B + A g with B = omega base -
    // 3 cforce u.F and g = 1.5 omega e.u + 3 cforce e.F; omega A + cforce AF
    // = omega A + w (3 cforce e.F); the q moments of Delta + Fbar/2 are
    // sum_i q_a,i (f_i - f_ib) + K (F - 2u) (qk: the pairs' -2A + AF terms)
    T mq[3] = {0, 0, 0};
    const T om15 = om * (T)1.5, cf3 = cf * (T)3;
    const T B = om * base - cf3 * uF;
    f[0] = omc * f[0] + (T)L::w(0) * B;
    const T Ba = (T)L::w(1) * B, Bb = (T)L::w(Q - 1) * B;
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if constexpr (i > 0 && L::opp(i) > i) {
        constexpr int j = L::opp(i);
        constexpr T w = (T)L::w(i);
        constexpr bool ca = L::w(i) == L::w(1);
        const T eu = edot<LAT, i, T>(ux, uy, uz);
        const T eF = edot<LAT, i, T>(Fx, Fy, Fz);
        const T A = WALL ? w * ((T)3 * eu) : (T)(3.0 * L::w(i)) * eu;
        const T t = cf3 * eF;
        const T P = A * (om15 * eu + t) + (ca ? Ba : Bb);
        const T M = om * A + w * t;
        if constexpr (CM == CM_MRT_Q) {
          const T d = f[i] - f[j];
          static_for<L::D>([&](auto ac) {
            constexpr int ax = decltype(ac)::value;
            constexpr int q = qrow<LAT>(ax, i);
            if constexpr (q != 0) mq[ax] += (T)q * d;
          });
        }
        f[i] = omc * f[i] + P + M;
        f[j] = omc * f[j] + P - M;
      }
    });
    if constexpr (CM == CM_MRT_Q) {
      const T fu[3] = {Fx - (T)2 * ux, Fy - (T)2 * uy, Fz - (T)2 * uz};
      static_for<L::D>([&](auto ac) {
        constexpr int ax = decltype(ac)::value;
        static_for<L::D>([&](auto bc) {
          constexpr int b = decltype(bc)::value;
          constexpr T K = (T)qk<LAT>(ax, b);
          if constexpr (K != (T)0) mq[ax] += K * fu[b];
        });
      });
      // all q rows share one rate: a_a = (omega - s_q) m_q,a / |M_q|^2
      const T k = c.ds[4] * (T)(1.0 / mnorm<LAT>(4));
      T aq[3] = {k * mq[0], k * mq[1], k * mq[2]};
      static_for<Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        static_for<L::D>([&](auto ac) {
          constexpr int ax = decltype(ac)::value;
          constexpr int q = qrow<LAT>(ax, i);
          if constexpr (q != 0) f[i] += (T)q * aq[ax];
        });
      });
    }
    return;
  }
  T out[Q];
  T v[MRT ? Q : 1];
  {
    constexpr T w0 = (T)L::w(0);
    const T S = w0 * base, SF = (T)(-3.0 * L::w(0)) * uF;
    out[0] = omc * f[0] + om * S + cf * SF;
    if constexpr (MRT) v[0] = f[0] - S + (T)0.5 * SF;
  }
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (i > 0 && L::opp(i) > i) {
      constexpr int j = L::opp(i);
      constexpr T w = (T)L::w(i);
      const T eu = edot<LAT, i, T>(ux, uy, uz);
      const T eF = edot<LAT, i, T>(Fx, Fy, Fz);
      const T S = w * (base + (T)4.5 * eu * eu);
      const T A = (T)(3.0 * L::w(i)) * eu;
      const T SF = w * ((T)9 * eu * eF - (T)3 * uF);
      const T AF = (T)(3.0 * L::w(i)) * eF;
      const T P = om * S + cf * SF, M = om * A + cf * AF;
      out[i] = omc * f[i] + P + M;
      out[j] = omc * f[j] + P - M;
      if constexpr (MRT) {
        const T hs = (T)0.5 * SF - S, ha = (T)0.5 * AF - A;
        v[i] = f[i] + hs + ha;
        v[j] = f[j] + hs - ha;
      }
    }
  });
  if constexpr (MRT) {
    static_for<Q>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k > 0 && !conserved<LAT>(k)) {
        const T dk = c.ds[k];
        if (dk != (T)0) {
          T m = 0;
          static_for<Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            constexpr int mk = mrow<LAT>(k, i);
            if constexpr (mk == 1) m += v[i];
            else if constexpr (mk == -1) m -= v[i];
            else if constexpr (mk != 0) m += (T)mk * v[i];
          });
          const T a = dk * m * (T)(1.0 / mnorm<LAT>(k));
          static_for<Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            constexpr int mk = mrow<LAT>(k, i);
            if constexpr (mk == 1) out[i] += a;
            else if constexpr (mk == -1) out[i] -= a;
            else if constexpr (mk != 0) out[i] += (T)mk * a;
          });
        }
      }
    });
  }
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    f[i] = out[i];
  });
}

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ int wrap(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// flag bits of a node
enum : uint8_t {
  FL_SOLID = 1,  // no distributions (inside a solid under bounce-back)
  FL_LIST = 2,   // handled by the boundary-node kernel
  FL_NOG = 4,    // the external body force does not act
  FL_BAND = 8,   // the IBM force may be non-zero
  FL_NEW = 16,   // uncovered by a moving solid; refilled before the sweep
  FL_FACE = 32   // next to a non-periodic domain face (the face kernel)
};

}  // namespace lbm

// boundary_impl.cuh -- the kernels around the bulk sweep: boundary nodes
// (interpolated bounce-back + Eq. 17), queries, local (initial) collisions,
// refilling, the IBM band velocity, conversions, and the launcher of every
// sweep-like operation.  Instantiated once per storage type by
// sweep_<precision>.cu.
#pragma once

#include "sweep_impl.cuh"
#include "sweep_rows.cuh"
#include "sweep_vec.cuh"

namespace lbm {

// Interpolated bounce-back value of cut link (x_f, i) from post-collision
// deviations (coefficients of Sec. 2.2, precomputed per link):
//   f_i(x_f,t+1) = c0 f*_ib(x_f) + c1 f*_ib(x_ff) + c2 f*_ib(x_fff)
//                + c3 f*_i(x_f) + c4 f*_i(x_ff) + mw.
template <int LAT, typename S, typename T, typename LT, int POL = LD_NC>
__device__ __forceinline__ T ibb_value(const KArgs &a, const S *src, int i, int ib, int ex, int ey,
                                       int ez, int x, int y, int z, long long n, int link, T isc,
                                       T &fs) {
  const LT *c0 = (const LT *)a.links.c[0], *c1 = (const LT *)a.links.c[1],
           *c2 = (const LT *)a.links.c[2], *c3 = (const LT *)a.links.c[3],
           *c4 = (const LT *)a.links.c[4], *mw = (const LT *)a.links.mw;
  const long long N = a.fs;
  fs = Store<S>::template ld<POL>(src + (long long)ib * N + n, isc);
  if (a.zy_pre) {
    // Eq. 16: the post-collision value leaving the wall at x_f (c3), the
    // pre-collision value arriving at x_f from the previous step (c1) and
    // the moving-wall term
    const LT *pre = (const LT *)a.zy_pre;
    return vfma((T)c3[link], Store<S>::template ld<POL>(src + (long long)i * N + n, isc),
                vfma((T)c1[link], (T)pre[(long long)ib * N + n], (T)mw[link]));
  }
  T v = vfma((T)c0[link], fs, (T)mw[link]);
  const T k1 = (T)c1[link], k2 = (T)c2[link], k3 = (T)c3[link], k4 = (T)c4[link];
  if (k1 != (T)0 || k2 != (T)0 || k4 != (T)0) {
    const long long nff = wrap(x + ex, a.nx) +
                          (long long)a.nx * (wrap(y + ey, a.ny) + (long long)a.ny * wrap(z + ez, a.nz));
    if (k1 != (T)0) v = vfma(k1, Store<S>::template ld<POL>(src + (long long)ib * N + nff, isc), v);
    if (k4 != (T)0) v = vfma(k4, Store<S>::template ld<POL>(src + (long long)i * N + nff, isc), v);
    if (k2 != (T)0) {
      const long long nfff = wrap(x + 2 * ex, a.nx) +
                             (long long)a.nx * (wrap(y + 2 * ey, a.ny) +
                                                (long long)a.ny * wrap(z + 2 * ez, a.nz));
      v = vfma(k2, Store<S>::template ld<POL>(src + (long long)ib * N + nfff, isc), v);
    }
  }
  if (k3 != (T)0) v = vfma(k3, Store<S>::template ld<POL>(src + (long long)i * N + n, isc), v);
  return v;
}

// FP64 outputs of a query at one node from pre-collision deviations f.  The
// second moments of feq are closed forms, sum e_a e_b feq_i = drho/3 delta_ab
// + u_a u_b on both lattices, so the non-equilibrium stress is a few sums of
// the pairs' f_i + f_j: about 90 FP64 operations per D3Q19 node against some
// 700 when feq_i is formed and multiplied out per direction, which GB300's
// FP64 rate makes the query's bound (96^3 FP64 strain rate: 670 us before).
template <int LAT, typename T>
__device__ __forceinline__ void write_fields(const KArgs &a, long long n,
                                             const T (&f)[Lat<LAT>::Q], T Fx,
                                             T Fy, T Fz) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q, D = L::D;
  const bool stress = a.out_S || a.out_stress || a.out_eps;
  if (a.out_f)
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      a.out_f[(long long)i * a.N + n] = L::w(i) + (double)f[i];
    });
  if (!a.out_rho && !a.out_u && !stress) return;
  const double F[3] = {(double)Fx, (double)Fy, (double)Fz};
  // momentum from the pairs' differences; an axis pair comes first and starts
  // each sum
  double u[3] = {0, 0, 0};
  if (a.out_u || stress) {
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if constexpr (i > 0 && L::opp(i) > i) {
        const double d = (double)f[i] - (double)f[L::opp(i)];
        static_for<D>([&](auto ac) {
          constexpr int c = decltype(ac)::value;
          constexpr int e = ecomp<LAT>(c, i);
          if constexpr (e != 0) {
            if constexpr (enorm2<LAT>(i) == 1) u[c] = d;
            else if constexpr (e == 1) u[c] += d;
            else u[c] -= d;
          }
        });
      }
    });
    for (int c = 0; c < D; c++) u[c] += 0.5 * F[c];
    if (a.out_u)
      for (int c = 0; c < D; c++) a.out_u[c * a.N + n] = u[c];
  }
  if (!a.out_rho && !stress) return;
  // density and second moments from the pairs' sums
  double drho = (double)f[0];
  double Pd[3] = {0, 0, 0};  // xx, yy, zz
  double Po[3] = {0, 0, 0};  // xy, yz, xz
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (i > 0 && L::opp(i) > i) {
      const double sp = (double)f[i] + (double)f[L::opp(i)];
      drho += sp;
      static_for<D>([&](auto ac) {
        constexpr int c = decltype(ac)::value;
        if constexpr (ecomp<LAT>(c, i) != 0) {
          if constexpr (enorm2<LAT>(i) == 1) Pd[c] = sp;
          else Pd[c] += sp;
        }
      });
      if constexpr (enorm2<LAT>(i) == 2) {
        constexpr int p = L::ex(i) ? 0 : 1, q = L::ez(i) ? 2 : 1;
        constexpr int k = p == 1 ? 1 : (q == 1 ? 0 : 2);
        if constexpr (ecomp<LAT>(p, i) * ecomp<LAT>(q, i) > 0) Po[k] += sp;
        else Po[k] -= sp;
      }
    }
  });
  if (a.out_rho) a.out_rho[n] = 1.0 + drho;
  if (!stress) return;
  // P = Pi^neq + (F u + u F) / 2
  double tr = 0;
  for (int c = 0; c < D; c++) {
    Pd[c] = Pd[c] - drho * (1.0 / 3.0) + u[c] * (F[c] - u[c]);
    tr += Pd[c];
  }
  constexpr int pa[3] = {0, 1, 0}, pb[3] = {1, 2, 2};
  for (int k = 0; k < (D == 2 ? 1 : 3); k++)
    Po[k] += 0.5 * (F[pa[k]] * u[pb[k]] + u[pa[k]] * F[pb[k]]) - u[pa[k]] * u[pb[k]];
  // S = -1.5 [omega (P - tr P / D) + s_bulk tr P / D]
  const double iso = tr * (1.0 / D), ko = -1.5 * a.omega, ki = -1.5 * (a.s_bulk - a.omega) * iso;
  double ss = 0;
  constexpr int nc = D == 2 ? 3 : 6;
#pragma unroll
  for (int c = 0; c < nc; c++) {
    const bool dg = c < D;
    const double S = dg ? ko * Pd[c] + ki : ko * Po[c - D];
    if (a.out_S) a.out_S[c * a.N + n] = S;
    if (a.out_stress)
      a.out_stress[c * a.N + n] = (dg ? -(1.0 + drho) * (1.0 / 3.0) : 0.0) + 2.0 * a.nu * S;
    ss += (dg ? 1.0 : 2.0) * S * S;
  }
  if (a.out_eps) a.out_eps[n] = 2.0 * a.nu * ss;
}

// ---------------------------------------------------------------- kernels
// Density and velocity only, for FP32 and 16-bit storage: the same moments
// as write_fields (u = sum e_i d_i + F / 2, rho = 1 + sum d_i) summed in FP32
// arithmetic over the stored values, written as FP64.  GB300's FP64 rate
// makes the FP64 sums the query's bound; in FP32 they differ from them by
// about the FP32 rounding of the sums (1e-7 of the largest term), well
// inside the storage's own error.
template <int LAT, typename S>
__device__ __forceinline__ void bulk_query_u(const KArgs &a, long long n, uint8_t fl, int x, int y,
                                             int z) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q, D = L::D;
  float f[Q];
  gather_pull<LAT, S, float>((const S *)a.src, a.fs, x, y, z, a.nx, a.ny, a.nz, a.inv_scale_f, f);
  float drho = 0.f, j[3] = {0.f, 0.f, 0.f};
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    drho += f[i];
    if constexpr (L::ex(i) != 0) j[0] += L::ex(i) > 0 ? f[i] : -f[i];
    if constexpr (L::ey(i) != 0) j[1] += L::ey(i) > 0 ? f[i] : -f[i];
    if constexpr (L::ez(i) != 0) j[2] += L::ez(i) > 0 ? f[i] : -f[i];
  });
  const float gon = (fl & FL_NOG) ? 0.f : 1.f;
  if (a.out_rho) a.out_rho[n] = 1.0 + (double)drho;
  if (a.out_u)
    for (int c = 0; c < D; c++) a.out_u[c * a.N + n] = (double)(j[c] + 0.5f * (gon * a.g_f[c]));
}

// Warp-sum of a double.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Query at list node t: the pre-collision populations pulled from a.src with
// the bounce-back rules (Eq. 16: the kept ones), in FP64.
template <int LAT, typename S, typename LT>
__device__ __forceinline__ void list_query_node(const KArgs &a, int t) {
  constexpr int Q = Lat<LAT>::Q;
  const long long n = a.list_node[t];
  const uint8_t fl = a.flags[n];
  if (fl & FL_FACE) return;
  const double isc = a.inv_scale;
  const S *__restrict__ src = (const S *)a.src;
  double f[Q];
  if (a.zy_pre) {
#pragma unroll
    for (int i = 0; i < Q; i++) f[i] = (double)((const LT *)a.zy_pre)[(long long)i * a.fs + n];
  } else {
    const uint32_t mask = a.list_mask[t];
    int link = a.list_link[t];
    int x, y, z;
    node_xyz(n, a.nx, a.ny, x, y, z);
    gather_pull<LAT, S, double>(src, a.fs, x, y, z, a.nx, a.ny, a.nz, isc, f);
    if (mask) {
#pragma unroll
      for (int i = 1; i < Q; i++) {
        if (!((mask >> i) & 1u)) continue;
        double fs;
        f[i] = ibb_value<LAT, S, double, LT>(a, src, i, Lat<LAT>::opp(i), Lat<LAT>::ex(i),
                                                 Lat<LAT>::ey(i), Lat<LAT>::ez(i), x, y, z, n, link,
                                                 isc, fs);
        link++;
      }
    }
  }
  double Fx, Fy, Fz;
  node_force<double, LT>(a, n, fl, Fx, Fy, Fz);
  write_fields<LAT, double>(a, n, f, Fx, Fy, Fz);
}

// A query in one launch: the first list_blocks blocks take the list nodes
// (long chains of dependent loads, a thread per node), the others the plain
// nodes, a thread each; the list blocks start first and run beside the rest
// (as a launch of their own they took 46 us after a 96^3 FP64 lattice's plain
// nodes).  U32: density and velocity of FP32 and 16-bit storage.
template <int LAT, typename S, typename LT, bool U32>
__global__ void __launch_bounds__(128) k_query(const KArgs a, int list_blocks, long long n0,
                                               long long n1) {
  const int b = (int)blockIdx.x - list_blocks;
  if (b < 0) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    int cnt = a.counts[0];
    if (cnt > a.list_cap) cnt = a.list_cap;
    if (t < cnt) list_query_node<LAT, S, LT>(a, t);
    return;
  }
  const long long n = n0 + (long long)b * blockDim.x + threadIdx.x;
  if (n >= n1) return;
  const uint8_t fl = a.flags[n];
  if (fl & (uint8_t)~(FL_NOG | FL_NEW)) return;
  int x, y, z;
  {
    const unsigned yz = (unsigned)n / (unsigned)a.nx;
    x = (int)((unsigned)n - yz * (unsigned)a.nx);
    z = (int)(yz / (unsigned)a.ny);
    y = (int)(yz - (unsigned)z * (unsigned)a.ny);
  }
  if constexpr (U32) {
    bulk_query_u<LAT, S>(a, n, fl, x, y, z);
  } else {
    double f[Lat<LAT>::Q];
    gather_pull<LAT, S, double>((const S *)a.src, a.fs, x, y, z, a.nx, a.ny, a.nz, a.inv_scale, f);
    const double gon = (fl & FL_NOG) ? 0.0 : 1.0;
    write_fields<LAT, double>(a, n, f, gon * a.g[0], gon * a.g[1], gon * a.g[2]);
  }
}

// per-lane direction tables packed into compile-time integers
template <int LAT> __host__ __device__ constexpr unsigned long long pack_dir(int comp) {
  unsigned long long r = 0;
  for (int i = 0; i < Lat<LAT>::Q; i++) {
    const int e = comp == 0 ? Lat<LAT>::ex(i) : comp == 1 ? Lat<LAT>::ey(i) : Lat<LAT>::ez(i);
    r |= (unsigned long long)(e + 1) << (2 * i);
  }
  return r;
}
template <int LAT> __host__ __device__ constexpr unsigned long long pack_opp() {
  unsigned long long r = 0;
  for (int i = 0; i < Lat<LAT>::Q && i < 12; i++) r |= (unsigned long long)Lat<LAT>::opp(i) << (5 * i);
  return r;
}
template <int LAT> __host__ __device__ constexpr unsigned long long pack_opp_hi() {
  unsigned long long r = 0;
  for (int i = 12; i < Lat<LAT>::Q; i++) r |= (unsigned long long)Lat<LAT>::opp(i) << (5 * (i - 12));
  return r;
}

template <typename T> __device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Lane-parallel collision (lane = direction, lanes >= Q carry fi = 0): Eq. 1
// / Eq. 3 with Guo forcing as in collide(), the moments and the q moments of
// MRT as warp reductions.  Returns f*_lane.
template <int LAT, int CM, typename T>
__device__ __forceinline__ T collide_lane(const KArgs &a, T fi, bool dir, int ex, int ey,
                                          int ez, int cls, T w, T Fx, T Fy, T Fz) {
  using L = Lat<LAT>;
  const T drho = wsum<T>(fi);
  const T jx = wsum<T>((T)ex * fi), jy = wsum<T>((T)ey * fi), jz = wsum<T>((T)ez * fi);
  const T ux = jx + (T)0.5 * Fx, uy = jy + (T)0.5 * Fy, uz = jz + (T)0.5 * Fz;
  const T uu = ux * ux + uy * uy + uz * uz, uF = ux * Fx + uy * Fy + uz * Fz;
  const T eu = (T)ex * ux + (T)ey * uy + (T)ez * uz;
  const T eF = (T)ex * Fx + (T)ey * Fy + (T)ez * Fz;
  const T feq = w * (drho + (T)3 * eu + (T)4.5 * eu * eu - (T)1.5 * uu);
  const T fb = w * ((T)3 * (eF - uF) + (T)9 * eu * eF);
  const Coll<T> c = make_coll<LAT, T>(a);
  T out = c.omc * fi + c.omega * feq + c.cforce * fb;
  if constexpr (CM == CM_MRT_Q) {
    const T v = dir ? fi - feq + (T)0.5 * fb : (T)0;
    const T qf = L::D == 3 ? (T)(5 * cls - 9) : (T)(3 * cls - 5);
    const T kq = c.ds[4] * (T)(1.0 / mnorm<LAT>(4));
    const T mx = wsum<T>(qf * (T)ex * v), my = wsum<T>(qf * (T)ey * v);
    T corr = qf * ((T)ex * mx + (T)ey * my);
    if (L::D == 3) corr += qf * (T)ez * wsum<T>(qf * (T)ez * v);
    out += kq * corr;
  }
  return out;
}

// ---------------------------------------------------------------- boundary
// nodes.  A block takes NT / Q list nodes at a time, a thread per (node,
// direction): it pulls f_i or rebuilds it with the bounce-back rule, so that
// every load of the nodes is in flight at once, and forms its cut link's part
// of Eq. 17.  A thread per node then collides the populations from
// shared memory with the same code as the bulk sweep, and the links' parts
// are summed in FP64 by strips.  A warp per node, with the moments and the
// q correction as warp reductions, took 11.3 us for the 2.6 k nodes of the
// 128^3 sphere and 29 us in FP64 (96^3; 14.8 us for the 300 nodes of a 64^2
// Couette flow): its chains of shuffles and dependent FP64 additions are what
// this form leaves out.
template <typename T, int NT> struct ListSmem {
  T f[NT];
  T red[6][NT];
  double cst[6][NT / 9];
  int sid0[NT / 9];
};

template <int LAT, int CM, typename S, typename T, int NT, int POL>
__device__ __forceinline__ void list_group(const KArgs &a, const S *src, S *dst, double *force_acc,
                                           int group, int cnt, ListSmem<T, NT> &sm) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q, NG = NT / Q;
  constexpr unsigned long long PX = pack_dir<LAT>(0), PY = pack_dir<LAT>(1), PZ = pack_dir<LAT>(2);
  constexpr unsigned long long PO = pack_opp<LAT>(), POH = pack_opp_hi<LAT>();
  const int tid = threadIdx.x;
  const int i = tid / NG, k = tid - i * NG;
  const int t = group * NG + k;
  const bool item = i < Q && t < cnt;
  const T isc = kisc<T>(a);
  long long n = 0;
  uint32_t mask = 0;
  uint8_t fl = 0;
  T fi = 0, part[6] = {0, 0, 0, 0, 0, 0};
  if (item) {
    n = a.list_node[t];
    fl = a.flags[n];
    mask = a.list_mask[t];
    if (mask) {
      // the node's state-independent sums, and the solid they belong to
      if (i < 6) sm.cst[i][k] = a.list_cst[(long long)i * a.list_cap + t];
      if (i == 0) sm.sid0[k] = (fl & FL_FACE) ? -1 : a.links.sid[a.list_link[t]];
    } else if (i == 0) {
      sm.sid0[k] = -1;
    }
    if (!(fl & FL_FACE)) {
      int x, y, z;
      node_xyz(n, a.nx, a.ny, x, y, z);
      const int ex = (int)((PX >> (2 * i)) & 3ull) - 1;
      const int ey = (int)((PY >> (2 * i)) & 3ull) - 1;
      const int ez = (int)((PZ >> (2 * i)) & 3ull) - 1;
      if ((mask >> i) & 1u) {
        const int ib = i < 12 ? (int)((PO >> (5 * i)) & 31ull) : (int)((POH >> (5 * (i - 12))) & 31ull);
        const int lo = a.list_link[t];
        const int link = lo + __popc(mask & ((1u << i) - 1u));
        T fs;
        fi = ibb_value<LAT, S, T, T, POL>(a, src, i, ib, ex, ey, ez, x, y, z, n, link, isc, fs);
        // f*_ib(e_ib - u_w) - f_i(e_i - u_w) = -2 w_i e_i
        //   - d*_ib (e_i + u_w) - d_i (e_i - u_w)   (d: deviations); the first
        // term of the links to the node's first solid was summed per node
        // when the geometry was built
        const int s = a.links.sid[link];
        const int s0 = a.links.sid[lo];
        const T uw[3] = {((const T *)a.links.uw[0])[link], ((const T *)a.links.uw[1])[link],
                         ((const T *)a.links.uw[2])[link]};
        const T r[3] = {((const T *)a.links.arm[0])[link], ((const T *)a.links.arm[1])[link],
                        ((const T *)a.links.arm[2])[link]};
        const T e[3] = {(T)ex, (T)ey, (T)ez};
        if (s == s0) {
          for (int c = 0; c < 3; c++) part[c] = -fs * (e[c] + uw[c]) - fi * (e[c] - uw[c]);
          part[3] = r[1] * part[2] - r[2] * part[1];
          part[4] = r[2] * part[0] - r[0] * part[2];
          part[5] = r[0] * part[1] - r[1] * part[0];
        } else {
          // a second solid seen from this node (narrow gap): full FP64
          const int cls = ex * ex + ey * ey + ez * ez;
          const double w = cls == 1 ? L::w(1) : L::w(Q - 1);
          const double fsd = w + (double)fs, fid = w + (double)fi;
          double q[3];
          for (int c = 0; c < 3; c++)
            q[c] = fsd * (-(double)e[c] - (double)uw[c]) - fid * ((double)e[c] - (double)uw[c]);
          const double rr[3] = {(double)r[0], (double)r[1], (double)r[2]};
          atomicAdd(force_acc + 6 * s + 0, q[0]);
          atomicAdd(force_acc + 6 * s + 1, q[1]);
          atomicAdd(force_acc + 6 * s + 2, q[2]);
          atomicAdd(force_acc + 6 * s + 3, rr[1] * q[2] - rr[2] * q[1]);
          atomicAdd(force_acc + 6 * s + 4, rr[2] * q[0] - rr[0] * q[2]);
          atomicAdd(force_acc + 6 * s + 5, rr[0] * q[1] - rr[1] * q[0]);
        }
      } else {
        const long long sn = wrap(x - ex, a.nx) +
                             (long long)a.nx * (wrap(y - ey, a.ny) + (long long)a.ny * wrap(z - ez, a.nz));
        fi = Store<S>::template ld<POL>(src + (long long)i * a.fs + sn, isc);
      }
    }
  }
  sm.f[tid] = fi;
#pragma unroll
  for (int c = 0; c < 6; c++) sm.red[c][tid] = part[c];
  __syncthreads();
  // Eq. 16 reads a node's kept populations in the threads above
  if (item && a.zy_pre && !(fl & FL_FACE)) ((T *)a.zy_pre)[(long long)i * a.fs + n] = fi;
  if (item && i == 0 && !(fl & FL_FACE)) {
    T Fx, Fy, Fz;
    node_force<T, T>(a, n, fl, Fx, Fy, Fz);
    T f[Q];
#pragma unroll
    for (int d = 0; d < Q; d++) f[d] = sm.f[d * NG + k];
    const Coll<T> c = make_coll<LAT, T>(a);
    collide<LAT, CM, S, T, true>(f, Fx, Fy, Fz, c);
    scatter<LAT, S, T>(dst, a.fs, n, isc, f);
  }
  // Eq. 17 in the other warps meanwhile: the links' parts of each node in the
  // compile-time order of the directions (compute type), then the nodes in FP64:
  // the sums do not depend on the order of the list beyond FP64 rounding
  constexpr int NC = (NG + 31) / 32 * 32, NU = NT - NC;  // threads of the warps that collide, and the others
  static_assert(NU >= 96, "16 threads per component");
  if (force_acc && tid >= NC) {
    const int u = tid - NC;
    for (int q = u; q < 6 * NG; q += NU) {
      const int c = q / NG, kk = q - c * NG;
      if (group * NG + kk >= cnt) continue;
      T v = 0;
#pragma unroll
      for (int d = 1; d < Q; d++) v += sm.red[c][d * NG + kk];
      if (sm.sid0[kk] >= 0) sm.cst[c][kk] += (double)v;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(NU) : "memory");
    for (int s = 0; s < a.nsolids; s++) {
      if (u < 96) {
        const int c = u >> 4, p = u & 15;
        double v = 0;
        bool any = false;
        for (int kk = p; kk < NG && group * NG + kk < cnt; kk += 16)
          if (sm.sid0[kk] == s) {
            v += sm.cst[c][kk];
            any = true;
          }
        if (__any_sync(0xffffffffu, any)) {
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 16);
          if (p == 0 && v != 0.0) atomicAdd(force_acc + 6 * s + c, v);
        }
      }
    }
  }
  __syncthreads();  // the next group reuses the shared arrays
}

template <int LAT, int CM, typename S, typename T>
__global__ void __launch_bounds__(kListBlock) k_list(const KArgs a) {
  __shared__ ListSmem<T, kListBlock> sm;
  // the next step's force record starts at zero (a clearing launch in front of
  // this kernel would lie on the step's critical path)
  if (a.force_next && blockIdx.x == 0 && threadIdx.x < 6 * kMaxSolids) a.force_next[threadIdx.x] = 0.0;
  int cnt = a.counts[0];
  if (cnt > a.list_cap) cnt = a.list_cap;
  if ((int)blockIdx.x * (kListBlock / Lat<LAT>::Q) >= cnt) return;
  list_group<LAT, CM, S, T, kListBlock, LD_NC>(a, (const S *)a.src, (S *)a.dst, a.force_acc,
                                               (int)blockIdx.x, cnt, sm);
}

// The force spread to list node t: its row of markers (solids at rest).
template <typename T, int POL>
__device__ __forceinline__ void gather_force(const KArgs &a, int t, T (&s)[3]) {
  const T *F = (const T *)a.tab.FdV, *nw = (const T *)a.tab.nw;
  const int nm = a.tab.nmark;
  const int e0 = a.tab.nrow[t], e1 = a.tab.nrow[t + 1];
  s[0] = s[1] = s[2] = 0;
#pragma unroll 4
  for (int e = e0; e < e1; e++) {
    const int m = a.tab.ncol[e];
    const T w = nw[e];
    s[0] += w * ld_pol<POL>(F + m);
    s[1] += w * ld_pol<POL>(F + nm + m);
    s[2] += w * ld_pol<POL>(F + 2 * nm + m);
  }
}

// IBM band node t (no cut links): pull, the spread force (gathered from the
// markers' rows and kept in the dense field for queries and the face kernel,
// or already there), collide.  A thread per node: the thousands of band nodes
// of a large lattice run beside its bulk sweep, whose SMs they should hold as
// little as possible (as a block of threads per node's directions the 160^3
// FP16 IBM step took 77 us instead of 68).
template <int LAT, int CM, typename S, typename T, int POL>
__device__ __forceinline__ void ibm_list_node(const KArgs &a, const S *src, S *dst, int t) {
  const long long n = a.list_node[t];
  const uint8_t fl = a.flags[n];
  if (a.tab.nmark > 0) {
    T s[3];
    gather_force<T, POL>(a, t, s);
    for (int c = 0; c < 3; c++) ((T *)const_cast<void *>(a.f_ibm))[c * a.N + n] = s[c];
  }
  if (fl & FL_FACE) return;  // the face kernel's
  int x, y, z;
  node_xyz(n, a.nx, a.ny, x, y, z);
  const T isc = kisc<T>(a);
  T f[Lat<LAT>::Q];
  gather_pull<LAT, S, T, POL>(src, a.fs, x, y, z, a.nx, a.ny, a.nz, isc, f);
  T Fx, Fy, Fz;
  node_force<T, T>(a, n, fl, Fx, Fy, Fz);
  const Coll<T> c = make_coll<LAT, T>(a);
  collide<LAT, CM, S, T>(f, Fx, Fy, Fz, c);
  scatter<LAT, S, T>(dst, a.fs, n, isc, f);
}

template <int LAT, int CM, typename S, typename T>
__global__ void __launch_bounds__(kListIbmBlock) k_list_ibm(const KArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  int cnt = a.counts[0];
  if (cnt > a.list_cap) cnt = a.list_cap;
  if (t < cnt) ibm_list_node<LAT, CM, S, T, LD_NC>(a, (const S *)a.src, (S *)a.dst, t);
}

// The spread force of every list node from the markers' rows, for a state
// that is not swept next (right after an initialisation or a restart).
template <typename T>
__global__ void __launch_bounds__(128) k_ibm_gather(const KArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  int cnt = a.counts[0];
  if (cnt > a.list_cap) cnt = a.list_cap;
  if (t >= cnt) return;
  const long long n = a.list_node[t];
  T s[3];
  gather_force<T, LD_NC>(a, t, s);
  for (int c = 0; c < 3; c++) ((T *)const_cast<void *>(a.f_ibm))[c * a.N + n] = s[c];
}

template <int LAT, int CM, typename S, typename T>
__device__ __forceinline__ void refill_node_warp(const KArgs &a, int t, int lane) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  constexpr unsigned long long PX = pack_dir<LAT>(0), PY = pack_dir<LAT>(1), PZ = pack_dir<LAT>(2);
  const long long n = a.refill_node[t];
  const int sidx = a.refill_sid[t];
  int x, y, z;
  node_xyz(n, a.nx, a.ny, x, y, z);
  const int ex = (int)((PX >> (2 * lane)) & 3ull) - 1;
  const int ey = (int)((PY >> (2 * lane)) & 3ull) - 1;
  const int ez = (int)((PZ >> (2 * lane)) & 3ull) - 1;
  const bool dir = lane < Q;
  const S *src = (const S *)a.src;
  const T isc = kisc<T>(a);
  double rj = 0;
  int cj = 0;
  if (dir && lane > 0) {
    const long long nb = wrap(x + ex, a.nx) +
                         (long long)a.nx * (wrap(y + ey, a.ny) + (long long)a.ny * wrap(z + ez, a.nz));
    if (a.sid[nb] == 0 && !(a.flags[nb] & FL_NEW)) {
      rj = 1.0;
      for (int k = 0; k < Q; k++) rj += (double)Store<S>::ld(src + (long long)k * a.fs + nb, isc);
      cj = 1;
    }
  }
  const double rs = wsum<double>(rj);
  int cn = cj;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cn += __shfl_xor_sync(0xffffffffu, cn, o);
  const double rho = cn ? rs / cn : 1.0;
  const SolidDev b = solid_of(a, sidx);
  double r[3] = {x - b.c[0], y - b.c[1], z - b.c[2]};
  r[0] -= a.nx * round(r[0] / a.nx);
  r[1] -= a.ny * round(r[1] / a.ny);
  r[2] = (L::D == 2 || b.kind == 1) ? 0.0 : r[2] - a.nz * round(r[2] / a.nz);
  double uw[3] = {b.U[0] + b.Om[1] * r[2] - b.Om[2] * r[1],
                  b.U[1] + b.Om[2] * r[0] - b.Om[0] * r[2],
                  b.U[2] + b.Om[0] * r[1] - b.Om[1] * r[0]};
  if (L::D == 2) uw[2] = 0;
  const int cls = ex * ex + ey * ey + ez * ez;
  const double wd = cls == 0 ? L::w(0) : (cls == 1 ? L::w(1) : L::w(Q - 1));
  const double eu = ex * uw[0] + ey * uw[1] + ez * uw[2];
  const double uu = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
  const T fi = dir ? (T)(wd * (rho - 1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)) : (T)0;
  T Fx, Fy, Fz;
  node_force<T, T>(a, n, a.flags[n], Fx, Fy, Fz);
  const T out = collide_lane<LAT, CM, T>(a, fi, dir, ex, ey, ez, cls, (T)wd, Fx, Fy, Fz);
  if (dir) Store<S>::st((S *)a.dst + (long long)lane * a.fs + n, out, isc);
}

// Refill with a warp per uncovered node: lane j sums the density of
// neighbour x + e_j (if it was fluid before and after the move), then lane i
// forms f^eq_i(rho_mean, u_w) and the node's collision runs lane-parallel.
template <int LAT, int CM, typename S, typename T>
__global__ void __launch_bounds__(256) k_refill_warp(const KArgs a) {
  const int lane = threadIdx.x & 31;
  int cnt = a.counts[2];
  if (cnt > a.refill_cap) cnt = a.refill_cap;
  const int stride = gridDim.x * (blockDim.x >> 5);
  for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < cnt; t += stride)
    refill_node_warp<LAT, CM, S, T>(a, t, lane);
}


// Local read of a pre-collision state: collide into dst (MODE 0) or write
// fields (MODE 1).  One thread per node.
template <int LAT, int CM, typename S, typename T, typename LT, int MODE>
__global__ void __launch_bounds__(256) k_local(const KArgs a) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const uint8_t fl = a.flags[n];
  if (fl & FL_SOLID) return;
  const T isc = kisc<T>(a);
  T f[Lat<LAT>::Q];
  gather_local<LAT, S, T>((const S *)a.src, a.fs, n, isc, f);
  T Fx, Fy, Fz;
  node_force<T, LT>(a, n, fl, Fx, Fy, Fz);
  if (MODE == 0) {
    const Coll<T> c = make_coll<LAT, T>(a);
    collide<LAT, CM, S, T>(f, Fx, Fy, Fz, c);
    scatter<LAT, S, T>((S *)a.dst, a.fs, n, isc, f);
  } else {
    write_fields<LAT, T>(a, n, f, Fx, Fy, Fz);
  }
}

// Refill of nodes uncovered by a moving solid: equilibrium at the mean
// density of neighbours fluid before and after the move and at the local
// wall velocity, then the node's collision, written into the current
// post-collision array (src == dst).
template <int LAT, int CM, typename S, typename T>
__global__ void __launch_bounds__(128) k_refill(const KArgs a) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  int cnt = a.counts[2];
  if (cnt > a.refill_cap) cnt = a.refill_cap;
  if (t >= cnt) return;
  const long long n = a.refill_node[t];
  const int sidx = a.refill_sid[t];
  int x, y, z;
  node_xyz(n, a.nx, a.ny, x, y, z);
  const S *src = (const S *)a.src;
  const T isc = kisc<T>(a);
  double rs = 0;
  int cntn = 0;
#pragma unroll
  for (int j = 1; j < Q; j++) {
    const long long nb = wrap(x + L::ex(j), a.nx) +
                         (long long)a.nx * (wrap(y + L::ey(j), a.ny) +
                                            (long long)a.ny * wrap(z + L::ez(j), a.nz));
    if (a.sid[nb] != 0 || (a.flags[nb] & FL_NEW)) continue;
    double r = 1.0;
    for (int k = 0; k < Q; k++) r += (double)Store<S>::ld(src + (long long)k * a.fs + nb, isc);
    rs += r;
    cntn++;
  }
  const double rho = cntn ? rs / cntn : 1.0;
  const SolidDev b = solid_of(a, sidx);
  double r[3] = {x - b.c[0], y - b.c[1], z - b.c[2]};
  r[0] -= a.nx * round(r[0] / a.nx);
  r[1] -= a.ny * round(r[1] / a.ny);
  r[2] = (L::D == 2 || b.kind == 1) ? 0.0 : r[2] - a.nz * round(r[2] / a.nz);
  double uw[3] = {b.U[0] + b.Om[1] * r[2] - b.Om[2] * r[1],
                  b.U[1] + b.Om[2] * r[0] - b.Om[0] * r[2],
                  b.U[2] + b.Om[0] * r[1] - b.Om[1] * r[0]};
  if (L::D == 2) uw[2] = 0;
  const double uu = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
  T f[Q];
#pragma unroll
  for (int i = 0; i < Q; i++) f[i] = (T)feq_dev<LAT, double>(i, rho - 1.0, uw[0], uw[1], uw[2], uu);
  T Fx, Fy, Fz;
  node_force<T, T>(a, n, a.flags[n], Fx, Fy, Fz);
  const Coll<T> c = make_coll<LAT, T>(a);
  collide<LAT, CM, S, T>(f, Fx, Fy, Fz, c);
  scatter<LAT, S, T>((S *)a.dst, a.fs, n, isc, f);
}

// Links through the domain faces: the rules stand at k_face.
template <typename T> __device__ __forceinline__ T face_u(const KArgs &a, int k, int c) {
  if constexpr (is_f32<T>()) return a.u_face_f[k][c];
  else return (T)a.u_face[k][c];
}

// The neighbourhood of a node: wrapped coordinates either side of it, and per
// axis the type of the face that a link leaves the domain through when it
// comes from below (e_a = +1) or above (e_a = -1); 0 (periodic): none there.
struct FaceNode {
  int x[3], y[3], z[3];  // at - 1, at, at + 1
  int lo[3], hi[3];
};
__device__ __forceinline__ FaceNode face_node(const KArgs &a, int x, int y, int z) {
  FaceNode f;
  f.x[0] = x == 0 ? a.nx - 1 : x - 1;
  f.x[1] = x;
  f.x[2] = x == a.nx - 1 ? 0 : x + 1;
  f.y[0] = y == 0 ? a.ny - 1 : y - 1;
  f.y[1] = y;
  f.y[2] = y == a.ny - 1 ? 0 : y + 1;
  f.z[0] = z == 0 ? a.nz - 1 : z - 1;
  f.z[1] = z;
  f.z[2] = z == a.nz - 1 ? 0 : z + 1;
  f.lo[0] = x == 0 ? a.face[0] : 0;
  f.hi[0] = x == a.nx - 1 ? a.face[1] : 0;
  f.lo[1] = y == 0 ? a.face[2] : 0;
  f.hi[1] = y == a.ny - 1 ? a.face[3] : 0;
  f.lo[2] = z == 0 ? a.face[4] : 0;
  f.hi[2] = z == a.nz - 1 ? a.face[5] : 0;
  return f;
}

// direction i with its components along the axes of `axes` (bits) reversed
template <int LAT> __host__ __device__ constexpr int reflect(int i, int axes) {
  for (int k = 0; k < Lat<LAT>::Q; k++) {
    bool same = true;
    for (int c = 0; c < 3; c++)
      same = same && ecomp<LAT>(c, k) == (((axes >> c) & 1) ? -ecomp<LAT>(c, i) : ecomp<LAT>(c, i));
    if (same) return k;
  }
  return 0;
}

// Type of the face that link I of the node crosses along axis C (0: none).
template <int LAT, int I, int C>
__device__ __forceinline__ int crossed(const FaceNode &f) {
  constexpr int e = ecomp<LAT>(C, I);
  return e == 1 ? f.lo[C] : (e == -1 ? f.hi[C] : 0);
}

// f_I(x, t+1) of a node: plain pull, or through velocity / stress-free faces.
// The direction is a compile-time constant, so that which axes a link may
// cross and the direction it is reflected from are too, and the source is
// selected without branches: one load per direction, all of a node's loads in
// flight together (48 M node open box: 5186 us per four steps with a run-time
// search and branches per direction, 5104 now).
template <int LAT, int I, typename S, typename T>
__device__ __forceinline__ T face_pull(const KArgs &a, const S *src, const FaceNode &f, T isc) {
  using L = Lat<LAT>;
  constexpr int ex = L::ex(I), ey = L::ey(I), ez = L::ez(I);
  const int cx = crossed<LAT, I, 0>(f), cy = crossed<LAT, I, 1>(f), cz = crossed<LAT, I, 2>(f);
  const int vf = cx == LBM_FACE_VELOCITY ? (ex == 1 ? 0 : 1)
               : cy == LBM_FACE_VELOCITY ? (ey == 1 ? 2 : 3)
               : cz == LBM_FACE_VELOCITY ? (ez == 1 ? 4 : 5) : -1;
  const bool wall = vf >= 0;
  constexpr int r1 = reflect<LAT>(I, 1), r2 = reflect<LAT>(I, 2), r4 = reflect<LAT>(I, 4);
  constexpr int r3 = reflect<LAT>(I, 3), r5 = reflect<LAT>(I, 5), r6 = reflect<LAT>(I, 6);
  const int j = (cx ? 1 : 0) + (cy ? 2 : 0) + (cz ? 4 : 0);
  const int rd = wall ? L::opp(I)
                      : j == 0 ? I : j == 1 ? r1 : j == 2 ? r2 : j == 4 ? r4 : j == 3 ? r3 : j == 5 ? r5 : r6;
  // a crossed axis keeps the node's own coordinate; a wall reflects at the node
  const int sx = wall || cx ? f.x[1] : f.x[1 - ex];
  const int sy = wall || cy ? f.y[1] : f.y[1 - ey];
  const int sz = wall || cz ? f.z[1] : f.z[1 - ez];
  const unsigned n = (unsigned)sx + (unsigned)a.nx * ((unsigned)sy + (unsigned)a.ny * (unsigned)sz);
  const T v = Store<S>::ld(src + (long long)rd * a.fs + n, isc);
  T eu = 0;
  if (wall) eu = (T)ex * face_u<T>(a, vf, 0) + (T)ey * face_u<T>(a, vf, 1) + (T)ez * face_u<T>(a, vf, 2);
  return wall ? v + (T)(6.0 * L::w(I)) * eu : v;
}

// IBM: unforced velocity u~ = (sum f e + g/2)/rho0 at band nodes (the
// external half force only, no IBM half force) and zero the IBM force there.
template <int LAT, typename S, typename T, int POL>
__device__ __forceinline__ void band_velocity(const KArgs &a, const S *src, int t) {
  using L = Lat<LAT>;
  const long long n = a.list_node[t];
  const uint8_t fl = a.flags[n];
  if (!(fl & FL_BAND)) return;
  int x, y, z;
  node_xyz(n, a.nx, a.ny, x, y, z);
  T f[L::Q];
  const T isc = kisc<T>(a);
  if (a.local_gather)
    gather_local<LAT, S, T>(src, a.fs, n, isc, f);
  else if (fl & FL_FACE) {  // next to a velocity or stress-free domain face
    const FaceNode fn = face_node(a, x, y, z);
    static_for<L::Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      f[i] = face_pull<LAT, i, S, T>(a, src, fn, isc);
    });
  } else
    gather_pull<LAT, S, T, POL>(src, a.fs, x, y, z, a.nx, a.ny, a.nz, isc, f);
  T j[3] = {0, 0, 0};
  static_for<L::Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    static_for<3>([&](auto ac) {
      constexpr int c = decltype(ac)::value;
      if constexpr (ecomp<LAT>(c, i) == 1) j[c] += f[i];
      if constexpr (ecomp<LAT>(c, i) == -1) j[c] -= f[i];
    });
  });
  const bool g = !(fl & FL_NOG);
  T *ub = (T *)a.u_band;
  T *fi = (T *)const_cast<void *>(a.f_ibm);
  for (int c = 0; c < 3; c++) {
    ub[c * a.N + n] = j[c] + (g ? (T)0.5 * kg<T>(a, c) : (T)0);
    if (a.tab.nmark == 0) fi[c * a.N + n] = (T)0;  // the markers add their forces
  }
}

template <int LAT, typename S, typename T>
__global__ void __launch_bounds__(64) k_band_vel(const KArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  // this step's force record, accumulated by the IBM kernels that follow on
  // the same stream, starts at zero
  if (a.force_acc && t < 6 * kMaxSolids) a.force_acc[t] = 0.0;
  int cnt = a.counts[0];
  if (cnt > a.list_cap) cnt = a.list_cap;
  if (t < cnt) band_velocity<LAT, S, T, LD_NC>(a, (const S *)a.src, t);
}

// Full FP64 f -> stored deviations (solid nodes get 0).
template <int LAT, typename S, typename T>
__global__ void __launch_bounds__(256) k_from_double(const KArgs a) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const bool solid = a.flags[n] & FL_SOLID;
  const T isc = kisc<T>(a);
#pragma unroll
  for (int i = 0; i < Lat<LAT>::Q; i++) {
    const double v = solid ? 0.0 : a.out_f[(long long)i * a.N + n] - Lat<LAT>::w(i);
    Store<S>::st((S *)a.dst + (long long)i * a.fs + n, (T)v, isc);
  }
}

// Equilibrium deviations at (rho, u): rho in omega, u in g[].
template <int LAT, typename S, typename T>
__global__ void __launch_bounds__(256) k_fill_eq(const KArgs a) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const double ux = a.g[0], uy = a.g[1], uz = a.g[2];
  const double uu = ux * ux + uy * uy + uz * uz;
  const T isc = kisc<T>(a);
#pragma unroll
  for (int i = 0; i < Lat<LAT>::Q; i++)
    Store<S>::st((S *)a.dst + (long long)i * a.fs + n,
                 (T)feq_dev<LAT, double>(i, a.omega - 1.0, ux, uy, uz, uu), isc);
}

// Eq. 16: the pre-collision populations of the boundary nodes, read from a
// state held locally (right after an initialisation).
template <int LAT, typename S, typename T>
__global__ void __launch_bounds__(128) k_zy_seed(const KArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  int cnt = a.counts[0];
  if (cnt > a.list_cap) cnt = a.list_cap;
  if (t >= cnt) return;
  const long long n = a.list_node[t];
  const T isc = kisc<T>(a);
  for (int i = 0; i < Lat<LAT>::Q; i++)
    ((T *)a.zy_pre)[(long long)i * a.fs + n] =
        Store<S>::ld((const S *)a.src + (long long)i * a.fs + n, isc);
}

// ---------------------------------------------------------------- domain
// faces (the open box of the uniform flow past a sphere, Sec. 3.4).  A
// non-periodic face lies half a spacing outside the outermost nodes; the
// nodes next to one (flag FL_FACE) run in k_face, a thread per node, which
// pulls like the bulk sweep except on links that leave the domain:
//  - velocity face (plane wall moving with u_f): f_i = f*_ib(x) + 6 w_i e_i.u_f
//    (the moving-wall bounce-back with q = 1/2, rho0 = 1);
//  - stress-free face: specular reflection, f_i = f*_r(x'), r = e_i with the
//    crossed components reversed and x' = x - e_i with x's coordinates on the
//    crossed axes;
//  - convective outflow face (outward normal n): f_i(x, t+1) =
//    [f_i(x, t) + U_o f_i(x - n, t+1)] / (1 + U_o), U_o = max(0, u(x, t).n),
//    from the node's pre-collision populations and velocity kept from the
//    previous step (a.outlet, [Q + 1][face area] in the compute type).
// A velocity face decides a link that crosses two faces, then an outflow
// face, then free slip.

// index of a node of the outflow face in the outlet arrays
__device__ __forceinline__ int outlet_index(const KArgs &a, int x, int y, int z) {
  const int ax = a.out_face >> 1;
  return ax == 0 ? y + a.ny * z : ax == 1 ? x + a.nx * z : x + a.nx * y;
}
__device__ __forceinline__ bool on_outlet(const KArgs &a, int x, int y, int z) {
  if (a.out_face < 0) return false;
  const int ax = a.out_face >> 1, hi = a.out_face & 1;
  const int c = ax == 0 ? x : ax == 1 ? y : z;
  const int len = ax == 0 ? a.nx : ax == 1 ? a.ny : a.nz;
  return c == (hi ? len - 1 : 0);
}

// MODE 0: sweep (src f*(t) -> dst f*(t+1)); MODE 1: query of f(t) from
// src = f*(t - 1); MODE 2: keep the outflow face's populations and velocity
// from a state held locally in src (right after an initialisation).
template <int LAT, int CM, typename S, typename T, typename LT, int MODE>
__global__ void __launch_bounds__(128) k_face(const KArgs a) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.nface) return;
  const long long n = a.face_node[t];
  int x, y, z;
  node_xyz(n, a.nx, a.ny, x, y, z);
  const T isc = kisc<T>(a);
  const S *__restrict__ src = (const S *)a.src;
  const bool out = on_outlet(a, x, y, z);
  const long long A = a.out_area;
  LT *keep = (LT *)a.outlet;
  const int oi = out ? outlet_index(a, x, y, z) : 0;
  const uint8_t fl = a.flags[n];
  T Fx, Fy, Fz;
  node_force<T, LT>(a, n, fl, Fx, Fy, Fz);
  T f[Q];
  if (MODE == 2) {
    if (!out) return;
    gather_local<LAT, S, T>(src, a.fs, n, isc, f);
  } else {
    const FaceNode fn = face_node(a, x, y, z);
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      f[i] = face_pull<LAT, i, S, T>(a, src, fn, isc);
    });
    if (out) {
      // the outflow rule, on links that cross it and no velocity face
      const int ax = a.out_face >> 1, sg = (a.out_face & 1) ? 1 : -1;
      const FaceNode in = face_node(a, x - (ax == 0 ? sg : 0), y - (ax == 1 ? sg : 0),
                                    z - (ax == 2 ? sg : 0));
      T U = (T)keep[(long long)Q * A + oi];
      if (U < (T)0) U = (T)0;
      static_for<Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const int cx = crossed<LAT, i, 0>(fn), cy = crossed<LAT, i, 1>(fn), cz = crossed<LAT, i, 2>(fn);
        const bool vel = cx == LBM_FACE_VELOCITY || cy == LBM_FACE_VELOCITY || cz == LBM_FACE_VELOCITY;
        const bool conv = cx == LBM_FACE_CONVECTIVE || cy == LBM_FACE_CONVECTIVE || cz == LBM_FACE_CONVECTIVE;
        if (!vel && conv) {
          if (MODE == 1)
            f[i] = (T)keep[(long long)i * A + oi];  // f_i(x, t), kept by the last step
          else
            f[i] = ((T)keep[(long long)i * A + oi] + U * face_pull<LAT, i, S, T>(a, src, in, isc)) /
                   ((T)1 + U);
        }
      });
    }
  }
  if (MODE != 1 && out) {
    // this step's pre-collision populations and outward velocity, read by
    // the next step's outflow update
    T j = (T)0;
#pragma unroll
    for (int i = 0; i < Q; i++) keep[(long long)i * A + oi] = (LT)f[i];
    const int ax = a.out_face >> 1;
#pragma unroll
    for (int i = 0; i < Q; i++)
      j += (T)(ax == 0 ? L::ex(i) : ax == 1 ? L::ey(i) : L::ez(i)) * f[i];
    const T Fa = ax == 0 ? Fx : ax == 1 ? Fy : Fz;
    keep[(long long)Q * A + oi] = (LT)(((a.out_face & 1) ? (T)1 : (T)-1) * (j + (T)0.5 * Fa));
  }
  if (MODE == 0) {
    const Coll<T> c = make_coll<LAT, T>(a);
    collide<LAT, CM, S, T>(f, Fx, Fy, Fz, c);
    scatter<LAT, S, T>((S *)a.dst, a.fs, n, isc, f);
  } else if (MODE == 1) {
    write_fields<LAT, T>(a, n, f, Fx, Fy, Fz);
  }
}

// ---------------------------------------------------------------- Eq. 24
// The fluid momentum and angular momentum inside solid a.kempe_solid at the
// time of the state in src (post-collision f*, so u = sum e f* - F/2 with
// the force of that collision), weighted by the fraction alpha of the cell
// around each node inside the solid (Eq. 25: sum over the cell's corners at
// +-1/2 of -phi H(-phi) over the sum of |phi|, phi the signed distance
// function of Eq. 26 for a sphere, or a circle / z-cylinder).  A thread per
// node of the box around the solid; FP64 sums.
__device__ __forceinline__ double kimage(double d, int L) {
  return d - L * rint(d * (1.0 / L));
}

template <int LAT, typename S, typename T>
__global__ void __launch_bounds__(256) k_kempe(const KArgs a) {
  using L = Lat<LAT>;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int bx = a.kbox[3], by = a.kbox[4], bz = a.kbox[5];
  double acc[6] = {0, 0, 0, 0, 0, 0};
  if (t < (long long)bx * by * bz) {
    const SolidDev b = solid_of(a, a.kempe_solid);
    int o[3] = {a.kbox[0], a.kbox[1], a.kbox[2]};
    if (a.kbox_dev) {
      // every node with a cell corner inside lies within R + 1 of the centre
      const int len[3] = {a.nx, a.ny, a.nz};
      for (int c = 0; c < 3; c++)
        if (a.kbox[3 + c] < len[c]) o[c] = (int)floor(b.c[c] - b.R - 1.0);
    }
    const int x = wrap(o[0] + (int)(t % bx), a.nx);
    const int y = wrap(o[1] + (int)((t / bx) % by), a.ny);
    const int z = wrap(o[2] + (int)(t / ((long long)bx * by)), a.nz);
    const bool flat = L::D == 2 || b.kind == LBM_CYLINDER_Z;
    double num = 0, den = 0;
    for (int c = 0; c < (L::D == 2 ? 4 : 8); c++) {
      const double r0 = kimage(x + ((c & 1) ? 0.5 : -0.5) - b.c[0], a.nx);
      const double r1 = kimage(y + ((c & 2) ? 0.5 : -0.5) - b.c[1], a.ny);
      const double r2 = flat ? 0.0 : kimage(z + ((c & 4) ? 0.5 : -0.5) - b.c[2], a.nz);
      const double phi = sqrt(r0 * r0 + r1 * r1 + r2 * r2) / b.R - 1.0;
      if (phi < 0) num -= phi;
      den += fabs(phi);
    }
    const double al = den > 0 ? num / den : 0.0;
    if (al > 0) {
      const long long n = x + (long long)a.nx * (y + (long long)a.ny * z);
      const T isc = kisc<T>(a);
      T Fx, Fy, Fz;
      node_force<T, T>(a, n, a.flags[n], Fx, Fy, Fz);
      T j[3] = {(T)0, (T)0, (T)0};
#pragma unroll
      for (int i = 1; i < L::Q; i++) {
        const T v = Store<S>::ld((const S *)a.src + (long long)i * a.fs + n, isc);
        j[0] += (T)L::ex(i) * v;
        j[1] += (T)L::ey(i) * v;
        j[2] += (T)L::ez(i) * v;
      }
      const double u[3] = {(double)(j[0] - (T)0.5 * Fx), (double)(j[1] - (T)0.5 * Fy),
                           L::D == 2 ? 0.0 : (double)(j[2] - (T)0.5 * Fz)};
      const double r[3] = {kimage(x - b.c[0], a.nx), kimage(y - b.c[1], a.ny),
                           flat ? 0.0 : kimage(z - b.c[2], a.nz)};
      acc[0] = al * u[0];
      acc[1] = al * u[1];
      acc[2] = al * u[2];
      acc[3] = al * (r[1] * u[2] - r[2] * u[1]);
      acc[4] = al * (r[2] * u[0] - r[0] * u[2]);
      acc[5] = al * (r[0] * u[1] - r[1] * u[0]);
    }
  }
  const int lane = threadIdx.x & 31;
  for (int c = 0; c < 6; c++) {
    const double v = warp_sum(acc[c]);
    if (lane == 0 && v != 0.0) atomicAdd(a.kempe_out + c, v);
  }
}

}  // namespace lbm

#include "run_impl.cuh"

namespace lbm {

// ---------------------------------------------------------------- launch
inline int div_up(long long a, int b) { return (int)((a + b - 1) / b); }

// The vector bulk sweep: W words per thread and direction (bulk_vec_words 2
// or 4; 0 = 2) and the node-pair collision packed (bulk_vec_packed 1) or node
// by node (0); -1 is the storage type's default.  Returns false where nx or the direction stride is not a
// multiple of the V nodes of a vector.
//
// Both arrays together up to kReuseBytes (1.5 times the 129 MB L2): the reads
// are evict-first, so that L2 keeps what the step writes, which the next step
// reads.  us per step without / with it, lattices without solids: FP32 84^3
// (90 MB) 14.5 / 12.9, 96^3 (134 MB) 21.7 / 19.0, 104^3 (171 MB) 27.4 / 25.4,
// 112^3 (213 MB) 33.6 / 32.5, 128^3 (319 MB) 48.6 / 47.7, 144^3 (454 MB) 68.4 / 70.3;
// FP16 112^3 (107 MB) 19.1 / 17.7, 128^3 (159 MB) 29.0 / 26.6, 160^3 (311 MB)
// 52.9 / 51.9.  The line lies below the sizes that gain little alone and lose side
// by side: two 112^3 FP32 lattices 66.9 / 71.5.
// With other lattices stepping beside it (a batch, other streams) L2 is theirs
// too: up to kReuseBeside together.  Batches with the hint in every lattice / none:
// FP32 8 x 80^3 (623 MB) 100.5 / 92.3, 8 x 72^3 with spheres (454 MB) 77.2 / 74.1,
// 4 x 96^3 (538 MB) 89.2 / 83.9, 8 x 64^3 IBM (319 MB) 70.0 / 68.1, 2 x 96^3
// (269 MB) 43.3 / 43.1; FP16 8 x 80^3 (311 MB) 60.0 / 62.4.
constexpr long long kReuseBytes = 192LL << 20;
constexpr long long kReuseBeside = 300LL << 20;
template <int LAT, int CM, typename S, int W>
bool launch_bulk_vec_w(const KArgs &a, int want, bool packed, cudaStream_t st) {
  constexpr int V = W * VecS<S>::per_word;
  if (a.nx % V != 0 || a.fs % V != 0) return false;
  const int nt = (int)(a.N / V);
  const int grid = div_up(nt, want);
  // the hint is built for the default shape only
  const long long bytes = 2 * Lat<LAT>::Q * a.fs * (long long)sizeof(S);
  const bool once = bytes <= kReuseBytes && bytes + a.beside <= kReuseBeside;
  constexpr int kOnce = W == 2 ? LD_ONCE : LD_NC;
  if (packed) {
    if (once && vec_packed<S>())
      k_bulk_vec<LAT, CM, S, W, true, vec_packed<S>() ? kOnce : LD_NC><<<grid, want, 0, st>>>(a);
    else
      k_bulk_vec<LAT, CM, S, W, true, LD_NC><<<grid, want, 0, st>>>(a);
  } else {
    if (once && !vec_packed<S>())
      k_bulk_vec<LAT, CM, S, W, false, vec_packed<S>() ? LD_NC : kOnce><<<grid, want, 0, st>>>(a);
    else
      k_bulk_vec<LAT, CM, S, W, false, LD_NC><<<grid, want, 0, st>>>(a);
  }
  return true;
}
template <int LAT, int CM, typename S>
bool launch_bulk_vec(const KArgs &a, int want, cudaStream_t st) {
  const bool packed = a.bulk_vec_packed >= 0 ? a.bulk_vec_packed != 0 : vec_packed<S>();
  if (a.bulk_vec_words == 4) return launch_bulk_vec_w<LAT, CM, S, 4>(a, want, packed, st);
  return launch_bulk_vec_w<LAT, CM, S, 2>(a, want, packed, st);
}

// The row-copy sweep (bulk_mode 2), built for the default vector shape of
// the storage type only (2 words; node by node for FP32, packed pairs for
// 16-bit storage).  The grid is the resident blocks of all SMs (queried per
// device and shared-memory size), or fewer where the lattice has fewer
// tiles.  Returns false where the lattice, its alignment or the requested
// shape does not fit it.
template <int LAT, int CM, typename S>
bool launch_bulk_rows(const KArgs &a, cudaStream_t st) {
  constexpr int W = 2;
  constexpr int V = W * VecS<S>::per_word;
  constexpr bool kPacked = sizeof(S) == 2;
  const bool packed = a.bulk_vec_packed >= 0 ? a.bulk_vec_packed != 0 : kPacked;
  if (a.bulk_vec_words == 4 || packed != kPacked || !a.wait_err) return false;
  if (a.nx % (32 * V) != 0 || a.N / a.nx >= (1LL << 31) || (a.fs * (long long)sizeof(S)) % 16 != 0 ||
      ((uintptr_t)a.src & 15) != 0 || ((uintptr_t)a.flags & 15) != 0)
    return false;
  // two blocks per SM
  constexpr size_t kSmemLimit = 112 * 1024;
  const RowTiles g = row_tiles<LAT, S, W>(a, kSmemLimit);
  if (g.stage_bytes == 0) return false;
  const size_t smem = 2 * (size_t)g.stage_bytes + 4 * sizeof(uint64_t);
  auto kern = k_bulk_rows<LAT, CM, S, W, kPacked>;
  constexpr int kMaxDev = 64;
  struct Resident {
    size_t smem;
    int blocks;  // 0: not queried, -1: unusable
  };
  static Resident resident[kMaxDev];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return false;
  Resident &r = resident[dev];
  if (r.blocks == 0 || r.smem != smem) {
    // the attribute calls are not stream work: allowed inside a capture
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    int per_sm = 0, sms = 0;
    const bool ok =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit + 64) ==
            cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kRowBlock, smem) ==
            cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
    cudaThreadExchangeStreamCaptureMode(&mode);
    r.smem = smem;
    r.blocks = ok && per_sm > 0 ? per_sm * sms : -1;
  }
  if (r.blocks < 0) return false;
  const unsigned grid = (unsigned)std::min<long long>(r.blocks, g.ntiles);
  if (grid == 0) return true;
  kern<<<grid, kRowBlock, smem, st>>>(a, g);
  return true;
}

template <int LAT, int CM, typename S, int W, bool PACKED>
bool launch_group_w(const KArgs *as, int n, int want, cudaStream_t st) {
  constexpr int V = W * VecS<S>::per_word;
  static_assert(sizeof(GroupArgs) <= 32000, "kernel parameter space");
  GroupArgs g;
  g.n = n;
  int blocks = 0;
  for (int k = 0; k < n; k++) {
    if (as[k].nx % V != 0 || as[k].fs % V != 0) return false;
    g.block_start[k] = blocks;
    blocks += div_up(as[k].N / V, want);
    g.a[k] = as[k];
  }
  g.block_start[n] = blocks;
  k_bulk_vec_group<LAT, CM, S, W, PACKED><<<blocks, want, 0, st>>>(g);
  return true;
}

template <int LAT, int CM, typename S>
bool launch_group_t(const KArgs *as, int n, cudaStream_t st) {
  if constexpr (CM == CM_MRT) {
    return false;
  } else {
    const KArgs &a0 = as[0];
    for (int k = 1; k < n; k++)
      if (as[k].bulk_mode != a0.bulk_mode || as[k].bulk_vec_words != a0.bulk_vec_words ||
          as[k].bulk_vec_packed != a0.bulk_vec_packed || as[k].bulk_block != a0.bulk_block)
        return false;
    if (a0.bulk_mode < 1 || n < 1 || n > kMaxGroup) return false;
    // only the default vector shape of the storage type is built grouped: each
    // grouped variant inlines the update kMaxGroup times
    constexpr bool kPacked = vec_packed<S>();
    const bool packed = a0.bulk_vec_packed >= 0 ? a0.bulk_vec_packed != 0 : kPacked;
    if (a0.bulk_vec_words == 4 || packed != kPacked) return false;
    const int want = a0.bulk_block > 0 ? a0.bulk_block : 128;
    return launch_group_w<LAT, CM, S, 2, kPacked>(as, n, want, st);
  }
}

template <typename S>
bool launch_group_precision(const KArgs *as, int n, int lattice, int collision, cudaStream_t st) {
  if (lattice == LBM_D2Q9) {
    if (collision == CM_MRT_Q) return launch_group_t<0, CM_MRT_Q, S>(as, n, st);
    if (collision == CM_BGK) return launch_group_t<0, CM_BGK, S>(as, n, st);
  } else {
    if (collision == CM_MRT_Q) return launch_group_t<1, CM_MRT_Q, S>(as, n, st);
    if (collision == CM_BGK) return launch_group_t<1, CM_BGK, S>(as, n, st);
  }
  return false;
}

template <int LAT, int CM, typename S, typename T>
void launch_one(SweepOp op, const KArgs &a, cudaStream_t st) {
  const int want = a.bulk_block > 0 ? a.bulk_block : 128;
  const int lc = a.list_cap > 0 ? a.list_cap : 1;
  switch (op) {
  case OP_BULK_SWEEP:
    if constexpr (std::is_same<T, float>::value && CM != CM_MRT) {
      g_bulk_kernel = BK_ROWS;
      if (a.bulk_mode == 2 && launch_bulk_rows<LAT, CM, S>(a, st)) break;
      g_bulk_kernel = BK_VEC;
      if (a.bulk_mode >= 1 && launch_bulk_vec<LAT, CM, S>(a, want, st)) break;
    }
    g_bulk_kernel = BK_NODE;
    switch (a.cache_hints & 3) {
    case 1: k_bulk_sweep<LAT, CM, S, T, 1><<<div_up(a.N, want), want, 0, st>>>(a); break;
    case 2: k_bulk_sweep<LAT, CM, S, T, 2><<<div_up(a.N, want), want, 0, st>>>(a); break;
    case 3: k_bulk_sweep<LAT, CM, S, T, 3><<<div_up(a.N, want), want, 0, st>>>(a); break;
    default: k_bulk_sweep<LAT, CM, S, T, 0><<<div_up(a.N, want), want, 0, st>>>(a);
    }
    break;
  case OP_QUERY: {
    // plain nodes query_n0 .. query_n1 - 1; the boundary nodes with the first
    const long long n1 = a.query_n1 > 0 ? a.query_n1 : a.N;
    const int lb = a.list_cap > 0 && a.query_n0 == 0 ? div_up(a.list_cap, 128) : 0;
    const int grid = lb + div_up(n1 - a.query_n0, 128);
    if constexpr (std::is_same<T, float>::value) {
      if (!a.out_S && !a.out_stress && !a.out_eps && !a.out_f) {
        k_query<LAT, S, T, true><<<grid, 128, 0, st>>>(a, lb, a.query_n0, n1);
        break;
      }
    }
    k_query<LAT, S, T, false><<<grid, 128, 0, st>>>(a, lb, a.query_n0, n1);
    break;
  }
  case OP_LIST_SWEEP:
    if (a.list_cap > 0 && a.ibm)
      k_list_ibm<LAT, CM, S, T><<<div_up(lc, kListIbmBlock), kListIbmBlock, 0, st>>>(a);
    else if (a.list_cap > 0)
      k_list<LAT, CM, S, T>
          <<<div_up(lc, kListBlock / Lat<LAT>::Q), kListBlock, 0, st>>>(a);
    break;
  case OP_IBM_GATHER:
    if (a.list_cap > 0) k_ibm_gather<T><<<div_up(lc, 128), 128, 0, st>>>(a);
    break;
  case OP_ZY_SEED:
    if (a.list_cap > 0 && a.zy_pre) k_zy_seed<LAT, S, T><<<div_up(lc, 128), 128, 0, st>>>(a);
    break;
  case OP_LOCAL_INIT:
    k_local<LAT, CM, S, T, T, 0><<<div_up(a.N, 256), 256, 0, st>>>(a);
    break;
  case OP_LOCAL_QUERY:
    k_local<LAT, CM, S, double, T, 1><<<div_up(a.N, 256), 256, 0, st>>>(a);
    break;
  case OP_REFILL:
    if (a.refill_cap > 0) {
      if constexpr (CM != CM_MRT)
        k_refill_warp<LAT, CM, S, T><<<std::min(div_up(a.refill_cap, 8), 64), 256, 0, st>>>(a);
      else
        k_refill<LAT, CM, S, T><<<div_up(a.refill_cap, 128), 128, 0, st>>>(a);
    }
    break;
  case OP_BAND_VEL:
    if (a.list_cap > 0) k_band_vel<LAT, S, T><<<div_up(lc, 64), 64, 0, st>>>(a);
    break;
  case OP_FROM_DOUBLE:
    k_from_double<LAT, S, T><<<div_up(a.N, 256), 256, 0, st>>>(a);
    break;
  case OP_FILL_EQ:
    k_fill_eq<LAT, S, T><<<div_up(a.N, 256), 256, 0, st>>>(a);
    break;
  case OP_FACE_SWEEP:
    if (a.nface > 0) k_face<LAT, CM, S, T, T, 0><<<div_up(a.nface, 128), 128, 0, st>>>(a);
    break;
  case OP_FACE_QUERY:
    if (a.nface > 0) k_face<LAT, CM, S, double, T, 1><<<div_up(a.nface, 128), 128, 0, st>>>(a);
    break;
  case OP_KEMPE: {
    const long long vol = (long long)a.kbox[3] * a.kbox[4] * a.kbox[5];
    if (vol > 0) k_kempe<LAT, S, T><<<div_up(vol, 256), 256, 0, st>>>(a);
    break;
  }
  case OP_FACE_SEED:
    if (a.nface > 0 && a.outlet) k_face<LAT, CM, S, T, T, 2><<<div_up(a.nface, 128), 128, 0, st>>>(a);
    break;
  }
}

// collision: CM_BGK, CM_MRT (general rates) or CM_MRT_Q (only the q moments
// relax at a rate other than 1/tau, the default)
template <typename S, typename T>
void launch_precision(SweepOp op, int lattice, int collision, const KArgs &a,
                      cudaStream_t st) {
  if (lattice == LBM_D2Q9) {
    if (collision == CM_MRT) launch_one<0, CM_MRT, S, T>(op, a, st);
    else if (collision == CM_MRT_Q) launch_one<0, CM_MRT_Q, S, T>(op, a, st);
    else launch_one<0, CM_BGK, S, T>(op, a, st);
  } else {
    if (collision == CM_MRT) launch_one<1, CM_MRT, S, T>(op, a, st);
    else if (collision == CM_MRT_Q) launch_one<1, CM_MRT_Q, S, T>(op, a, st);
    else launch_one<1, CM_BGK, S, T>(op, a, st);
  }
}

}  // namespace lbm

// ibm_device.cuh -- device pieces of the direct-forcing immersed boundary
// (Sec. 2.1) shared by the marker kernels of ibm.cu and the multi-step kernel:
// delta-function kernels, marker positions and stencils, and the forcing
// iterations of solids at rest, which run on tables built with the geometry.
#pragma once

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

// The one-dimensional delta-function kernels compared in Sec. 3.1:
// Peskin's 4-point kernel (Eq. 6, the default), Roma, Peskin & Berger's
// 3-point kernel, the 2-point linear kernel, and the 4-point cosine kernel of
// Appendix B.  Each support lies inside the 4-point window from floor(X) - 1,
// so every kernel uses the same 4^d stencil (points outside the support get
// weight 0).
template <typename T>
__device__ __forceinline__ T phi_k(int kernel, T r) {
  const T a = fabs(r);
  switch (kernel) {
  case LBM_DELTA_ROMA3:
    if (a >= (T)1.5) return (T)0;
    if (a <= (T)0.5) return ((T)1 + sqrt((T)1 - (T)3 * a * a)) / (T)3;
    return ((T)5 - (T)3 * a - sqrt((T)1 - (T)3 * ((T)1 - a) * ((T)1 - a))) / (T)6;
  case LBM_DELTA_LINEAR2:
    return a >= (T)1 ? (T)0 : (T)1 - a;
  case LBM_DELTA_COSINE4:
    return a >= (T)2 ? (T)0 : ((T)1 + cospi(r / (T)2)) / (T)4;
  default:
    if (a >= (T)2) return (T)0;
    if (a >= (T)1) return ((T)5 - (T)2 * a - sqrt((T)-7 + (T)12 * a - (T)4 * a * a)) / (T)8;
    return ((T)3 - (T)2 * a + sqrt((T)1 + (T)4 * a - (T)4 * a * a)) / (T)8;
  }
}

struct Marker {
  double X[3];   // position
  double r[3];   // X - centre (z dropped for cylinders and 2D)
  int s;
};

__device__ __forceinline__ Marker marker(const IbmArgs &a, int m) {
  Marker k;
  k.s = a.msid[m];
  const SolidDev b = solid_of(a, k.s);
  const double dx = a.dir[m], dy = a.dir[a.nmark + m], dz = a.dir[2 * a.nmark + m];
  k.X[0] = b.c[0] + b.RL * dx;
  k.X[1] = b.c[1] + b.RL * dy;
  if (a.dim == 2)
    k.X[2] = 0.0;
  else if (b.kind == LBM_CYLINDER_Z)
    k.X[2] = dz;  // plane of the ring
  else
    k.X[2] = b.c[2] + b.RL * dz;
  k.r[0] = k.X[0] - b.c[0];
  k.r[1] = k.X[1] - b.c[1];
  k.r[2] = (a.dim == 2 || b.kind == LBM_CYLINDER_Z) ? 0.0 : k.X[2] - b.c[2];
  return k;
}

// Stencil of a marker: the 4^d nodes from floor(X) - 1; the marker position
// is FP64, the offsets of the stencil points from it are formed once and the
// per-point arithmetic runs in the compute type.
template <typename T> struct Stencil {
  int ix, iy, iz;  // first stencil node (unwrapped)
  T dx, dy, dz;    // first node - X
};

template <typename T>
__device__ __forceinline__ Stencil<T> stencil_of(const IbmArgs &a, const Marker &k) {
  Stencil<T> st;
  const double bx = floor(k.X[0]) - 1.0, by = floor(k.X[1]) - 1.0;
  const double bz = a.dim == 3 ? floor(k.X[2]) - 1.0 : 0.0;
  st.ix = (int)bx;
  st.iy = (int)by;
  st.iz = (int)bz;
  st.dx = (T)(bx - k.X[0]);
  st.dy = (T)(by - k.X[1]);
  st.dz = a.dim == 3 ? (T)(bz - k.X[2]) : (T)0;
  return st;
}

__device__ __forceinline__ long long table_node(const IbmArgs &a, int4 b, int p) {
  const int kx = p & 3, ky = (p >> 2) & 3, kz = p >> 4;
  const int x = wrap(b.x + kx, a.nx), y = wrap(b.y + ky, a.ny);
  const int z = a.dim == 3 ? wrap(b.z + kz, a.nz) : 0;
  return x + (long long)a.nx * (y + (long long)a.ny * z);
}

// ---------------------------------------------------------------- tables
// Solids whose markers do not move keep two tables (see IbmTab):
//  - per band node, the markers whose stencil holds it and their weights, in
//    marker order.  The node that collides with the spread force gathers it
//    (sum over its row of w F dV) instead of the markers scattering it with
//    atomics: no zeroing, no spreading launch, and the same bits every run;
//  - per marker m, the coupling A_mk = dV_k sum over nodes of w_m w_k to every
//    marker k whose stencil meets its own.  Interpolating the velocity that
//    the spread increment dF adds is then (A dF)_m, so the forcing iterations
//    of Eq. 9, U^(k+1) = U^(k) + A dF^(k), dF^(k+1) = dF^(k) - A dF^(k), need
//    no lattice field: one pass over the markers each.

// sums over a warp, in all lanes
template <typename T> __device__ __forceinline__ T warp_all_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The solid's reaction -F dV to marker m's force and its torque (one thread).
__device__ __forceinline__ void marker_reaction(const IbmTab &tb, int m, const double F[3],
                                                double *part, int *psid) {
  const double dV = tb.dV[m];
  const double r[3] = {tb.arm[m], tb.arm[tb.nmark + m], tb.arm[2 * tb.nmark + m]};
  const double Fs[3] = {-F[0] * dV, -F[1] * dV, -F[2] * dV};
  part[0] = Fs[0];
  part[1] = Fs[1];
  part[2] = Fs[2];
  part[3] = r[1] * Fs[2] - r[2] * Fs[1];
  part[4] = r[2] * Fs[0] - r[0] * Fs[2];
  part[5] = r[0] * Fs[1] - r[1] * Fs[0];
  *psid = tb.msid[m];
}

// Marker m of a warp, its last forcing pass done: total force F (FP64, the same
// in all lanes): keep F dV for the nodes' rows and the reaction in the block's
// sums (part: 6 per warp, psid its solid).
template <typename T>
__device__ __forceinline__ void marker_done(const IbmTab &tb, int m, int lane, const double F[3],
                                            double *part, int *psid) {
  const double dV = tb.dV[m];
  if (lane < 3)
    ((T *)tb.FdV)[lane * tb.nmark + m] = (T)((lane == 0 ? F[0] : lane == 1 ? F[1] : F[2]) * dV);
  if (lane == 0) marker_reaction(tb, m, F, part, psid);
}

// First pass of marker m (a warp): F = dF = U^d - interpolated u~.
template <typename T>
__device__ __forceinline__ void marker_first(const IbmTab &tb, const KArgs &a, int dim, int m,
                                             int lane, bool last, double *part, int *psid) {
  const int npts = dim == 3 ? 64 : 16;
  const int4 b = tb.base[m];
  const T *wts = (const T *)tb.wts + (long long)m * npts;
  const T *ub = (const T *)a.u_band;
  T U[3] = {0, 0, 0};
  for (int p = lane; p < npts; p += 32) {
    const T w = wts[p];
    const int kx = p & 3, ky = (p >> 2) & 3, kz = p >> 4;
    const long long n = wrap(b.x + kx, a.nx) +
                        (long long)a.nx * (wrap(b.y + ky, a.ny) +
                                           (long long)a.ny * (dim == 3 ? wrap(b.z + kz, a.nz) : 0));
    for (int c = 0; c < dim; c++) U[c] += w * ub[c * a.N + n];
  }
  double F[3] = {0, 0, 0};
  for (int c = 0; c < dim; c++) F[c] = tb.Ud[c * tb.nmark + m] - (double)warp_all_sum<T>(U[c]);
  if (last) {
    marker_done<T>(tb, m, lane, F, part, psid);
  } else if (lane < 3) {
    const double v = lane == 0 ? F[0] : lane == 1 ? F[1] : F[2];
    tb.dF[lane * tb.nmark + m] = v;
    tb.Fm[lane * tb.nmark + m] = v;
    ((T *)tb.dFT)[lane * tb.nmark + m] = (T)v;
  }
}

// A later pass: dF <- dF - A dF, F += dF.  The neighbours' previous increments
// are read from the compute-type copies, which alternate between two arrays.
template <typename T>
__device__ __forceinline__ void marker_next(const IbmTab &tb, int dim, int m, int lane, int pass,
                                            bool last, double *part, int *psid) {
  const int nm = tb.nmark;
  const T *in = (const T *)tb.dFT + (size_t)((pass + 1) & 1) * 3 * nm;
  T *out = (T *)tb.dFT + (size_t)(pass & 1) * 3 * nm;
  const int e0 = tb.mrow[m], e1 = tb.mrow[m + 1];
  T s[3] = {0, 0, 0};
  for (int e = e0 + lane; e < e1; e += 32) {
    const int k = tb.mcol[e];
    const T w = ((const T *)tb.mw)[e];
#pragma unroll
    for (int c = 0; c < 3; c++) s[c] += w * in[c * nm + k];
  }
  double F[3], d[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    d[c] = tb.dF[c * nm + m] - (double)warp_all_sum<T>(s[c]);
    F[c] = tb.Fm[c * nm + m] + d[c];
  }
  __syncwarp();
  if (last) {
    marker_done<T>(tb, m, lane, F, part, psid);
  } else if (lane < 3) {
    const double v = lane == 0 ? d[0] : lane == 1 ? d[1] : d[2];
    tb.dF[lane * nm + m] = v;
    out[lane * nm + m] = (T)v;
    tb.Fm[lane * nm + m] = lane == 0 ? F[0] : lane == 1 ? F[1] : F[2];
  }
}

// Block sums of NW warps' parts, one FP64 atomic per component and solid
// (psid -1: the warp has none).  Every thread of the block calls it.
template <int NW>
__device__ __forceinline__ void marker_block_force(double *force_acc, int nsolids,
                                                   const double (&part)[NW][6],
                                                   const int (&psid)[NW]) {
  __syncthreads();
  if (threadIdx.x < 6) {
    const int c = threadIdx.x;
    for (int s = 0; s < nsolids; s++) {
      double sum = 0;
      bool any = false;
      for (int w = 0; w < NW; w++)
        if (psid[w] == s) {
          sum += part[w][c];
          any = true;
        }
      if (any) atomicAdd(force_acc + 6 * s + c, sum);
    }
  }
  __syncthreads();
}

}  // namespace lbm

// run_impl.cuh -- many steps of small lattices in one launch.
//
// A small lattice's step is a chain of short kernels on two streams: with the
// launches, the fork and the join between them it took 11-17 us per step for
// the 64^2 and 301^2 Couette flows and 47-75 us with five IBM forcing
// iterations at 48^3, against 1-6 us of work.  k_run takes the steps of a
// call (up to 256 at a time) in one cooperative launch: the lattice's blocks (one per SM at most)
// keep stepping, with a barrier over them wherever one phase reads what
// another wrote:
//   bounce-back or no solids: boundary nodes and plain nodes read f*(t) and
//     write f*(t+1): one barrier per step;
//   IBM at rest (tables): band velocity and plain nodes | marker passes, one
//     barrier each | band nodes gather the force and collide.
// Up to kMaxRun lattices share a launch, each with its own blocks and barrier.
// Populations are read through L2 (LD_L2); everything written by other blocks
// is ordered by the barrier's release and acquire.
#pragma once

#include "ibm_device.cuh"

namespace lbm {

// Barrier over the nb blocks of a lattice, in two halves, so that work the
// other blocks do not wait for runs in between.  ctr counts arrivals since the
// launch began (target: nb per barrier so far), both modulo 2^32: they are never
// further apart than a barrier's blocks, so their difference has a sign.
// run_wait is false when the barrier was not reached within a second: the kernel
// then records it and returns.
__device__ __forceinline__ void run_arrive(unsigned *ctr) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
  }
}
__device__ __forceinline__ bool run_wait(unsigned *ctr, unsigned target, int *err, int *ok) {
  if (threadIdx.x == 0) {
    unsigned v;
    unsigned long long t0 = 0, now;
    for (unsigned spin = 0;; spin++) {
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((spin & 255u) == 255u) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
        if (t0 == 0) t0 = now;
        if (now - t0 > 1000000000ull) {
          *err = 1;
          *ok = 0;
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *ok != 0;
}

// What a thread of a boundary-node group reads again every step: its node,
// direction and cut link do not change while the solids rest, so the record
// stays in registers and a step's populations are one memory latency away.
// Element offsets into an array of populations; those of unused terms repeat
// the link's own node (a finite value for a zero coefficient).
template <typename T> struct ListItem {
  bool item, cut, other;  // other: the link belongs to a second solid
  int sid;
  long long n, o0, o1, o2, o3, o4;
  T c0, c1, c2, c3, c4, mw, uw[3], r[3], e[3];
  double w;
};

template <int LAT, typename S, typename T>
__device__ __forceinline__ void list_item(const KArgs &a, int group, int cnt, int NG, ListItem<T> &q) {
  using L = Lat<LAT>;
  constexpr int Q = L::Q;
  constexpr unsigned long long PX = pack_dir<LAT>(0), PY = pack_dir<LAT>(1), PZ = pack_dir<LAT>(2);
  constexpr unsigned long long PO = pack_opp<LAT>(), POH = pack_opp_hi<LAT>();
  const int i = threadIdx.x / NG, k = threadIdx.x - i * NG, t = group * NG + k;
  q.item = i < Q && t < cnt;
  q.cut = q.other = false;
  q.sid = -1;
  q.n = 0;
  if (!q.item) return;
  const long long n = a.list_node[t];
  const uint32_t mask = a.list_mask[t];
  q.n = n;
  int x, y, z;
  node_xyz(n, a.nx, a.ny, x, y, z);
  const int ex = (int)((PX >> (2 * i)) & 3ull) - 1;
  const int ey = (int)((PY >> (2 * i)) & 3ull) - 1;
  const int ez = (int)((PZ >> (2 * i)) & 3ull) - 1;
  const int ib = i < 12 ? (int)((PO >> (5 * i)) & 31ull) : (int)((POH >> (5 * (i - 12))) & 31ull);
  auto at = [&](int m) {
    return wrap(x + m * ex, a.nx) +
           (long long)a.nx * (wrap(y + m * ey, a.ny) + (long long)a.ny * wrap(z + m * ez, a.nz));
  };
  const long long fi = (long long)i * a.fs, fb = (long long)ib * a.fs;
  q.cut = (mask >> i) & 1u;
  if (!q.cut) {
    q.o0 = fi + at(-1);
    return;
  }
  const int lo = a.list_link[t], link = lo + __popc(mask & ((1u << i) - 1u));
  auto ld = [&](const void *p) { return ((const T *)p)[link]; };
  q.c0 = ld(a.links.c[0]);
  q.c1 = ld(a.links.c[1]);
  q.c2 = ld(a.links.c[2]);
  q.c3 = ld(a.links.c[3]);
  q.c4 = ld(a.links.c[4]);
  q.mw = ld(a.links.mw);
  for (int c = 0; c < 3; c++) {
    q.uw[c] = ld(a.links.uw[c]);
    q.r[c] = ld(a.links.arm[c]);
  }
  q.e[0] = (T)ex;
  q.e[1] = (T)ey;
  q.e[2] = (T)ez;
  const int cls = ex * ex + ey * ey + ez * ez;
  q.w = cls == 1 ? L::w(1) : L::w(Q - 1);
  q.sid = a.links.sid[link];
  q.other = q.sid != a.links.sid[lo];
  q.o0 = fb + n;
  q.o3 = q.c3 != (T)0 ? fi + n : q.o0;
  if (a.zy_pre) {
    q.o1 = q.o0;  // into the kept populations
    q.o2 = q.o4 = q.o0;
  } else {
    q.o1 = q.c1 != (T)0 ? fb + at(1) : q.o0;
    q.o4 = q.c4 != (T)0 ? fi + at(1) : q.o0;
    q.o2 = q.c2 != (T)0 ? fb + at(2) : q.o0;
  }
}

// f_i(t + 1) of a thread's item and its link's part of Eq. 17: the same
// operations, in the same order, as ibb_value and list_group.
template <typename S, typename T>
__device__ __forceinline__ T item_value(const KArgs &a, const S *src, const ListItem<T> &q, T isc,
                                        T (&part)[6], double *force_acc) {
  for (int c = 0; c < 6; c++) part[c] = 0;
  if (!q.item) return (T)0;
  const T fs = Store<S>::template ld<LD_L2>(src + q.o0, isc);
  if (!q.cut) return fs;
  const T f3 = Store<S>::template ld<LD_L2>(src + q.o3, isc);
  T v;
  if (a.zy_pre) {
    v = vfma(q.c3, f3, vfma(q.c1, ld_pol<LD_L2>((const T *)a.zy_pre + q.o1), q.mw));
  } else {
    const T f1 = Store<S>::template ld<LD_L2>(src + q.o1, isc);
    const T f4 = Store<S>::template ld<LD_L2>(src + q.o4, isc);
    const T f2 = Store<S>::template ld<LD_L2>(src + q.o2, isc);
    v = vfma(q.c3, f3, vfma(q.c2, f2, vfma(q.c4, f4, vfma(q.c1, f1, vfma(q.c0, fs, q.mw)))));
  }
  if (!q.other) {
    for (int c = 0; c < 3; c++) part[c] = -fs * (q.e[c] + q.uw[c]) - v * (q.e[c] - q.uw[c]);
    part[3] = q.r[1] * part[2] - q.r[2] * part[1];
    part[4] = q.r[2] * part[0] - q.r[0] * part[2];
    part[5] = q.r[0] * part[1] - q.r[1] * part[0];
  } else {
    const double fsd = q.w + (double)fs, fid = q.w + (double)v;
    double d[3];
    for (int c = 0; c < 3; c++)
      d[c] = fsd * (-(double)q.e[c] - (double)q.uw[c]) - fid * ((double)q.e[c] - (double)q.uw[c]);
    const double rr[3] = {(double)q.r[0], (double)q.r[1], (double)q.r[2]};
    atomicAdd(force_acc + 6 * q.sid + 0, d[0]);
    atomicAdd(force_acc + 6 * q.sid + 1, d[1]);
    atomicAdd(force_acc + 6 * q.sid + 2, d[2]);
    atomicAdd(force_acc + 6 * q.sid + 3, rr[1] * d[2] - rr[2] * d[1]);
    atomicAdd(force_acc + 6 * q.sid + 4, rr[2] * d[0] - rr[0] * d[2]);
    atomicAdd(force_acc + 6 * q.sid + 5, rr[0] * d[1] - rr[1] * d[0]);
  }
  return v;
}

// A thread's constant data under IBM.
// Markers (a warp each, when every marker has a warp): a lane's two stencil
// points, and its entries of the marker's coupling row.
constexpr int kRunRow = 4;  // entries per lane kept in registers; longer rows are read
template <typename T> struct MarkerItem {
  int m;            // marker of this warp, -1: none
  long long n[2];   // stencil nodes (n[1] < 0: none)
  T w[2];
  int e0, e1;       // row
  int col[kRunRow];
  T cw[kRunRow];
  double Ud;        // lane c < 3
};

template <int LAT, typename T>
__device__ __forceinline__ void marker_item(const KArgs &a, int m, int lane, bool rows,
                                            MarkerItem<T> &q) {
  constexpr int D = Lat<LAT>::D, npts = D == 3 ? 64 : 16;
  const IbmTab &tb = a.tab;
  q.m = m;
  q.n[0] = q.n[1] = -1;
  q.w[0] = q.w[1] = (T)0;
  q.e0 = q.e1 = 0;
  for (int j = 0; j < kRunRow; j++) {
    q.col[j] = 0;
    q.cw[j] = (T)0;
  }
  q.Ud = 0;
  if (m < 0) return;
  const int4 b = tb.base[m];
  for (int j = 0; j < 2; j++) {
    const int p = lane + 32 * j;
    if (p >= npts) continue;
    const int kx = p & 3, ky = (p >> 2) & 3, kz = p >> 4;
    q.n[j] = wrap(b.x + kx, a.nx) +
             (long long)a.nx * (wrap(b.y + ky, a.ny) +
                                (long long)a.ny * (D == 3 ? wrap(b.z + kz, a.nz) : 0));
    q.w[j] = ((const T *)tb.wts)[(long long)m * npts + p];
  }
  if (lane < D) q.Ud = tb.Ud[lane * tb.nmark + m];
  if (rows) {
    q.e0 = tb.mrow[m] + lane;
    q.e1 = tb.mrow[m + 1];
    for (int j = 0; j < kRunRow; j++)
      if (q.e0 + 32 * j < q.e1) {
        q.col[j] = tb.mcol[q.e0 + 32 * j];
        q.cw[j] = ((const T *)tb.mw)[q.e0 + 32 * j];
      }
  }
}

// IBM: whether the launch's lattices have IBM tables (all of them or none).
template <int LAT, int CM, typename S, typename T, int NL, bool IBM>
__global__ void __launch_bounds__(kRunBlock, 1) k_run(const __grid_constant__ RunArgs<NL> g) {
  constexpr int Q = Lat<LAT>::Q, D = Lat<LAT>::D;
  constexpr int NT = kRunBlock, NW = NT / 32, NG = NT / Q;
  constexpr bool kVecType = std::is_same<T, float>::value;
  __shared__ ListSmem<T, NT> sm;
  __shared__ double part[NW][6];
  __shared__ int psid[NW];
  __shared__ int ok;
  int k = 0;
  while (k + 1 < NL && k + 1 < g.n && (int)blockIdx.x >= g.block_start[k + 1]) k++;
  const RunLat &r = g.l[k];
  const KArgs &a = r.a;
  const int nb = g.block_start[k + 1] - g.block_start[k];
  const int vb = (int)blockIdx.x - g.block_start[k];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // plain nodes start from the last block, boundary and band nodes from the
  // first: a lattice with fewer of either than blocks spreads them
  const int rb = nb - 1 - vb;
  if (tid == 0) ok = 1;
  int cnt = a.counts[0];
  if (cnt > a.list_cap) cnt = a.list_cap;
  constexpr bool ibm = IBM;
  const int ngr = (cnt + NG - 1) / NG;
  const bool one_group = ngr <= nb;        // a boundary-node group per block
  const bool mine = one_group && vb < ngr; // this block has one
  const int kk = tid % NG, dd = tid / NG;  // node and direction of the thread
  const T isc = kisc<T>(a);
  const int nm = a.tab.nmark;
  const bool one_marker = nm <= nb * NW;   // a marker per warp
  ListItem<T> li;
  li.item = li.cut = false;
  double cst = 0;  // list_cst of (component, node) = (tid / NG, tid % NG)
  MarkerItem<T> mi;
  mi.m = -1;
  double dF = 0, Fm = 0;  // lane c < 3: component c of this warp's marker
  int rcol = 0, rn = 0;   // first entry of a band node's row, entries of this thread
  T rw = 0;
  uint8_t lfl = 0;
  if (mine) list_item<LAT, S, T>(a, vb, cnt, NG, li);
  if (mine && !ibm && dd < 6 && vb * NG + kk < cnt) {
    const int t = vb * NG + kk;
    cst = a.list_cst[(long long)dd * a.list_cap + t];
    if (dd == 0) sm.sid0[kk] = a.list_mask[t] ? a.links.sid[a.list_link[t]] : -1;
  }
  if (mine && ibm && li.item) {
    const int t = vb * NG + kk;
    lfl = a.flags[li.n];
    const int e = a.tab.nrow[t] + dd, e1 = a.tab.nrow[t + 1];
    rn = e < e1 ? (e1 - e + Q - 1) / Q : 0;
    if (rn > 0) {
      rcol = a.tab.ncol[e];
      rw = ((const T *)a.tab.nw)[e];
    }
  }
  if (ibm && one_marker) {
    const int m = warp * nb + vb;
    marker_item<LAT, T>(a, m < nm ? m : -1, lane, r.iters > 1, mi);
  }
  unsigned target = 0;
  for (int s = 0; s < r.nsteps; s++) {
    const int cur = (r.cur + s) & 1;
    const S *src = (const S *)r.f[cur];
    S *dst = (S *)r.f[1 - cur];
    const bool more = s + 1 < r.nsteps;
    double *acc = r.hist + (size_t)((r.slot0 + 1 + s) % r.hist_cap) * kMaxSolids * 6;
    // the next step's force record starts at zero (this step's was zeroed by
    // the step before, or before the launch)
    if (vb == nb - 1 && tid < 6 * kMaxSolids)
      r.hist[(size_t)((r.slot0 + 2 + s) % r.hist_cap) * kMaxSolids * 6 + tid] = 0.0;
    if (ibm) {
      for (int t = (warp * nb + vb) * 32 + lane; t < cnt; t += nb * NT)
        band_velocity<LAT, S, T, LD_L2>(a, src, t);
    } else if (one_group) {
      if (mine) {
        T p6[6];
        sm.f[tid] = item_value<S, T>(a, src, li, isc, p6, acc);
        const T keep = sm.f[tid];
#pragma unroll
        for (int c = 0; c < 6; c++) sm.red[c][tid] = p6[c];
        __syncthreads();
        if (li.item && a.zy_pre) ((T *)a.zy_pre)[(long long)dd * a.fs + li.n] = keep;
        if (li.item && dd == 0) {
          T f[Q];
#pragma unroll
          for (int d = 0; d < Q; d++) f[d] = sm.f[d * NG + kk];
          const Coll<T> c = make_coll<LAT, T>(a);
          collide<LAT, CM, S, T, true>(f, kg<T>(a, 0), kg<T>(a, 1), kg<T>(a, 2), c);
          scatter<LAT, S, T>(dst, a.fs, li.n, isc, f);
        }
      }
    } else {
      for (int gr = vb; gr < ngr; gr += nb)
        list_group<LAT, CM, S, T, NT, LD_L2>(a, src, dst, acc, gr, cnt, sm);
    }
    bool done = false;
    if constexpr (kVecType) {
      if (r.vec) {
        constexpr int V = 2 * VecS<S>::per_word;
        const unsigned nt = (unsigned)a.N / V, nu = (nt + 31) / 32;
        for (unsigned u = (unsigned)(warp * nb + rb); u < nu; u += (unsigned)(nb * NW))
          bulk_vec_update<LAT, CM, S, 2, vec_packed<S>(), LD_L2>(a, src, dst, u * 32 + lane, nt);
        done = true;
      }
    }
    if (!done)
      for (unsigned n = (unsigned)(warp * nb + rb) * 32u + lane; n < (unsigned)a.N;
           n += (unsigned)(nb * NT))
        bulk_node_update<LAT, CM, S, T, LD_L2, false, true>(a, src, dst, n);
    if (!ibm) {
      if (more) run_arrive(r.bar);
      else __syncthreads();
      if (mine) {
        // Eq. 17 while the other blocks arrive: the links' parts by node in
        // the directions' order, then the nodes in FP64 (see list_group)
        for (int q = tid; q < 6 * NG; q += NT) {
          const int c = q / NG, kn = q - c * NG;
          T v = 0;
#pragma unroll
          for (int d = 1; d < Q; d++) v += sm.red[c][d * NG + kn];
          sm.cst[c][kn] = (q == tid ? cst : a.list_cst[(long long)c * a.list_cap + vb * NG + kn]) + (double)v;
        }
        __syncthreads();
        for (int sd = 0; sd < a.nsolids; sd++)
          if (tid < 96) {
            const int c = tid >> 4, p = tid & 15;
            double v = 0;
            for (int kn = p; kn < NG && vb * NG + kn < cnt; kn += 16)
              if (sm.sid0[kn] == sd) v += sm.cst[c][kn];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 16);
            if (p == 0 && v != 0.0) atomicAdd(acc + 6 * sd + c, v);
          }
      }
      if (more && !run_wait(r.bar, target += (unsigned)nb, a.wait_err, &ok)) break;
      continue;
    }
    // ---- IBM: forcing passes over the markers, then the band nodes
    run_arrive(r.bar);
    if (!run_wait(r.bar, target += (unsigned)nb, a.wait_err, &ok)) break;
    bool lost = false;
    for (int it = 0; it < r.iters && !lost; it++) {
      const bool last = it == r.iters - 1;
      if (one_marker) {
        T v[3] = {0, 0, 0};
        if (mi.m >= 0) {
          if (it == 0) {
            const T *ub = (const T *)a.u_band;
#pragma unroll
            for (int j = 0; j < 2; j++)
              if (mi.n[j] >= 0)
#pragma unroll
                for (int c = 0; c < D; c++) v[c] += mi.w[j] * ld_pol<LD_L2>(ub + c * a.N + mi.n[j]);
          } else {
            const T *in = (const T *)a.tab.dFT + (size_t)((it + 1) & 1) * 3 * nm;
#pragma unroll
            for (int j = 0; j < kRunRow; j++)
              if (mi.e0 + 32 * j < mi.e1)
#pragma unroll
                for (int c = 0; c < D; c++) v[c] += mi.cw[j] * ld_pol<LD_L2>(in + c * nm + mi.col[j]);
            for (int e = mi.e0 + 32 * kRunRow; e < mi.e1; e += 32) {
              const int col = a.tab.mcol[e];
              const T w = ((const T *)a.tab.mw)[e];
#pragma unroll
              for (int c = 0; c < D; c++) v[c] += w * ld_pol<LD_L2>(in + c * nm + col);
            }
          }
        }
#pragma unroll
        for (int c = 0; c < D; c++) v[c] = warp_all_sum<T>(v[c]);
        const double sum = (double)(lane == 0 ? v[0] : lane == 1 ? v[1] : v[2]);
        if (mi.m >= 0 && lane < D) {
          dF = (it == 0 ? mi.Ud : dF) - sum;
          Fm = it == 0 ? dF : Fm + dF;
          if (!last) ((T *)a.tab.dFT)[(size_t)((it & 1) * 3 + lane) * nm + mi.m] = (T)dF;
        }
        // all three components (z is zero in 2D): the band nodes gather three
        if (last && mi.m >= 0 && lane < 3)
          ((T *)a.tab.FdV)[lane * nm + mi.m] = (T)(Fm * a.tab.dV[mi.m]);
        run_arrive(r.bar);
        if (last) {
          // the solids' reaction while the other blocks arrive
          double F[3] = {0, 0, 0};
#pragma unroll
          for (int c = 0; c < D; c++) F[c] = __shfl_sync(0xffffffffu, Fm, c);
          if (lane == 0) {
            psid[warp] = -1;
            if (mi.m >= 0) marker_reaction(a.tab, mi.m, F, part[warp], &psid[warp]);
          }
          marker_block_force<NW>(acc, a.nsolids, part, psid);
        }
      } else {
        const int rounds = (nm + nb * NW - 1) / (nb * NW);
        for (int q = 0; q < rounds; q++) {
          const int m = (q * NW + warp) * nb + vb;
          if (lane == 0) psid[warp] = -1;
          __syncwarp();
          if (m < nm) {
            if (it == 0) marker_first<T>(a.tab, a, D, m, lane, last, part[warp], &psid[warp]);
            else marker_next<T>(a.tab, D, m, lane, it, last, part[warp], &psid[warp]);
          }
          if (last) marker_block_force<NW>(acc, a.nsolids, part, psid);
        }
        run_arrive(r.bar);
      }
      lost = !run_wait(r.bar, target += (unsigned)nb, a.wait_err, &ok);
    }
    if (lost) break;
    if (one_group) {
      if (mine) {
        T p3[3] = {0, 0, 0}, fi = 0;
        if (li.item) {
          fi = Store<S>::template ld<LD_L2>(src + li.o0, isc);
          const T *F = (const T *)a.tab.FdV;
          if (rn > 0)
            for (int c = 0; c < 3; c++) p3[c] = rw * ld_pol<LD_L2>(F + c * nm + rcol);
          for (int j = 1; j < rn; j++) {
            const int e = a.tab.nrow[vb * NG + kk] + dd + Q * j;
            const int col = a.tab.ncol[e];
            const T w = ((const T *)a.tab.nw)[e];
            for (int c = 0; c < 3; c++) p3[c] += w * ld_pol<LD_L2>(F + c * nm + col);
          }
        }
        sm.f[tid] = fi;
        for (int c = 0; c < 3; c++) sm.red[c][tid] = p3[c];
        __syncthreads();
        if (li.item && dd == 0) {
          T F3[3] = {0, 0, 0}, f[Q];
#pragma unroll
          for (int d = 0; d < Q; d++) {
            f[d] = sm.f[d * NG + kk];
            for (int c = 0; c < 3; c++) F3[c] += sm.red[c][d * NG + kk];
          }
          const bool gon = !(lfl & FL_NOG);
          for (int c = 0; c < 3; c++) {
            ((T *)const_cast<void *>(a.f_ibm))[c * a.N + li.n] = F3[c];
            F3[c] = (gon ? kg<T>(a, c) : (T)0) + F3[c];
          }
          const Coll<T> c = make_coll<LAT, T>(a);
          collide<LAT, CM, S, T>(f, F3[0], F3[1], F3[2], c);
          scatter<LAT, S, T>(dst, a.fs, li.n, isc, f);
        }
      }
    } else {
      for (int t = (warp * nb + vb) * 32 + lane; t < cnt; t += nb * NT)
        ibm_list_node<LAT, CM, S, T, LD_L2>(a, src, dst, t);
    }
    if (more) {
      run_arrive(r.bar);
      if (!run_wait(r.bar, target += (unsigned)nb, a.wait_err, &ok)) break;
    }
  }
  // the last block out resets the counters for the next launch
  __syncthreads();
  if (tid == 0 && atomicAdd(r.bar + 1, 1u) == (unsigned)nb - 1u) {
    r.bar[0] = 0;
    r.bar[1] = 0;
    __threadfence();
  }
}

template <int LAT, int CM, typename S, typename T, int NL>
cudaError_t launch_run_n(const RunArgs<kMaxRun> &g, cudaStream_t st) {
  RunArgs<NL> s;
  s.n = g.n;
  for (int k = 0; k <= NL; k++) s.block_start[k] = g.block_start[k];
  for (int k = 0; k < NL; k++) s.l[k] = g.l[k];
  void *args[1] = {&s};
  const void *kern = g.l[0].a.tab.nmark > 0 ? (const void *)k_run<LAT, CM, S, T, NL, true>
                                            : (const void *)k_run<LAT, CM, S, T, NL, false>;
  return cudaLaunchCooperativeKernel(kern, dim3((unsigned)g.block_start[g.n]), dim3(kRunBlock),
                                     args, 0, st);
}

template <typename S, typename T>
cudaError_t launch_run_precision(const RunArgs<kMaxRun> &g, int lattice, int collision,
                                 cudaStream_t st) {
  auto go = [&](auto lat, auto cm) {
    constexpr int LAT = decltype(lat)::value, CM = decltype(cm)::value;
    return g.n == 1 ? launch_run_n<LAT, CM, S, T, 1>(g, st)
                    : launch_run_n<LAT, CM, S, T, kMaxRun>(g, st);
  };
  using I = std::integral_constant<int, 0>;
  using J = std::integral_constant<int, 1>;
  if (lattice == LBM_D2Q9) {
    if (collision == CM_BGK) return go(I{}, std::integral_constant<int, CM_BGK>{});
    return go(I{}, std::integral_constant<int, CM_MRT_Q>{});
  }
  if (collision == CM_BGK) return go(J{}, std::integral_constant<int, CM_BGK>{});
  return go(J{}, std::integral_constant<int, CM_MRT_Q>{});
}

}  // namespace lbm

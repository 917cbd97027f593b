// sweep_vec.cuh -- the bulk sweep with vector loads and stores.
//
// Each thread updates V consecutive nodes of one x-row, held as W 32-bit
// words per direction (W = 2 or 4: 8- or 16-byte accesses; V = W for FP32
// storage, 2W for 16-bit storage).  For the directions with e_x = +-1
// the pulled values are the row shifted by one node: the thread takes the
// missing end node from its neighbour lane's vector (or loads it itself at a
// row or warp edge).  The collision then runs on pairs of nodes in packed
// FP32x2 arithmetic (one instruction for two nodes; 16-bit storage's default)
// or node by node (FP32 storage's): Eq. 1 (BGK) or Eq. 3 (MRT) with Guo
// forcing, where MRT differs from BGK only on the energy-flux (q) moments.
//
// Requirements (checked by the launcher, which otherwise runs the one-node
// kernel): nx % V == 0 and a direction stride that is a multiple of V.
#pragma once

#include "sweep_impl.cuh"

namespace lbm {

// ---------------------------------------------------------------- FP32x2
__device__ __forceinline__ float2 bc2(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// ---------------------------------------------------------------- storage
// W words of a direction's vector; node k of the vector is word k (FP32) or
// the low (k even) / high (k odd) half of word k / 2 (16-bit).
template <int W> struct Words {
  uint32_t w[W];
};
template <int W, int POL = LD_NC> __device__ __forceinline__ Words<W> ld_words(const void *p) {
  Words<W> r;
  if constexpr (W == 4) {
    const uint4 v = ld_pol<POL>(reinterpret_cast<const uint4 *>(p));
    r.w[0] = v.x, r.w[1] = v.y, r.w[2] = v.z, r.w[3] = v.w;
  } else {
    static_assert(W == 2, "8- or 16-byte vectors");
    const uint2 v = ld_pol<POL>(reinterpret_cast<const uint2 *>(p));
    r.w[0] = v.x, r.w[1] = v.y;
  }
  return r;
}
template <int W> __device__ __forceinline__ void st_words(void *p, const Words<W> &r) {
  if constexpr (W == 4) {
    *reinterpret_cast<uint4 *>(p) = make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]);
  } else {
    *reinterpret_cast<uint2 *>(p) = make_uint2(r.w[0], r.w[1]);
  }
}

// high half of a, low half of b
__device__ __forceinline__ uint32_t join16(uint32_t a, uint32_t b) {
  return __byte_perm(a, b, 0x5432);
}

template <typename S> struct VecS;
template <> struct VecS<float> {
  static constexpr int per_word = 1;
  static constexpr int kScaleLog2 = 0;  // stored values are the deviations
  // the end node fetched from outside the vector, as the word the shift
  // below expects
  template <int POL> __device__ static uint32_t left_word(const float *p) {
    return __float_as_uint(ld_pol<POL>(p));
  }
  template <int POL> __device__ static uint32_t right_word(const float *p) {
    return __float_as_uint(ld_pol<POL>(p));
  }
  // shift by one node: e_x = +1 pulls from x - 1, e_x = -1 from x + 1
  template <int W> __device__ static void shift_in_left(Words<W> &v, uint32_t l) {
#pragma unroll
    for (int k = W - 1; k > 0; k--) v.w[k] = v.w[k - 1];
    v.w[0] = l;
  }
  template <int W> __device__ static void shift_in_right(Words<W> &v, uint32_t r) {
#pragma unroll
    for (int k = 0; k < W - 1; k++) v.w[k] = v.w[k + 1];
    v.w[W - 1] = r;
  }
  // pair p (nodes 2p, 2p + 1) as float2, and back
  template <int W> __device__ static float2 get(const Words<W> &v, int p, float2) {
    return make_float2(__uint_as_float(v.w[2 * p]), __uint_as_float(v.w[2 * p + 1]));
  }
  template <int W> __device__ static void put(Words<W> &v, int p, float2 f, float2) {
    v.w[2 * p] = __float_as_uint(f.x);
    v.w[2 * p + 1] = __float_as_uint(f.y);
  }
  template <int W> __device__ static void store_node(float *p, const Words<W> &v, int k) {
    *p = __uint_as_float(v.w[k]);
  }
};

template <typename H> struct VecS16 {
  static constexpr int per_word = 2;
  static constexpr int kScaleLog2 = 0;
  template <int POL> __device__ static uint32_t ld16(const H *p) {
    return (uint32_t)ld_pol<POL>(reinterpret_cast<const unsigned short *>(p));
  }
  // node x0 - 1 in the high half, node x0 + V in the low half
  template <int POL> __device__ static uint32_t left_word(const H *p) { return ld16<POL>(p) << 16; }
  template <int POL> __device__ static uint32_t right_word(const H *p) { return ld16<POL>(p); }
  template <int W> __device__ static void shift_in_left(Words<W> &v, uint32_t l) {
#pragma unroll
    for (int k = W - 1; k > 0; k--) v.w[k] = join16(v.w[k - 1], v.w[k]);
    v.w[0] = join16(l, v.w[0]);
  }
  template <int W> __device__ static void shift_in_right(Words<W> &v, uint32_t r) {
#pragma unroll
    for (int k = 0; k < W - 1; k++) v.w[k] = join16(v.w[k], v.w[k + 1]);
    v.w[W - 1] = join16(v.w[W - 1], r);
  }
  template <int W> __device__ static void store_node(H *p, const Words<W> &v, int k) {
    const uint32_t w = v.w[k >> 1];
    *reinterpret_cast<unsigned short *>(p) = (unsigned short)((k & 1) ? (w >> 16) : (w & 0xffffu));
  }
};

template <> struct VecS<__nv_bfloat16> : VecS16<__nv_bfloat16> {
  template <int W> __device__ static float2 get(const Words<W> &v, int p, float2) {
    const uint32_t w = v.w[p];
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
  }
  template <int W> __device__ static void put(Words<W> &v, int p, float2 f, float2) {
    const __nv_bfloat162 h = __float22bfloat162_rn(f);
    v.w[p] = *reinterpret_cast<const uint32_t *>(&h);
  }
};

// FP16 holds deviations times 2^k (k = kFp16ScaleLog2): get multiplies by
// inv_scale = 2^-k, put by scale = 2^k (both exact); get_scaled / put_scaled
// keep the scaled units, for the packed collision that works in them
template <> struct VecS<__half> : VecS16<__half> {
  static constexpr int kScaleLog2 = kFp16ScaleLog2;
  template <int W> __device__ static float2 get_scaled(const Words<W> &v, int p) {
    const uint32_t w = v.w[p];
    return __half22float2(*reinterpret_cast<const __half2 *>(&w));
  }
  template <int W> __device__ static void put_scaled(Words<W> &v, int p, float2 f) {
    const __half2 h = __float22half2_rn(f);
    v.w[p] = *reinterpret_cast<const uint32_t *>(&h);
  }
  template <int W> __device__ static float2 get(const Words<W> &v, int p, float2 inv_scale) {
    return mul2(get_scaled(v, p), inv_scale);
  }
  template <int W> __device__ static void put(Words<W> &v, int p, float2 f, float2 scale) {
    put_scaled(v, p, mul2(f, scale));
  }
};

// flag bytes of V consecutive nodes (V = 2, 4 or 8, aligned), as words
template <int V> __device__ __forceinline__ void ld_flags(const uint8_t *p, uint32_t (&f)[(V + 3) / 4]) {
  if constexpr (V == 8) {
    const uint2 w = *reinterpret_cast<const uint2 *>(p);
    f[0] = w.x;
    f[1] = w.y;
  } else if constexpr (V == 4) {
    f[0] = *reinterpret_cast<const uint32_t *>(p);
  } else {
    f[0] = *reinterpret_cast<const uint16_t *>(p);
  }
}

// ---------------------------------------------------------------- kernel
// The second half of a vector update: collide the V pulled nodes of a
// thread (v, their flag bytes fl) and store the plain fluid ones at n0.  A
// node is updated when its flag byte has no bit but FL_NOG / FL_NEW; the
// other nodes of a vector (boundary-list nodes, solid nodes) are computed but
// not stored, since the boundary-node kernel writes them.
template <int LAT, int CM, typename S, int W, bool PACKED>
__device__ __forceinline__ void vec_collide_store(const KArgs &a, S *dst,
                                                  Words<W> (&v)[Lat<LAT>::Q],
                                                  const uint32_t (&fl)[(W * VecS<S>::per_word + 3) / 4],
                                                  unsigned n0, bool valid) {
  using L = Lat<LAT>;
  using VS = VecS<S>;
  constexpr int Q = L::Q, V = W * VS::per_word, NP = V / 2;
  static_assert(V % 2 == 0, "nodes are collided in pairs");
  constexpr uint32_t kOther = (uint8_t)~(FL_NOG | FL_NEW);
  auto flag = [&](int k) { return (fl[k >> 2] >> (8 * (k & 3))) & 0xffu; };
  bool all = valid, any = false;
#pragma unroll
  for (int k = 0; k < V; k++) {
    const bool u = (flag(k) & kOther) == 0;
    all = all && u;
    any = any || u;
  }
  any = any && valid;
  const Coll<float> c = make_coll<LAT, float>(a);
  // the packed collision of FP16 storage runs in its scaled units (the host
  // sets a.inv_scale_f = 2^-SL for it); the rest unscale on load
  constexpr int SL = PACKED ? VS::kScaleLog2 : 0;
  const float2 isc = bc2(a.inv_scale_f), sc = bc2(1.0f / a.inv_scale_f);
  constexpr float kF = (float)(1 << SL);  // force in the same units (exact)
  const float gx = a.g_f[0] * kF, gy = a.g_f[1] * kF, gz = a.g_f[2] * kF;
  static_for<NP>([&](auto pc) {
    constexpr int p = decltype(pc)::value;
    float2 f[Q];
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if constexpr (SL != 0) f[i] = VS::get_scaled(v[i], p);
      else f[i] = VS::get(v[i], p, isc);
    });
    const float g0 = (flag(2 * p) & FL_NOG) ? 0.f : 1.f;
    const float g1 = (flag(2 * p + 1) & FL_NOG) ? 0.f : 1.f;
    if constexpr (PACKED) {
      collide_two_rate<LAT, CM, SL, even_first<S>(), float2, float>(
          f, make_float2(g0 * gx, g1 * gx), make_float2(g0 * gy, g1 * gy),
          make_float2(g0 * gz, g1 * gz), c);
    } else {
      float fa[Q], fb[Q];
      static_for<Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        fa[i] = f[i].x;
        fb[i] = f[i].y;
      });
      collide<LAT, CM, S, float>(fa, g0 * gx, g0 * gy, g0 * gz, c);
      collide<LAT, CM, S, float>(fb, g1 * gx, g1 * gy, g1 * gz, c);
      static_for<Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        f[i] = make_float2(fa[i], fb[i]);
      });
    }
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if constexpr (SL != 0) VS::put_scaled(v[i], p, f[i]);
      else VS::put(v[i], p, f[i], sc);
    });
  });
  if (all) {
    static_for<Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      st_words<W>(dst + (long long)i * a.fs + n0, v[i]);
    });
  } else if (any) {
#pragma unroll
    for (int k = 0; k < V; k++) {
      if (flag(k) & kOther) continue;
      static_for<Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        VS::store_node(dst + (long long)i * a.fs + n0 + k, v[i], k);
      });
    }
  }
}

// Thread t updates the vector of nodes [V t, V t + V), pulling the shifted
// rows straight from global memory.  Every lane of the warp calls this
// (threads past the end with t >= nt), for the shuffles.
template <int LAT, int CM, typename S, int W, bool PACKED, int POL = LD_NC>
__device__ __forceinline__ void bulk_vec_update(const KArgs &a, const S *src, S *dst, unsigned t,
                                                unsigned nt) {
  using L = Lat<LAT>;
  using VS = VecS<S>;
  constexpr int Q = L::Q, V = W * VS::per_word;
  const bool valid = t < nt;
  // threads past the end still take part in the lane shuffles (on node 0)
  const unsigned n0 = valid ? t * V : 0u;
  const unsigned yz = n0 / (unsigned)a.nx;
  const int x0 = (int)(n0 - yz * (unsigned)a.nx);
  const int z = (int)(yz / (unsigned)a.ny);
  const int y = (int)(yz - (unsigned)z * (unsigned)a.ny);
  uint32_t fl[(V + 3) / 4];
  ld_flags<V>(a.flags + n0, fl);
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  const int zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
  // source rows (y - e_y, z - e_z)
  const unsigned r[3][3] = {
      {(unsigned)nx * (ym + (unsigned)ny * zm), (unsigned)nx * (y + (unsigned)ny * zm),
       (unsigned)nx * (yp + (unsigned)ny * zm)},
      {(unsigned)nx * (ym + (unsigned)ny * z), (unsigned)nx * (y + (unsigned)ny * z),
       (unsigned)nx * (yp + (unsigned)ny * z)},
      {(unsigned)nx * (ym + (unsigned)ny * zp), (unsigned)nx * (y + (unsigned)ny * zp),
       (unsigned)nx * (yp + (unsigned)ny * zp)}};
  const int lane = threadIdx.x & 31;
  // the neighbour lane holds the adjacent vector of the same row
  const bool lnb = lane != 0 && x0 != 0;
  const bool rnb = lane != 31 && x0 + V != nx;
  const int xl = x0 == 0 ? nx - 1 : x0 - 1, xr = x0 + V == nx ? 0 : x0 + V;
  Words<W> v[Q];
  uint32_t edge[Q];
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    const S *row = src + (long long)i * a.fs + r[1 - L::ez(i)][1 - L::ey(i)];
    v[i] = ld_words<W, POL>(row + x0);
    edge[i] = 0u;
    if constexpr (L::ex(i) == 1) {
      if (!lnb) edge[i] = VS::template left_word<POL>(row + xl);
    } else if constexpr (L::ex(i) == -1) {
      if (!rnb) edge[i] = VS::template right_word<POL>(row + xr);
    }
  });
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (L::ex(i) == 1) {
      const uint32_t sw = __shfl_up_sync(0xffffffffu, v[i].w[W - 1], 1);
      VS::shift_in_left(v[i], lnb ? sw : edge[i]);
    } else if constexpr (L::ex(i) == -1) {
      const uint32_t sw = __shfl_down_sync(0xffffffffu, v[i].w[0], 1);
      VS::shift_in_right(v[i], rnb ? sw : edge[i]);
    }
  });
  vec_collide_store<LAT, CM, S, W, PACKED>(a, dst, v, fl, n0, valid);
}

// Whether a storage type's default vector kernel collides packed node pairs.
template <typename S> __host__ __device__ constexpr bool vec_packed() { return sizeof(S) == 2; }
// Registers a thread of the 2-word kernels: FP32 node by node 64 (8 blocks of
// 128 per SM, whose warps hide more of the boundary kernel's share of the SMs
// than 6 at 80), packed 80, BF16 112, FP16 128.  Measured on 128^3 / 160^3 /
// 192^3 lattices without solids, us per step: BF16 29.8 / 55.3 / 91.6 at 96,
// 26.7 / 49.0 / 82.0 at 112, 26.8 / 50.7 / 84.4 at 128; FP16 30.8 / 57.3 / 95.8
// at 96, 27.8 / 51.5 / 87.8 at 112, 26.7 / 49.5 / 84.0 at 128.  4-word vectors
// are left unbounded.
template <typename S, int W, bool PACKED> constexpr int vec_regs() {
  return W == 4 ? 255 : sizeof(S) == 4 ? (PACKED ? 80 : 64)
                      : std::is_same<S, __nv_bfloat16>::value ? 112 : 128;
}

// One thread per vector.  (A persistent grid walking the lattice measured
// slower: it holds more registers and leaves the boundary kernels less room;
// so did one that kept the next vector's loads in flight through a cp.async
// ring in shared memory.)
// Blocks walk the lattice from its end when a.rev is set (every other step):
// a step then starts on the nodes that the previous one wrote last, which L2
// still holds, instead of on those it has already evicted.  us per step without
// solids: FP32 112^3 36.5 -> 33.6, 128^3 51.9 -> 48.6, 160^3 96.5 -> 94.3; FP16 128^3
// 31.2 -> 29.0 (26.6 with evict-first reads, LD_ONCE).
template <int LAT, int CM, typename S, int W, bool PACKED, int POL>
__global__ void __maxnreg__((vec_regs<S, W, PACKED>()))
    k_bulk_vec(const KArgs a) {
  constexpr int V = W * VecS<S>::per_word;
  const unsigned b = a.rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  bulk_vec_update<LAT, CM, S, W, PACKED, POL>(a, (const S *)a.src, (S *)a.dst,
                                              b * blockDim.x + threadIdx.x, (unsigned)a.N / V);
}

// The same update for several lattices in one grid: block b belongs to the
// last lattice k with block_start[k] <= b.
// Each lattice gets its own inlined copy of the update, so that its
// arguments stay constant-bank operands (indexing the argument array by a
// run-time k holds them in registers: 92 instead of 80, one block per SM
// fewer).
// The single-lattice kernel's register limits (FP32 at 64, with 404 bytes of spill
// stores: two empty 128^3 101.7 us per step against 100.6 at 80, eight 64^3 spheres
// 77.2 against 86.5).
template <int LAT, int CM, typename S, int W, bool PACKED>
__global__ void __maxnreg__((vec_regs<S, W, PACKED>()))
    k_bulk_vec_group(const __grid_constant__ GroupArgs g) {
  constexpr int V = W * VecS<S>::per_word;
  const int b = (int)blockIdx.x;
  static_for<kMaxGroup>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if (k < g.n && b >= g.block_start[k] && b < g.block_start[k + 1])
      bulk_vec_update<LAT, CM, S, W, PACKED>(
          g.a[k], (const S *)g.a[k].src, (S *)g.a[k].dst,
          (unsigned)(g.a[k].rev ? g.block_start[k + 1] - 1 - b : b - g.block_start[k]) * blockDim.x +
              threadIdx.x,
          (unsigned)g.a[k].N / V);
  });
}

}  // namespace lbm

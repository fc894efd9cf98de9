// MERBIT SpMM: Y = A X for a row-major X (n_cols x k) and Y (n_rows x k), f32,
// on the same plan as the SpMV (the batching extension of the hot path: k
// personalisation vectors in one pass).
//
// The lane-walk kernel of the SpMV (spmv_walk_kernel.cuh), k values wide: a warp takes units
// of consecutive tiles on its own, with one buffer each for a tile's columns and values.  A
// column chunk of KC columns is split into slices of VW consecutive columns (one load each);
// T = KC / VW threads share a lane of the tile, so a warp walks L = 32 / T lanes at once and a
// tile's 32 lanes in T passes.  Per pass:
//   1. the lane descriptor (Sec. 4.1.1) says which nonzero every right step consumes, so the
//      row slices of a batch of steps are gathered before any is used;
//   2. the steps are walked: a right step adds vals * slice into the running sum, a down step
//      ends a row.  Rows that begin and end inside the lane go straight to Y; the lane's
//      first row end is kept (`head`);
//   3. the runs open at the lanes' ends are joined by a segmented shuffle scan; a lane's first
//      row totals its head plus the run that reaches it, and the run open after the pass is
//      carried into the next pass, the next tile and to the unit's end.  A run that takes whole
//      passes or tiles keeps what its sum loses to rounding, and joins its row's end last: a long
//      row has one rounding at its full size, whatever the width (in f32 alone the root mean square
//      of rows above 448 nonzeros was 7.2e-8 at k = 32, 4.7e-8 at k = 4; 3.4e-8 and 3.5e-8).
// A unit's first row and the row open at its end are added into FP64 accumulators (KC wide,
// one set per distinct row at the unit boundaries), which a second pass writes and clears.
//
// What bounds it.  Narrow chunks: the L1 data pipe, one wavefront per gathered row slice line
// (k = 8: 82 % busy, a quarter of it shared-memory work).  Wide ones: the bytes in flight (16
// warps, 14 slices of 16 bytes a thread: 114 KB an SM).  Multiply-adds and stores are predicated
// on the descriptor's bits instead of branched over, and no table, arrival count or block barrier
// joins the warps: 2.6 warp instructions per nonzero at k = 8 instead of 3.2.  R-MAT scale 21
// (32.4 M nonzeros), before and after: k = 4 0.189 / 0.170 ms, k = 8 0.224 / 0.192, k = 16 0.302 /
// 0.275, k = 32 0.495 / 0.474.
#pragma once

#include <climits>
#include <type_traits>

#include "spmv_kernel.cuh"

namespace merbit {

// Two f32 operations of one packed instruction (sm_100 on); each rounds as the scalar one does.
// They halve the multiply-adds of a slice, and the products with alpha of personalised PageRank's
// stores, made at every step whether it stores or not (2^22 vertices, k = 32, an update: 1.34 ms
// with scalar ones, 1.22; k = 16 0.745 and 0.704).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ void fma2(uint64_t w, float x0, float x1, float& s0, float& s1) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(w), "l"(pack2(x0, x1)), "l"(pack2(s0, s1)));
  unpack2(r, s0, s1);
}
__device__ __forceinline__ void mul2(uint64_t w, float& x0, float& x1) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(x0, x1)), "l"(w));
  unpack2(r, x0, x1);
}

template <int VW> struct SpmmVec;
template <> struct SpmmVec<1> {
  using T = float;
  static __device__ __forceinline__ T zero() { return 0.f; }
  static __device__ __forceinline__ T load_plain(const float* p) { return *p; }
  static __device__ __forceinline__ void store(float* p, const float (&a)[1]) { *p = a[0]; }
  static __device__ __forceinline__ T load_shared(const float* p) { return *p; }
  static __device__ __forceinline__ void store_shared(float* p, const T& v) { *p = v; }
  static __device__ __forceinline__ void store_shared_if(uint32_t pred, float* p, const T& v) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.f32 [%1], %2;\n\t}" ::"r"(pred),
                 "r"(smem_addr(p)), "f"(v));
  }
  static __device__ __forceinline__ void fma(float w, const T& x, T& s) { s = fmaf(w, x, s); }
  static __device__ __forceinline__ float get(const T& v, int) { return v; }
  static __device__ __forceinline__ void add(T& s, const T& x) { s += x; }
  static __device__ __forceinline__ void add_exact(T& s, T& lost, const T& x) { add_lost(s, lost, x); }
  static __device__ __forceinline__ T shfl_up(const T& v, int d) {
    return __shfl_up_sync(0xffffffffu, v, d);
  }
  static __device__ __forceinline__ T shfl_xor(const T& v, int d) {
    return __shfl_xor_sync(0xffffffffu, v, d);
  }
};
template <> struct SpmmVec<4> {
  using T = float4;
  static __device__ __forceinline__ T zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ T load_plain(const float* p) {
    return *reinterpret_cast<const float4*>(p);
  }
  static __device__ __forceinline__ void store(float* p, const float (&a)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(a[0], a[1], a[2], a[3]);
  }
  static __device__ __forceinline__ T load_shared(const float* p) { return load_plain(p); }
  static __device__ __forceinline__ void store_shared(float* p, const T& v) { *reinterpret_cast<float4*>(p) = v; }
  static __device__ __forceinline__ void store_shared_if(uint32_t pred, float* p, const T& v) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n\t}" ::"r"(
                     pred),
                 "r"(smem_addr(p)), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
  }
  static __device__ __forceinline__ void fma(float w, const T& x, T& s) {
    const uint64_t w2 = pack2(w, w);
    fma2(w2, x.x, x.y, s.x, s.y);
    fma2(w2, x.z, x.w, s.z, s.w);
  }
  static __device__ __forceinline__ float get(const T& v, int i) {
    return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
  }
  static __device__ __forceinline__ void add(T& s, const T& x) {
    s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
  }
  static __device__ __forceinline__ void add_exact(T& s, T& lost, const T& x) {
    add_lost(s.x, lost.x, x.x);
    add_lost(s.y, lost.y, x.y);
    add_lost(s.z, lost.z, x.z);
    add_lost(s.w, lost.w, x.w);
  }
  static __device__ __forceinline__ T shfl_up(const T& v, int d) {
    return make_float4(__shfl_up_sync(0xffffffffu, v.x, d), __shfl_up_sync(0xffffffffu, v.y, d),
                       __shfl_up_sync(0xffffffffu, v.z, d), __shfl_up_sync(0xffffffffu, v.w, d));
  }
  static __device__ __forceinline__ T shfl_xor(const T& v, int d) {
    return make_float4(__shfl_xor_sync(0xffffffffu, v.x, d), __shfl_xor_sync(0xffffffffu, v.y, d),
                       __shfl_xor_sync(0xffffffffu, v.z, d), __shfl_xor_sync(0xffffffffu, v.w, d));
  }
};

// Y[r, c..c+VW) = (scale *) sum.  YVEC: the slices of Y are 16-byte aligned and kc is a multiple
// of VW; otherwise single columns below kc are stored.
struct SpmmOut {
  float* y;
  int64_t ldy;
  float scale;
  int kc;          // columns of the chunk
  bool gated;      // the launch does nothing once an iterative driver has set the stop flag
  __device__ __forceinline__ bool skip(const RedState* red) const {
    return gated && *reinterpret_cast<const volatile int*>(&red->done) != 0;
  }
};

template <bool SCALED>
__device__ __forceinline__ float spmm_scaled(float v, float scale) {
  if constexpr (SCALED) return scale * v;
  else return v;
}

// Predicated stores of a slice (no branch: lanes of a warp end rows at different steps; no memory
// clobber: nothing in the kernel reads Y, and loads may move over them).
template <int VW, bool YVEC, bool SCALED>
__device__ __forceinline__ void spmm_store_if(uint32_t pred, float* p, const typename SpmmVec<VW>::T& v, float scale,
                                              int left) {
  using V = SpmmVec<VW>;
  if constexpr (YVEC && VW == 4) {
    float4 s = v;
    if constexpr (SCALED) {
      const uint64_t k2 = pack2(scale, scale);
      mul2(k2, s.x, s.y);
      mul2(k2, s.z, s.w);
    }
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t"
        "@q st.global.v4.f32 [%1], {%2, %3, %4, %5};\n\t}" ::"r"(pred),
        "l"(p), "f"(s.x), "f"(s.y), "f"(s.z), "f"(s.w));
  } else {
#pragma unroll
    for (int i = 0; i < VW; ++i)
      asm volatile(
          "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t"
          "@q st.global.f32 [%1], %2;\n\t}" ::"r"(i < left ? pred : 0u),
          "l"(p + i), "f"(spmm_scaled<SCALED>(V::get(v, i), scale)));
  }
}

// Gathers of a slice, kept in order so that a batch is in flight before its first use.  They are
// not predicated: a register that a predicated load may leave unwritten stays allocated through
// the whole loop (168 registers instead of 96).  Steps that take no nonzero load the tile's
// first one again.
__device__ __forceinline__ void spmm_load(const float* p, float& v) {
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
}
__device__ __forceinline__ void spmm_load(const float* p, float4& v) {
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
}

constexpr int kSpmmWarps = 4;
constexpr int kSpmmThreads = kSpmmWarps * 32;

// FP64 accumulators of unit boundary row: set index of tile boundary i (the first unit boundary
// in that row, which is the first one at or after the row's first tile boundary).
__device__ __forceinline__ int spmm_set(const Geometry& g, int i) {
  return (__ldg(g.tile_slot + i) + g.unit - 1) / g.unit;
}

// A warp's units: whole rounds give consecutive units to a CTA's warps, the rest is spread over
// the CTAs first (as in the SpMV's kernel); computed on the host.
struct SpmmUnits {
  int nfull, rest;
};

// Shared memory of a warp: values, columns, per thread the head sum of its lane's pass, and per
// column of the chunk the carried run and what its sum lost to rounding.
template <int VW>
__host__ __device__ constexpr size_t spmm_warp_bytes(int sigma) {
  return sizeof(float) * (2 * (size_t)walk_cap(sigma) + 32 * VW + 2 * 32);
}

template <int KC, int VW, int KS, bool YVEC, bool SCALED, int CTAS>
__global__ void __launch_bounds__(kSpmmThreads, CTAS)
    merbit_spmm_kernel(const Geometry g, const SpmmUnits un, double* __restrict__ acc, const float* __restrict__ vals,
                       const float* __restrict__ X, const int64_t ldx, const SpmmOut out) {
  using V = SpmmVec<VW>;
  using VT = typename V::T;
  constexpr int T = KC / VW;                   // threads per lane, one slice of VW columns each
  constexpr int L = 32 / T;                    // lanes walked at once (one pass)
  constexpr int U1 = VW == 1 ? 16 : 8;         // row slices per round of a single-row tile
  __shared__ __align__(8) uint64_t bars[kSpmmWarps][2];
  extern __shared__ __align__(128) unsigned char dyn_smem[];

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int gl = lane / T;                     // lane of the pass this thread walks
  const int c = (lane % T) * VW;               // first column of this thread's slice
  const int left = out.kc - c;                 // its columns
  const uint32_t c_ok = left > 0 ? ~0u : 0u;
  if (out.skip(g.red)) return;

  const int cap = walk_cap(g.sigma);
  float* const sv = reinterpret_cast<float*>(dyn_smem + (size_t)warp * spmm_warp_bytes<VW>(g.sigma));
  int32_t* const sc = reinterpret_cast<int32_t*>(sv + cap);
  float* const s_head = sv + 2 * cap + lane * VW;              // this thread's head sum
  float* const s_carry = sv + 2 * cap + 32 * VW + c;           // this slice's carried run
  float* const s_lost = s_carry + 32;                          // what its sum lost to rounding
  if (lane == 0) {
    mbar_init(&bars[warp][0], 1);
    mbar_init(&bars[warp][1], 1);
    fence_mbar_init();
  }
  __syncwarp();

  // row `col` of X at this thread's slice; slices wider than a column come with ldx < 2^30, so
  // that the byte offset is one 32 x 32-bit multiply-add
  const float* const Xc = X + (c_ok ? c : 0);
  auto x_row = [&](int col) {
    if constexpr (VW == 1) return Xc + (int64_t)col * ldx;
    else
      return reinterpret_cast<const float*>(reinterpret_cast<const char*>(Xc) +
                                            (uint64_t)(uint32_t)col * ((uint32_t)ldx * 4u));
  };
  auto y_row = [&](int r) { return out.y + c + (int64_t)r * out.ldy; };
  auto unit_start = [&](int r) {
    const int i = warp * (int)gridDim.x + (int)blockIdx.x;
    if (r >= un.nfull + (i < un.rest ? 1 : 0)) return -1;
    const int round = (int)gridDim.x * kSpmmWarps;
    return (r < un.nfull ? r * round + (int)blockIdx.x * kSpmmWarps + warp : un.nfull * round + i) * g.unit;
  };
  // bounds of tile ti, a word a lane: its first nonzero and row in lanes 0 and 2, the next
  // tile's in lanes 1 and 3
  auto load_meta = [&](int ti) { return __ldg((lane & 2 ? g.tile_y : g.tile_x) + ti + (lane & 1)); };
  auto load_desc = [&](int ti) {
    const int j = ti * kOmega + lane;
    return j < g.lane_num ? ld_stream(g.lane_desc + j, policy_evict_first()) : 0u;
  };
  auto issue = [&](const void* src, void* dst, uint32_t meta, int which) {
    const int a = (int)__shfl_sync(0xffffffffu, meta, 0), b = (int)__shfl_sync(0xffffffffu, meta, 1);
    if (lane == 0)
      walk_issue(static_cast<const int32_t*>(src), dst, a, b, g.nnz, &bars[warp][which], policy_evict_first());
  };
  auto add_acc = [&](int tile, const VT& v, const VT& lost) {
    double* a = acc + (size_t)spmm_set(g, tile) * KC + c;
#pragma unroll
    for (int i = 0; i < VW; ++i)
      if (i < left) {
        double q = (double)V::get(v, i);
        if (V::get(lost, i) != 0.f) q += (double)V::get(lost, i);
        atomicAdd(a + i, q);
      }
  };

  int rd = 0;
  int t = unit_start(0);
  if (t < 0) return;
  int t_start = t;
  uint32_t meta = load_meta(t), desc = load_desc(t);
  issue(g.col, sc, meta, 0);
  issue(vals, sv, meta, 1);
  uint32_t par = 0;
  int y_unit = (int)(__shfl_sync(0xffffffffu, meta, 2) & ~kMsb);   // the unit's first row
  if (gl == 0) {                                               // the unit's run starts at zero
    V::store_shared(s_carry, V::zero());
    V::store_shared(s_lost, V::zero());
  }
  auto extend_run = [&](const VT& x) {
    VT run = V::load_shared(s_carry), lost = V::load_shared(s_lost);
    V::add_exact(run, lost, x);
    V::store_shared(s_carry, run);
    V::store_shared(s_lost, lost);
  };
  while (true) {
    // the tile after this one, of this unit or of the next (-1: none)
    const bool next_unit = t + 1 >= min(t_start + g.unit, g.tile_num);
    const int tn = next_unit ? unit_start(rd + 1) : t + 1;
    uint32_t nmeta = 0, ndesc = 0;
    if (tn >= 0) {
      nmeta = load_meta(tn);
      ndesc = load_desc(tn);
    }
    const int xs = (int)__shfl_sync(0xffffffffu, meta, 0), xe = (int)__shfl_sync(0xffffffffu, meta, 1);
    const uint32_t tys = __shfl_sync(0xffffffffu, meta, 2);
    const int y_ws = (int)(tys & ~kMsb);
    bool ok = mbar_wait_bounded(&bars[warp][0], par, g.wait_limit);
    if (__all_sync(0xffffffffu, ok)) ok = mbar_wait_bounded(&bars[warp][1], par, g.wait_limit);
    if (!__all_sync(0xffffffffu, ok)) {
      // give up: record it and let this tile's copies land (bounded) before leaving
      if (lane == 0) {
        atomicOr(&g.red->err, 1);
        mbar_wait_bounded(&bars[warp][0], par);
        mbar_wait_bounded(&bars[warp][1], par);
      }
      return;
    }
    const WalkSpan<int32_t> span(xs, xe, g.nnz);   // columns and values: both 4 bytes wide
    if (span.end < xe) {
      // the arrays' last nonzeros, short of a whole 16-byte unit
      for (int k = span.end + lane; k < xe; k += 32) {
        sc[k - span.a0] = __ldg(g.col + k);
        sv[k - span.a0] = __ldg(vals + k);
      }
      __syncwarp();
    }
    const int pad = xs - span.a0;
    auto columns_read = [&]() {
      // every gather's address has been formed: the column buffer takes the next tile
      fence_proxy_async_smem();
      __syncwarp();
      if (tn >= 0) issue(g.col, sc, nmeta, 0);
    };

    const bool any = xe > xs;                      // the tile has nonzeros (the same in every lane)
    const int col0 = any ? sc[pad] : 0;
    if (tys & kMsb) {
      // one row: lane gl takes every L-th nonzero, the lanes' sums are added across the warp.  Each
      // round's products are summed apart: all in one chain would be 112 roundings a lane at L = 4
      const int ntile = xe - xs;
      VT sum = V::zero();
#pragma unroll 1
      for (int b0 = gl; b0 - gl < ntile; b0 += L * U1) {
        VT xv[U1];
#pragma unroll
        for (int u = 0; u < U1; ++u) spmm_load(x_row(b0 + u * L < ntile ? sc[pad + b0 + u * L] : col0), xv[u]);
        VT part = V::zero();
#pragma unroll
        for (int u = 0; u < U1; ++u)
          if (b0 + u * L < ntile) V::fma(sv[pad + b0 + u * L], xv[u], part);
        V::add(sum, part);
      }
      columns_read();
#pragma unroll
      for (int o = T; o < 32; o <<= 1) V::add(sum, V::shfl_xor(sum, o));
      if (gl == 0) extend_run(sum);
    } else {
#pragma unroll 1
      for (int p = 0; p < T; ++p) {
        const int l = p * L + gl;
        const uint32_t d = __shfl_sync(0xffffffffu, desc, l);
        const int j = t * kOmega + l;
        const int len = j < g.lane_num ? min(g.sigma, g.steps - j * g.sigma) : 0;
        const uint32_t valid = (1u << len) - 1u;
        const uint32_t dm = (d >> 18) & valid;                 // down steps
        const uint32_t rm = ~(d >> 18) & valid;                // right steps
        const uint32_t first = dm & (0u - dm);                 // the lane's first down step
        const int i0 = pad + (int)(d & 511u);
        const int y0 = y_ws + (int)((d >> 9) & 511u);          // row of the first down step
        const int32_t* cp = sc + i0;
        const float* vp = sv + i0;
        float* yp = y_row(y0);                                 // the row that ends next
        VT sum = V::zero();
        VT xv[KS];
        if (any) {
#pragma unroll
          for (int k = 0; k < KS; ++k) {
            const int col = cp[k];                             // step k takes nonzero k - downs before
            spmm_load(x_row((rm >> k) & 1u ? col : col0), xv[k]);
            if ((dm >> k) & 1u) --cp;
          }
        }
        if (p == T - 1) columns_read();
        // the walk tests the masks anew: bits kept from the gathers would hold 28 registers
        uint32_t rw = rm, dw = dm;
        asm volatile("" : "+r"(rw), "+r"(dw));
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          const float w = vp[k];
          if ((rw >> k) & 1u) V::fma(w, xv[k], sum);
          V::store_shared_if(first & (1u << k), s_head, sum);
          spmm_store_if<VW, YVEC, SCALED>((dw ^ first) & c_ok & (1u << k), yp, sum, out.scale, left);
          if ((dw >> k) & 1u) {
            sum = V::zero();
            yp += out.ldy;
            --vp;
          }
        }
        // inclusive scan of the open runs over the pass's lanes (threads of one slice are T
        // apart); a lane that ends a row starts a new run
        const bool hd = dm != 0u;
        __syncwarp();
        const uint32_t slice = (uint32_t)(0xffffffffull / ((1ull << T) - 1ull)) << (lane % T);   // this slice's threads
        const uint32_t heads = __ballot_sync(0xffffffffu, hd);
        const uint32_t upto = heads & slice & (0xffffffffu >> (31 - lane));
        const int dist = (upto ? lane - (31 - __clz(upto)) : lane) / T;
        uint32_t run = ~heads & (T < 32 ? ~((1u << (T & 31)) - 1u) : 0u);   // threads that continue a run
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
          if (run == 0u) break;                                // no run is longer
          const VT up = V::shfl_up(sum, o * T);
          if (o <= dist) V::add(sum, up);
          run &= run >> (o * T);
        }
        VT in = V::zero();                                     // the run that reaches this lane
        if constexpr (L > 1) {
          const VT up = V::shfl_up(sum, T);
          if (gl > 0) in = up;
        }
        if (hd) {
          V::add(in, V::load_shared(s_head));
          if ((upto & (upto - 1u)) == 0u) {                    // the pass's first row
            V::add(in, V::load_shared(s_lost));
            V::add(in, V::load_shared(s_carry));
          }
          if (y0 == y_unit) {
            if (c_ok) add_acc(t_start, in, V::zero());
          } else {
            spmm_store_if<VW, YVEC, SCALED>(c_ok, y_row(y0), in, out.scale, left);
          }
        }
        __syncwarp();
        if (heads == 0u) {
          if (gl == L - 1) extend_run(sum);                      // the whole pass belongs to the run
        } else {
          if (gl == L - 1) {
            V::store_shared(s_carry, sum);
            V::store_shared(s_lost, V::zero());
          }
        }
      }
    }
    __syncwarp();
    if (next_unit) {
      const int y_end = (int)(__shfl_sync(0xffffffffu, meta, 3) & ~kMsb);
      if (gl == 0) {
        if (c_ok && y_end < g.n_rows) add_acc(t + 1, V::load_shared(s_carry), V::load_shared(s_lost));
        V::store_shared(s_carry, V::zero());
        V::store_shared(s_lost, V::zero());
      }
      if (tn < 0) break;
      ++rd;
      t_start = tn;
      y_unit = (int)(__shfl_sync(0xffffffffu, nmeta, 2) & ~kMsb);
    }
    // every lane has read its values: the value buffer takes the next tile
    fence_proxy_async_smem();
    __syncwarp();
    issue(vals, sv, nmeta, 1);
    t = tn;
    meta = nmeta;
    desc = ndesc;
    par ^= 1u;
  }
}

// Rows of the unit boundaries: Y[r, c] = scale * acc[set][c], accumulator cleared.  Every
// distinct row is written once, by its first boundary.
template <int KC>
__global__ void __launch_bounds__(256) merbit_spmm_finalize_kernel(const Geometry g, double* __restrict__ acc,
                                                                   SpmmOut out) {
  if (out.skip(g.red)) return;
  const int c = g.unit;
  const int nbnd = (g.tile_num + c - 1) / c + 1;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < (int64_t)nbnd * KC; p += stride) {
    const int k = (int)(p / KC), cc = (int)(p % KC);
    const int r = (int)(__ldg(g.tile_y + min(k * c, g.tile_num)) & ~kMsb);
    const int prev = k > 0 ? (int)(__ldg(g.tile_y + (k - 1) * c) & ~kMsb) : -1;
    if (cc >= out.kc || r == prev || r >= g.n_rows) continue;
    double* a = acc + p;
    const double tot = *a;
    *a = 0.0;
    out.y[(int64_t)r * out.ldy + cc] = static_cast<float>(static_cast<double>(out.scale) * tot);
  }
}

// Resident CTAs (of 4 warps) per SM: 16 warps of 128 registers hold 14 slices a thread.  Batches
// of 7 slices at 20 warps took the same time for k <= 8 and 5 % more for k = 32; 12 warps took
// 10 % more for k = 32.  Slices of 8 columns (one 32-byte load) need 168 registers: k = 32 took
// 0.538 ms against 0.466 ms (R-MAT scale 21).
template <int VW>
constexpr int kSpmmCtas = VW == 4 ? 4 : 7;

// Unit length and the number of accumulator sets (unit boundaries) of a plan's SpMM.
inline int spmm_unit(const merbit_plan_s* p) { return walk_unit(p->tile_num, (int64_t)p->num_sms * 16, kTilesPerBlock); }
inline int64_t spmm_sets(const merbit_plan_s* p) {
  const int c = spmm_unit(p);
  return (p->tile_num + c - 1) / c + 1;
}

template <int KC, int VW, bool YVEC, bool SCALED>
cudaError_t launch_spmm(const merbit_plan_s* p, const float* vals, const float* X, int64_t ldx, const SpmmOut& out,
                        double* acc, cudaStream_t st) {
  if (p->nb == 0) return cudaSuccess;
  // A lane's steps are unrolled, 7, 10 or 14 of them: the steps beyond sigma gather for nothing
  // (R-MAT scale 20, k = 32, unrolled 14 times and as here: sigma 5 489 and 419 us, sigma 8 369 and 339).
  auto kern = p->sigma <= 7 ? merbit_spmm_kernel<KC, VW, 7, YVEC, SCALED, kSpmmCtas<VW>>
              : p->sigma <= 10 ? merbit_spmm_kernel<KC, VW, 10, YVEC, SCALED, kSpmmCtas<VW>>
                               : merbit_spmm_kernel<KC, VW, kSigmaMax, YVEC, SCALED, kSpmmCtas<VW>>;
  const void* kp = reinterpret_cast<const void*>(kern);
  const size_t smem = kSpmmWarps * spmm_warp_bytes<VW>(p->sigma);
  int grid = persistent_grid(kp, kSpmmThreads, smem, kSpmmWarps * spmm_warp_bytes<VW>(kSigmaMax), p->num_sms);
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  Geometry g = p->geom();
  g.unit = spmm_unit(p);
  const int64_t units = (p->tile_num + g.unit - 1) / g.unit;
  const int64_t few = std::max<int64_t>((units + kSpmmWarps - 1) / kSpmmWarps, std::min<int64_t>(units, p->num_sms));
  if (grid > few) grid = (int)few;
  const int round = grid * kSpmmWarps;
  const SpmmUnits un{(int)(units / round), (int)(units % round)};
  kern<<<grid, kSpmmThreads, smem, st>>>(g, un, acc, vals, X, ldx, out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t work = (units + 1) * KC;
  const int fgrid = (int)std::min<int64_t>((work + 255) / 256, (int64_t)p->num_sms * 8);
  merbit_spmm_finalize_kernel<KC><<<fgrid, 256, 0, st>>>(g, acc, out);
  return cudaGetLastError();
}

}  // namespace merbit

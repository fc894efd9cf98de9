// Plain PageRank of a small graph in one launch (Sec. 5.5.1): the matrix stays in shared memory.
//
// An update of a graph of a few thousand tiles is a chain of latencies: a launch, the plan's and
// the matrix's reads, the gathers, the arrival count of the CTAs, the second pass over the rows
// shared between units.  Here a cooperative launch of at most one CTA per SM copies a tile into
// every warp's shared memory once and runs all updates; what is left of the chain is the gathers, the
// walk and two grid barriers (the rows shared between tiles are finished between them).  No FP64
// atomics: on neighbouring words from many SMs they took 5,000 cycles and more.  A tile stores its
// share of its first row and of the row open at its end, and the first tile that starts in a row
// adds the row's shares up; the CTAs store their sums, and all of them add all up in the same order
// while their next gathers are in flight, so all take the same stop decision.
// 100 f32 updates at R-MAT scale 14 (546 tiles): 1.80 ms with a launch per update, 1.06 ms.
#include "spmv_kernel.cuh"

namespace merbit {

namespace {

constexpr int kResWarps = 16;          // most warps of a CTA

struct ResidentParams {
  double alpha, inv_n, tol;
  const uint32_t* dang;
  double* head;                        // per tile: its share of its first row, if the row ends in it
  double* tail;                        // per tile: its share of the row open at its end
  double* hist;                        // [k][2]: L1 size of update k - 1, dangling mass of iterate k
  int max_iter;
};

// Gathers of an iterate that other SMs wrote before the last grid barrier: plain loads, cached in
// L1 until the barrier's fence drops its lines (the read-only path could return older ones; loads
// past L1 all queue at the few L2 slices that hold a power-law graph's hottest columns).
__device__ __forceinline__ void gather_weak_if(float& v, const float* p, uint32_t pred) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.f32 %0, [%1];\n\t}"
               : "=f"(v) : "l"(p), "r"(pred) : "memory");
}
__device__ __forceinline__ void gather_weak_if(double& v, const double* p, uint32_t pred) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.f64 %0, [%1];\n\t}"
               : "=d"(v) : "l"(p), "r"(pred) : "memory");
}

__device__ __forceinline__ float ld_weak(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_weak(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}

// A warp's shared memory: its tile's values, columns and row sums.
template <typename T>
__host__ __device__ constexpr size_t resident_warp_bytes(int sigma) {
  return (2 * sizeof(T) + sizeof(int32_t)) * (size_t)walk_cap(sigma);
}

// The double equal to f, by integer operations (nothing is rounded): a conversion instruction runs
// in the FP64 pipe, which takes two lanes per SM and clock, and the tiles of empty rows are bound
// by it.  Subnormals, infinities and NaN take the conversion.
__device__ __forceinline__ double exact64(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t mag = u & 0x7fffffffu;
  if (mag - 1u < 0x007fffffu || mag >= 0x7f800000u) return static_cast<double>(f);
  const uint32_t hi = (mag >> 3) + (mag ? 0x38000000u : 0u);
  return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}
__device__ __forceinline__ double exact64(double f) { return f; }

// The warp's sums of a (in lanes 0-15) and of b (in lanes 16-31), in one butterfly.
__device__ __forceinline__ double pair_sum(double a, double b, int lane) {
  const bool low = lane < 16;
  double q = (low ? a : b) + __shfl_xor_sync(0xffffffffu, low ? b : a, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  return q;
}

template <typename T>
__global__ void __launch_bounds__(kResWarps * 32, 1)
    pagerank_resident_kernel(const Geometry g, const ResidentParams p, const T* __restrict__ vals, T* x0, T* x1) {
  __shared__ __align__(8) uint64_t bars[kResWarps];
  __shared__ double sums[kResWarps][2];
  __shared__ int more_of[kResWarps];   // rows of each warp's tile beyond its first 32
  __shared__ int go;                   // the CTA goes on (cleared when a wait gave up anywhere)
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int warps = blockDim.x >> 5, G = gridDim.x;
  const int cap = walk_cap(g.sigma);

  // this warp's tile: w G + b, so that runs of tiles with many (empty) rows are spread over the CTAs
  const int t = warp * G + (int)blockIdx.x;
  const bool has = t < g.tile_num;
  auto row_sums = [&](int w) {
    return reinterpret_cast<T*>(dyn_smem + (size_t)w * resident_warp_bytes<T>(g.sigma) + (sizeof(T) + sizeof(int32_t)) * (size_t)cap);
  };
  T* const sv = reinterpret_cast<T*>(dyn_smem + (size_t)warp * resident_warp_bytes<T>(g.sigma));
  int32_t* const sc = reinterpret_cast<int32_t*>(sv + cap);
  T* const sy = row_sums(warp);
  if (tid == 0) go = 1;
  if (lane == 0) {
    mbar_init(&bars[warp], 1);
    fence_mbar_init();
  }
  __syncthreads();
  int xs = 0, xe = 0, y_ws = 0, n_t = 0, span = 0;
  bool single = false, own = false;
  uint32_t desc = 0;
  if (has) {
    xs = (int)__ldg(g.tile_x + t);
    xe = (int)__ldg(g.tile_x + t + 1);
    const uint32_t tys = __ldg(g.tile_y + t);
    single = (tys & kMsb) != 0u;
    y_ws = (int)(tys & ~kMsb);
    n_t = (int)(__ldg(g.tile_y + t + 1) & ~kMsb) - y_ws;       // rows that end in the tile
    const int j = t * kOmega + lane;
    desc = j < g.lane_num ? __ldg(g.lane_desc + j) : 0u;
  }
  const WalkSpan<T> vspan(xs, xe, g.nnz);
  const WalkSpan<int32_t> cspan(xs, xe, g.nnz);
  if (lane == 0 && has) {
    const uint32_t vb = (uint32_t)(vspan.end - vspan.a0) * (uint32_t)sizeof(T), cb = (uint32_t)(cspan.end - cspan.a0) * 4u;
    mbar_arrive_expect_tx(&bars[warp], vb + cb);
    if (vb) bulk_g2s(sv, vals + vspan.a0, vb, &bars[warp], policy_evict_first());
    if (cb) bulk_g2s(sc, g.col + cspan.a0, cb, &bars[warp], policy_evict_first());
  }
  // the tile's first row: the first tile that starts in it owns it, `span` tiles start in it
  uint32_t word = 0;                   // dangling bits of rows y_ws + lane
  if (has) {
    if (y_ws + lane < g.n_rows) word = __ldg(p.dang + ((y_ws + lane) >> 5));
    own = __ldg(g.tile_slot + t) == t;
    if (own) {
      int lo = t + 1, hi = g.tile_num;          // the first tile boundary in a later row
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((int)(__ldg(g.tile_y + mid) & ~kMsb) > y_ws) hi = mid; else lo = mid + 1;
      }
      span = lo - t;
    }
  }
  const bool ok = !has || mbar_wait_bounded(&bars[warp], 0u, g.wait_limit);
  if (!__all_sync(0xffffffffu, ok)) {
    if (lane == 0) {
      atomicOr(&g.red->err, 1);
      go = 0;
      mbar_wait_bounded(&bars[warp], 0u);
    }
  } else if (has) {
    // the arrays' last nonzeros, short of a whole 16-byte unit
    for (int k = vspan.end + lane; k < xe; k += 32) sv[k - vspan.a0] = vals[k];
    for (int k = cspan.end + lane; k < xe; k += 32) sc[k - cspan.a0] = __ldg(g.col + k);
  }
  // A tile of empty rows has up to 448 of them, and at one warp's FP64 rate every other CTA would
  // wait for it: the rows beyond a tile's first 32 are spread over the CTA.
  const int more = max(0, n_t - 32);
  if (lane == 0) more_of[warp] = more;
  const bool any_more = __syncthreads_or(more) != 0;

  const int j = t * kOmega + lane;
  const int len = has && j < g.lane_num ? min(g.sigma, g.steps - j * g.sigma) : 0;
  const uint32_t valid = (1u << len) - 1u;
  const uint32_t dm = single ? 0u : (desc >> 18) & valid, rm = single ? 0u : ~(desc >> 18) & valid;
  const int xo = (int)(desc & 511u), y0 = (int)((desc >> 9) & 511u);
  const int32_t* const cp0 = sc + (xs - cspan.a0) + (single ? lane : xo);
  const T* const vp0 = sv + (xs - vspan.a0) + (single ? lane : xo);

  unsigned int phase = 0;              // grid barriers passed
  auto arrive = [&]() {                // one thread, after the CTA's __syncthreads
    __threadfence();
    atomicAdd(&g.red->bar, 1u);
  };
  auto wait = [&]() {                  // one thread; false if the barrier does not fill up
    const unsigned int want = kBarStart + phase * (unsigned int)G;
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
      if ((int)(*reinterpret_cast<volatile unsigned int*>(&g.red->bar) - want) >= 0) {   // also past the wrap
        __threadfence();
        return true;
      }
      if ((i & 63u) == 63u && *reinterpret_cast<volatile int*>(&g.red->err)) return false;
    }
    atomicOr(&g.red->err, 1);
    return false;
  };

  if (go) {
    for (int it = 0;; ++it) {
      const T* xin = it & 1 ? x1 : x0;
      T* xout = it & 1 ? x0 : x1;
      // the CTAs' sums of the iterate and the gathers, all in flight together
      double qa = 0.0, qd = 0.0;
      if (it > 0) {
        for (int i = lane; i < G; i += 32) {
          const double2 v = __ldcg(g.part + i);
          qa += v.x;
          qd += v.y;
        }
      } else if (lane == 0) {
        qd = p.hist[1];
      }
      T xv[kSigmaMax];
      T old = T(0);                    // the old values of rows y_ws + lane
      if (has && it < p.max_iter) {
        if (!single) {
          const int32_t* cp = cp0;
#pragma unroll
          for (int k = 0; k < kSigmaMax; ++k) {
            const int col = cp[k];
            gather_weak_if(xv[k], xin + col, rm & (1u << k));
            if ((dm >> k) & 1u) --cp;
          }
        } else {
#pragma unroll
          for (int k = 0; k < kSigmaMax; ++k) {
            const bool in = lane + 32 * k < xe - xs;
            const int col = in ? cp0[32 * k] : 0;
            gather_weak_if(xv[k], xin + col, in);
          }
        }
        if (y_ws + lane < g.n_rows) old = ld_weak(xin + (y_ws + lane));
      }
      const double q = pair_sum(qa, qd, lane);
      const double step = __shfl_sync(0xffffffffu, q, 0), mass = __shfl_sync(0xffffffffu, q, 16);
      if (blockIdx.x == 0 && tid == 0) {
        p.hist[2 * it] = step;
        p.hist[2 * it + 1] = mass;
      }
      if (it > 0 && p.tol > 0.0 && step < p.tol) {
        if (blockIdx.x == 0 && tid == 0) {
          g.red->iters = it;
          g.red->done = 1;
        }
        break;
      }
      if (it == p.max_iter) break;
      const double cd = (p.alpha * mass + 1.0 - p.alpha) * p.inv_n;
      double p0 = 0.0, p1 = 0.0;
      auto put = [&](int r, double s, T before, uint32_t bits) {
        const double vd = fma(p.alpha, s, cd);
        const T v = static_cast<T>(vd);
        xout[r] = v;
        p0 += fabs(vd - exact64(before));
        if ((bits >> (r & 31)) & 1u) p1 += exact64(v);
      };
      if (has) {
        const T carry = single ? walk_row<T, T, T>(vp0, xv, xe - xs - lane)
                               : walk_lanes<T, T, T>(vp0, xv, rm, dm, sy, y0, T(0), lane);
        __syncwarp();
        if (lane < n_t) {
          const T s = sy[lane];
          if (lane == 0) __stcg(p.head + t, static_cast<double>(s));
          else put(y_ws + lane, exact64(s), old, word);
        }
        if (lane == 0) __stcg(p.tail + t, static_cast<double>(carry));
      }
      if (any_more) {
        __syncthreads();
        for (int w = 0; w < warps; ++w) {
          const int m = more_of[w];
          if (m == 0) continue;
          const int y_w = (int)(__ldg(g.tile_y + (w * G + (int)blockIdx.x)) & ~kMsb) + 32;
          const T* const s_w = row_sums(w) + 32;
          for (int r = tid; r < m; r += (int)blockDim.x)
            put(y_w + r, exact64(s_w[r]), ld_weak(xin + (y_w + r)), __ldg(p.dang + ((y_w + r) >> 5)));
        }
      }
      // barrier: every tile's shares are stored
      ++phase;
      __syncthreads();
      if (tid == 0) arrive();
      const double mine = pair_sum(p0, p1, lane);    // lane 0: p0, lane 16: p1
      if (tid == 0 && !wait()) go = 0;
      __syncthreads();
      if (!go) break;
      p0 = p1 = 0.0;
      if (own) {
        // the row's shares: the tail of the tile before the first that starts in it, those of all
        // these tiles but the last, and the head of the last, in which the row ends
        double s = lane == 0 ? __ldcg(p.head + (t + span - 1)) : 0.0;
        for (int i = lane; i < span; i += 32)
          if (t + i > 0) s += __ldcg(p.tail + (t + i - 1));
        if (span > 1) s = warp_sum(s);
        if (lane == 0) put(y_ws, s, old, word);
      }
      p1 = __shfl_sync(0xffffffffu, p1, 0);
      if (lane == 0) sums[warp][0] = mine + p0;
      if (lane == 16) sums[warp][1] = mine + p1;
      ++phase;
      __syncthreads();
      if (warp == 0) {
        double a = lane < 2 * warps ? sums[lane >> 1][lane & 1] : 0.0;
#pragma unroll
        for (int o = kResWarps; o > 1; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        const double d = __shfl_sync(0xffffffffu, a, 1);
        if (lane == 0) {
          __stcg(g.part + blockIdx.x, make_double2(a, d));
          arrive();
          if (!wait()) go = 0;
        }
      }
      __syncthreads();
      if (!go) break;
    }
  }
}

template <typename T>
cudaError_t run_resident(merbit_plan_s* p, const T* vals, const ResidentParams& prm, T* x0, T* x1, bool* taken,
                         cudaStream_t st) {
  *taken = false;
  if (p->spmv_kernel != MERBIT_KERNEL_AUTO || !walk_takes(p) || p->nb == 0) return cudaSuccess;
  // one tile a warp, at most 16 warps a CTA and one CTA per SM; few tiles: four to a CTA, so that
  // fewer CTAs meet at the barriers.  More tiles a warp gather one tile after the other and lose to a
  // launch per update (R-MAT-like graphs, f32: 65,536 vertices 16.6 us an update against 26.4; with
  // two tiles a warp 100,000 vertices 24.9 against 28.6, with three 150,000 vertices 37.4 against 32.6).
  const int grid = (int)std::min<int64_t>((p->tile_num + 3) / 4, std::min(p->num_sms, kMaxParts));
  const int64_t per_cta = (p->tile_num + grid - 1) / grid;
  if (per_cta > kResWarps) return cudaSuccess;
  const int warps = (int)per_cta;
  const size_t smem = (size_t)warps * resident_warp_bytes<T>(p->sigma);
  auto kern = pagerank_resident_kernel<T>;
  const void* kp = reinterpret_cast<const void*>(kern);
  int coop = 0;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, p->device);
  if (!coop || persistent_grid(kp, warps * 32, smem, kResWarps * resident_warp_bytes<T>(kSigmaMax), 1) < 1)
    return cudaSuccess;
  Geometry g = p->geom();
  ResidentParams params = prm;
  void* args[] = {&g, &params, &vals, &x0, &x1};
  cudaError_t e = cudaLaunchCooperativeKernel(kp, dim3(grid), dim3(warps * 32), args, smem, st);
  if (e != cudaSuccess) {
    // not co-resident here (a shared or partitioned device): the launch per update
    cudaGetLastError();
    return cudaSuccess;
  }
  *taken = true;
  return cudaSuccess;
}

}  // namespace

cudaError_t pagerank_resident(merbit_plan_s* p, merbit_dtype dt, const void* vals, double alpha, double tol,
                              int max_iter, void* x0, void* x1, double* hist, double* shares, bool* taken,
                              cudaStream_t st) {
  ResidentParams prm;
  prm.head = shares;
  prm.tail = shares + p->tile_num;
  prm.alpha = alpha;
  prm.inv_n = 1.0 / (double)p->n_rows;
  prm.tol = tol;
  prm.dang = p->dangling_bits;
  prm.hist = hist;
  prm.max_iter = max_iter;
  if (dt == MERBIT_F64)
    return run_resident<double>(p, static_cast<const double*>(vals), prm, static_cast<double*>(x0), static_cast<double*>(x1),
                                taken, st);
  return run_resident<float>(p, static_cast<const float*>(vals), prm, static_cast<float*>(x0), static_cast<float*>(x1), taken,
                             st);
}

}  // namespace merbit

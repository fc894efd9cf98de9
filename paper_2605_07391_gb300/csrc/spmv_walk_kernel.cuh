// The lane-walk SpMV kernel: every warp works on its own, from the copy of a tile's
// matrix data to its finished rows (included by spmv_kernel.cuh).
//
// A warp takes a unit of c consecutive tiles.  Per tile (Sec. 4.1):
//   1. the tile's column indices are in the warp's shared memory (one bulk copy); each
//      lane gathers x for all the right steps of its descriptor into registers;
//   2. the columns of the warp's next tile are copied into the same place while those
//      gathers are in flight;
//   3. each lane walks its steps: a right step adds val * x (one fused multiply-add) to
//      the running sum, a down step ends a row.  Rows that begin and end inside the lane
//      are stored at once; the lane's first row end is kept (`head`);
//   4. the runs open at the lanes' ends are joined by a segmented shuffle scan, a lane's
//      first row totals its head plus the run that reaches it, and the run open after the
//      tile is carried in a register into the next tile of the unit (with 4-byte sums, a
//      second one holds what whole tiles of one row lost to rounding);
//   5. the tile's rows go through the epilogue, consecutive lanes to consecutive rows, and
//      the next tile's values are copied in.
// So columns and values need one buffer each per warp: a column buffer is free once the
// gathers are issued, a value buffer once the rows are written, and the other phase of the
// tile hides each copy.  No step synchronises more than a warp.  Only a unit's first row
// and the row open at its end can belong to other units too; they are added into FP64
// accumulators, one per distinct row at a tile boundary, which a second pass
// (finish_bounds) writes out and clears.
//
// What bounds it.  f32: the rate at which an SM's L1 takes gathers (their misses go to L2
// one line at a time, and the most used columns sit in few L2 slices: at R-MAT scale 21 the
// busiest slice runs at 80 % of its peak).  With 32 warps of 14 gathers per lane there are
// up to 14,336 gathers in flight per SM, twice the split kernel's; a warp instruction count
// of 1.4 per nonzero instead of 2.4 (no atomics on shared memory, no zeroed sums, one pass
// over the products) leaves the load path to them.  R-MAT scale 24, f32: 1.158 -> 0.99 ms (0.93 to 1.03 on
// other boxes).
// f64: this GPU has two FP64 lanes per SM and clock, so a warp instruction of FP64 holds the
// SM's pipe for 16 cycles; the fused multiply-add halves the work per nonzero (the split
// kernel multiplies, stores and adds) and row ends cost one add instead of two atomics.
// R-MAT scale 22 with 30 % empty rows, f64: 0.336 -> 0.203 ms (pipe 56 % busy at 0.215).
#pragma once

namespace merbit {

// Elements of a tile's buffer in the kernels that share the walk: its 32 sigma steps, up to 7
// elements of alignment before its first nonzero, and the walk's reads past a lane's last product.
__host__ __device__ constexpr int walk_cap(int sigma) { return kOmega * sigma + 32; }

// This kernel's buffers are as small as the copies allow.  Values: the tile's nonzeros with less
// than 16 bytes before and after them (the copy's boundaries), and at the buffer's end the tile's
// row sums; nonzeros and rows are at most 32 sigma together.  Columns: the nonzeros with less than
// 16 bytes on either side.  What a lane reads past its last product (13 elements, never used)
// lies in the buffer behind, or in the CTA's kWalkTail bytes.  That leaves three f64 CTAs at
// sigma 14 (131 KB with the system's share) the next smaller carveout of shared memory, and L1 32
// KB more than with 32 elements of slack in each buffer (139 KB): R-MAT scale 24, f64, 1.324 ms
// and 1.155; scale 22 with 30 % empty rows 0.214 and 0.203.
template <typename VT, typename AT>
__host__ __device__ constexpr size_t walk_val_bytes(int sigma) {
  return (sizeof(VT) > sizeof(AT) ? sizeof(VT) : sizeof(AT)) * (size_t)(kOmega * sigma) + 32;
}
template <typename VT, typename AT>
__host__ __device__ constexpr size_t walk_warp_bytes(int sigma) {
  return walk_val_bytes<VT, AT>(sigma) + sizeof(int32_t) * (size_t)(kOmega * sigma) + 32;
}
constexpr size_t kWalkTail = 128;

__device__ __forceinline__ void gather_if(float& v, const float* p, uint32_t pred, uint64_t pol) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t"
      "@q ld.global.nc.L2::cache_hint.f32 %0, [%1], %3;\n\t}"
      : "=f"(v)
      : "l"(p), "r"(pred), "l"(pol));
}
__device__ __forceinline__ void gather_if(double& v, const double* p, uint32_t pred, uint64_t pol) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t"
      "@q ld.global.nc.L2::cache_hint.f64 %0, [%1], %3;\n\t}"
      : "=d"(v)
      : "l"(p), "r"(pred), "l"(pol));
}

__device__ __forceinline__ float mul_add(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mul_add(double a, double b, double c) { return fma(a, b, c); }

// The warp's bulk copies of a tile: nonzeros [a0, end) of the array, from the 16-byte
// boundary at or before the tile's first nonzero to the one at or after its last, inside the
// array's whole 16-byte units.
template <typename T>
struct WalkSpan {
  static constexpr int E = 16 / (int)sizeof(T);
  int a0, end;
  __device__ __forceinline__ WalkSpan(int xs, int xe, int nnz) {
    a0 = xs & ~(E - 1);
    end = max(a0, min((xe + E - 1) & ~(E - 1), nnz & ~(E - 1)));
  }
};

template <typename T>
__device__ __forceinline__ void walk_issue(const T* src, void* dst, int xs, int xe, int nnz, uint64_t* bar,
                                           uint64_t pol) {
  const WalkSpan<T> sp(xs, xe, nnz);
  const uint32_t bytes = (uint32_t)(sp.end - sp.a0) * (uint32_t)sizeof(T);
  mbar_arrive_expect_tx(bar, bytes);
  if (bytes) bulk_g2s(dst, src + sp.a0, bytes, bar, pol);
}

// s + x, and what the sum lost to rounding added to `lost` (Knuth's two-sum; nothing is lost by a
// sum that is not finite).
__device__ __forceinline__ void add_lost(float& s, float& lost, float x) {
  const float t = s + x;
  const float z = t - s;
  const float e = (s - (t - z)) + (x - z);
  lost += isfinite(t) ? e : 0.f;
  s = t;
}

// The walk of one tile by a warp: a lane's steps (rm: right steps, dm: down steps; vp its first
// value; xv its gathered x), the row sums into sy (y0: the row of the lane's first down step), the
// runs joined across the lanes.  carry is the run that reaches the tile (4-byte sums: added last
// where it ends); the run open after the tile is returned, in every lane.
template <typename VT, typename XT, typename AT>
__device__ __forceinline__ AT walk_lanes(const VT* vp, const XT (&xv)[kSigmaMax], uint32_t rm, uint32_t dm, AT* sy,
                                         int y0, AT carry, int lane) {
  const uint32_t first = dm & (0u - dm);             // the lane's first down step
  const uint32_t later = dm ^ first;
  AT* rp = sy + y0;
  AT sum = AT(0), head = AT(0);
#pragma unroll
  for (int k = 0; k < kSigmaMax; ++k) {
    if constexpr (!IsUnit<VT>::value) {
      const AT v = static_cast<AT>(widen(vp[k]));
      if ((rm >> k) & 1u) sum = mul_add(v, static_cast<AT>(xv[k]), sum);
    } else {
      if ((rm >> k) & 1u) sum += static_cast<AT>(xv[k]);
    }
    if ((first >> k) & 1u) head = sum;
    if ((later >> k) & 1u) *rp = sum;
    if ((dm >> k) & 1u) {
      sum = AT(0);
      ++rp;
      --vp;
    }
  }
  // inclusive scan of the open runs; a lane that ends a row starts a new run
  const bool hd = dm != 0u;
  const uint32_t heads = __ballot_sync(0xffffffffu, hd);
  if constexpr (sizeof(AT) == 8) {                    // one add fewer for the FP64 pipe
    if (lane == 0 && !hd) sum += carry;
  }
  const uint32_t upto = heads & (0xffffffffu >> (31 - lane));
  const int dist = upto ? lane - (31 - __clz(upto)) : lane;   // lanes back to the run's start
  uint32_t run = ~heads & ~1u;                        // lanes that continue a run
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (run == 0u) break;                             // no run is longer (the same in every lane)
    const AT up = __shfl_up_sync(0xffffffffu, sum, o);
    if (o <= dist) sum += up;
    run &= run >> o;
  }
  // the run that reaches this lane's first row
  const AT up = __shfl_up_sync(0xffffffffu, sum, 1);
  if constexpr (sizeof(AT) == 8) {
    if (hd) sy[y0] = head + (lane == 0 ? carry : up);
  } else if (hd) {
    AT s = lane > 0 ? head + up : head;
    if ((upto & (upto - 1u)) == 0u) s += carry;       // the tile's first row
    sy[y0] = s;
  }
  return __shfl_sync(0xffffffffu, sum, 31);
}

// The sum of a tile of one row: lanes take every 32nd nonzero (vp, left: from the lane's first).
template <typename VT, typename XT, typename AT>
__device__ __forceinline__ AT walk_row(const VT* vp, const XT (&xv)[kSigmaMax], int left) {
  AT sum = AT(0);
#pragma unroll
  for (int k = 0; k < kSigmaMax; ++k) {
    if (32 * k < left) {
      if constexpr (!IsUnit<VT>::value) sum = mul_add(static_cast<AT>(widen(vp[32 * k])), static_cast<AT>(xv[k]), sum);
      else sum += static_cast<AT>(xv[k]);
    }
  }
  return warp_sum(sum);
}

// Boundary k of the units (c tiles each): the row open there.  Every distinct row of the
// unit boundaries is written once, by its first boundary, from its FP64 accumulator.
template <typename Epi>
__device__ __forceinline__ void finish_bounds(const Geometry& g, const Epi& epi, int t0, int stride,
                                              double& p0, double& p1) {
  const int c = g.unit;
  const int nbnd = (g.tile_num + c - 1) / c + 1;
  constexpr int U = 4;             // boundaries in flight per thread
  for (int k0 = t0; k0 < nbnd; k0 += U * stride) {
    int r[U], slot[U];
    bool own[U];
    double tot[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + u * stride;
      own[u] = k < nbnd;
      r[u] = slot[u] = 0;
      if (own[u]) {
        const int i = min(k * c, g.tile_num);
        r[u] = (int)(__ldg(g.tile_y + i) & ~kMsb);
        const int prev = k > 0 ? (int)(__ldg(g.tile_y + (k - 1) * c) & ~kMsb) : -1;
        slot[u] = __ldg(g.tile_slot + i);
        own[u] = r[u] != prev && r[u] < g.n_rows;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      tot[u] = 0.0;
      if (own[u]) tot[u] = __ldcg(g.tile_acc + slot[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!own[u]) continue;
      __stcg(g.tile_acc + slot[u], 0.0);
      epi.row64(r[u], tot[u], p0, p1);
    }
  }
}

template <typename Epi>
__global__ void __launch_bounds__(256) merbit_walk_finalize_kernel(const Geometry g, Epi epi, int nparts) {
  if (epi.skip(g.red)) return;
  epi.init();
  double p0 = 0.0, p1 = 0.0;
  const int stride = gridDim.x * blockDim.x;
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
  finish_bounds(g, epi, t0, stride, p0, p1);
  if constexpr (Epi::kReduce) {
    for (int i = t0; i < nparts; i += stride) {
      const double2 q = g.part[i];
      p0 += q.x;
      p1 += q.y;
    }
    grid_sum2(p0, p1, g.red, [&](double A, double B) { epi.finish(A, B, g.red); });
  }
}

constexpr int kWalkWarps = 8;
constexpr int kWalkThreads = kWalkWarps * 32;

// Sums (p0, p1) over the CTA's threads; the result is in thread 0.
__device__ __forceinline__ void walk_cta_sum(double& p0, double& p1, double (*smem)[2]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  p0 = warp_sum(p0);
  p1 = warp_sum(p1);
  if (lane == 0) {
    smem[warp][0] = p0;
    smem[warp][1] = p1;
  }
  __syncthreads();
  if (warp == 0) {
    p0 = lane < kWalkWarps ? smem[lane][0] : 0.0;
    p1 = lane < kWalkWarps ? smem[lane][1] : 0.0;
#pragma unroll
    for (int o = kWalkWarps / 2; o > 0; o >>= 1) {
      p0 += __shfl_down_sync(0xffffffffu, p0, o);
      p1 += __shfl_down_sync(0xffffffffu, p1, o);
    }
  }
}

template <typename VT, typename XT, typename AT, typename Epi, int CTAS>
__global__ void __launch_bounds__(kWalkThreads, CTAS)
    merbit_spmv_walk_kernel(const Geometry g, const VT* __restrict__ vals, const XT* __restrict__ x, Epi epi) {
  constexpr bool kVals = !IsUnit<VT>::value;
  __shared__ __align__(8) uint64_t bars[kWalkWarps][2];
  __shared__ double red_smem[kWalkWarps][2];
  __shared__ int failed;
  extern __shared__ __align__(128) unsigned char dyn_smem[];

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  const int G = gridDim.x;
  if (epi.skip(g.red)) return;
  epi.init();

  const uint64_t pol_stream = policy_evict_first();
  const uint64_t pol_x = policy_evict_last();
  const BlockOrder<Epi> blk(g, epi);
  // units in the order of the blocks; c divides W
  const int c = g.unit;
  const int per_blk = g.W / c;
  const int nunits = blk.n * per_blk;
  // Whole rounds give consecutive units to a CTA's warps (they share x lines in L1); the
  // units left over are spread over the CTAs first, so every SM has its share.
  const int round = G * kWalkWarps;
  const int nfull = nunits / round;
  const int rest = nunits - nfull * round;
  const int mine = nfull + (warp * G + (int)blockIdx.x < rest ? 1 : 0);
  auto first_tile = [&](int r) {
    const int u = r < nfull ? r * round + (int)blockIdx.x * kWalkWarps + warp : nfull * round + warp * G + (int)blockIdx.x;
    return blk(u / per_blk) * g.W + (u % per_blk) * c;
  };

  unsigned char* base = dyn_smem + (size_t)warp * walk_warp_bytes<VT, AT>(g.sigma);
  VT* const sv = reinterpret_cast<VT*>(base);
  AT* const sy_end = reinterpret_cast<AT*>(base + walk_val_bytes<VT, AT>(g.sigma));
  int32_t* const sc = reinterpret_cast<int32_t*>(base + walk_val_bytes<VT, AT>(g.sigma));
  uint64_t* const bar_c = &bars[warp][0];
  uint64_t* const bar_v = &bars[warp][1];

  if (tid == 0) failed = 0;
  if (lane == 0) {
    mbar_init(bar_c, 1);
    mbar_init(bar_v, 1);
    fence_mbar_init();
  }
  __syncthreads();

  double p0 = 0.0, p1 = 0.0;
  // the tile in work, and what is known of the next one
  int rd = 0;                       // round of the current unit
  int t = 0;                        // current tile
  int t_start = 0, t_end = 0;       // its unit
  uint32_t txs = 0, txe = 0, tys = 0, tye = 0, desc = 0;
  auto load_meta = [&](int ti, uint32_t& a, uint32_t& b, uint32_t& ya, uint32_t& yb, uint32_t& d) {
    a = __ldg(g.tile_x + ti);
    b = __ldg(g.tile_x + ti + 1);
    ya = __ldg(g.tile_y + ti);
    yb = __ldg(g.tile_y + ti + 1) & ~kMsb;
    const int j = ti * kOmega + lane;
    d = j < g.lane_num ? ld_stream(g.lane_desc + j, pol_stream) : 0u;
  };
  // the first tile of round r's unit, or -1 (a unit past the path's last tile is empty)
  auto unit_start = [&](int r) {
    if (r >= mine) return -1;
    const int ti = first_tile(r);
    return ti < g.tile_num ? ti : -1;
  };
  t = mine > 0 ? unit_start(0) : -1;
  if (t >= 0) {
    t_start = t;
    t_end = min(t + c, g.tile_num);
    load_meta(t, txs, txe, tys, tye, desc);
    if (lane == 0) {
      walk_issue(g.col, sc, (int)txs, (int)txe, g.nnz, bar_c, pol_stream);
      if constexpr (kVals) walk_issue(vals, sv, (int)txs, (int)txe, g.nnz, bar_v, pol_stream);
    }
  }
  uint32_t par = 0;
  AT carry = AT(0);                 // run open after the unit's tiles so far
  float lost = 0.f;                 // what its sum lost to rounding (4-byte sums)
  int y_unit = (int)(tys & ~kMsb);  // the unit's first row
  bool ok = true;
  while (t >= 0) {
    // the tile after this one, of this unit or of the next
    int tn = t + 1;
    bool next_unit = false;
    if (tn >= t_end) {
      next_unit = true;
      tn = unit_start(rd + 1);
    }
    uint32_t nxs = 0, nxe = 0, nys = 0, nye = 0, ndesc = 0;
    if (tn >= 0) load_meta(tn, nxs, nxe, nys, nye, ndesc);

    const int xs = (int)txs, xe = (int)txe;
    const int y_ws = (int)(tys & ~kMsb);
    const int n_t = (int)tye - y_ws;                 // rows that end in this tile
    const bool single = (tys & kMsb) != 0u;
    const int j = t * kOmega + lane;
    const int len = j < g.lane_num ? min(g.sigma, g.steps - j * g.sigma) : 0;
    const uint32_t valid = (1u << len) - 1u;
    const uint32_t dm = single ? 0u : (desc >> 18) & valid;    // down steps
    const uint32_t rm = single ? 0u : ~(desc >> 18) & valid;   // right steps
    const int xo = (int)(desc & 511u);
    const int y0 = (int)((desc >> 9) & 511u);

    // ---- gather x for the tile's nonzeros
    if (!mbar_wait_bounded(bar_c, par, g.wait_limit)) ok = false;
    if (__any_sync(0xffffffffu, !ok)) {
      ok = false;
      if (lane == 0) {
        mbar_wait_bounded(bar_c, par);
        if constexpr (kVals) mbar_wait_bounded(bar_v, par);
      }
      break;
    }
    const WalkSpan<int32_t> cspan(xs, xe, g.nnz);
    if (cspan.end < xe) {
      // the array's last nonzeros, short of a whole 16-byte unit
      for (int k = cspan.end + lane; k < xe; k += 32) sc[k - cspan.a0] = __ldg(g.col + k);
      __syncwarp();
    }
    XT xv[kSigmaMax];
    if (!single) {
      const int32_t* cp = sc + (xs - cspan.a0 + xo);
#pragma unroll
      for (int k = 0; k < kSigmaMax; ++k) {
        const int col = cp[k];                       // step k takes nonzero xo + k - downs before
        gather_if(xv[k], x + col, rm & (1u << k), pol_x);
        if ((dm >> k) & 1u) --cp;
      }
    } else {
      // one row: lanes take every 32nd nonzero
      const int32_t* cp = sc + (xs - cspan.a0 + lane);
#pragma unroll
      for (int k = 0; k < kSigmaMax; ++k) {
        const bool in = lane + 32 * k < xe - xs;
        const int col = in ? cp[32 * k] : 0;
        gather_if(xv[k], x + col, in, pol_x);
      }
    }
    // the gathers' addresses have been read: the column buffer takes the next tile
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0 && tn >= 0) walk_issue(g.col, sc, (int)nxs, (int)nxe, g.nnz, bar_c, pol_stream);

    // ---- walk
    int vpad = 0;                                    // the tile's first value in sv
    if constexpr (kVals) {
      if (!mbar_wait_bounded(bar_v, par, g.wait_limit)) ok = false;
      if (__any_sync(0xffffffffu, !ok)) {
        ok = false;
        if (lane == 0) {
          mbar_wait_bounded(bar_v, par);
          if (tn >= 0) mbar_wait_bounded(bar_c, par ^ 1u);
        }
        break;
      }
      const WalkSpan<VT> vspan(xs, xe, g.nnz);
      vpad = xs - vspan.a0;
      if (vspan.end < xe) {
        for (int k = vspan.end + lane; k < xe; k += 32) sv[k - vspan.a0] = vals[k];
        __syncwarp();
      }
    }
    AT* const sy = sy_end - n_t;                     // the tile's row sums
    if (!single) {
      if constexpr (sizeof(AT) == 4) carry += lost;
      carry = walk_lanes<VT, XT, AT>(sv + (vpad + xo), xv, rm, dm, sy, y0, carry, lane);
      lost = 0.f;
    } else {
      const AT s = walk_row<VT, XT, AT>(sv + (vpad + lane), xv, xe - xs - lane);
      if constexpr (sizeof(AT) == 4) add_lost(carry, lost, s);
      else carry += s;
    }
    __syncwarp();

    // ---- commit: the tile's rows; the unit's first row may have begun in another unit
    for (int r = lane; r < n_t; r += 32) {
      const AT s = sy[r];
      if (y_ws + r == y_unit) atomicAdd(g.tile_acc + __ldg(g.tile_slot + t_start), static_cast<double>(s));
      else epi.row(y_ws + r, s, p0, p1);
    }
    if (next_unit) {
      if (lane == 0 && (int)tye < g.n_rows) {
        double run = static_cast<double>(carry);
        if constexpr (sizeof(AT) == 4) run += static_cast<double>(lost);
        atomicAdd(g.tile_acc + __ldg(g.tile_slot + t + 1), run);
      }
      carry = AT(0);
      lost = 0.f;
      ++rd;
    }
    if constexpr (kVals) {
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0 && tn >= 0) walk_issue(vals, sv, (int)nxs, (int)nxe, g.nnz, bar_v, pol_stream);
    } else {
      __syncwarp();
    }
    t = tn;
    txs = nxs; txe = nxe; tys = nys; tye = nye; desc = ndesc;
    if (next_unit) {
      t_start = t;
      t_end = min(t + c, g.tile_num);
      y_unit = (int)(tys & ~kMsb);
    }
    par ^= 1u;
  }
  if (!ok && lane == 0) {
    atomicOr(&g.red->err, 1);
    failed = 1;
  }
  if constexpr (Epi::kReduce) {
    walk_cta_sum(p0, p1, red_smem);
    if (tid == 0) g.part[blockIdx.x] = make_double2(p0, p1);
  }
  if (!g.fold) return;
  // few tiles: the CTA that finishes last runs the second pass.  A CTA that gave up does
  // not arrive, so none finishes the product (the error bit tells the host).
  __shared__ int last;
  __syncthreads();
  if (failed) return;
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(&g.red->arrive, 1u) + 1 == gridDim.x;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  p0 = p1 = 0.0;
  finish_bounds(g, epi, tid, kWalkThreads, p0, p1);
  if constexpr (Epi::kReduce) {
    for (int i = tid; i < G; i += kWalkThreads) {
      const double2 q = __ldcg(g.part + i);
      p0 += q.x;
      p1 += q.y;
    }
    walk_cta_sum(p0, p1, red_smem);
    if (tid == 0) epi.finish(p0, p1, g.red);
  }
  if (tid == 0) g.red->arrive = 0u;
}

// Resident CTAs per SM: 32 warps for 4-byte sums (R-MAT scale 24, on one box: 0.929 ms, 24 warps
// 0.952, 16 warps 1.012), 24 for 8-byte ones, whose buffers (5.3 KB a warp) would leave L1 too
// little at 32 (R-MAT scale 22 with 30 % empty rows, with 46 KB a CTA: 0.216 ms; 32 warps 0.261, 16 warps 0.224).
template <typename AT>
constexpr int kWalkCtas = sizeof(AT) == 8 ? 3 : 4;

// Whether the automatic choice takes the lane-walk kernel for a plan: 32-bit descriptors
// and no hot-column table (the split kernel's).  A plan without tile slots (the
// fixed-scratch entry point) keeps the block kernels.
inline bool walk_takes(const merbit_plan_s* p) {
  return p->tile_slot != nullptr && p->sigma <= kSigmaMax && p->hot_n <= 0;
}

// A unit is as long as leaves every warp two of them, at most four tiles.  Longer units have fewer
// rows in two units (two FP64 atomics and a second-pass row each); shorter ones leave less of a
// round undone at the end and spread a small matrix over more warps.  Against up to eight tiles
// with four units a warp: 64 graphs of 2^10 to 2^18 vertices, f64 (48 tiles a warp) 293 us a
// product, 283; SpMM updates of a personalised PageRank at 16 tiles a warp 1781 us, 1718; a road
// grid's BiCGSTAB iteration (6 tiles a warp) 196 us, 192; uniform 8 M nonzeros, f64, 53.2 us, 49.8.
// One unit a warp: SpMM at 12 tiles a warp 170 us against 153.
constexpr int kUnitMax = 4;
inline int walk_unit(int64_t tiles, int64_t warps, int W) {
  int c = W < kUnitMax ? W : kUnitMax;
  while (c > 1 && tiles < 2 * c * warps) c >>= 1;
  return c;
}

// Products of at most this many unit boundaries are finished by the kernel's last CTA: a launch less,
// but one CTA for all of them.  R-MAT-like graphs, refinement to 1e-10 with this limit at 1,024 and
// at 2,048: 1,237 tiles 2.27 and 2.10 ms, 1,369 tiles 2.69 and 2.55, 1,718 and 1,897 tiles level;
// BiCGSTAB, an iteration: 1,499 tiles 59.2 and 59.9 us.
constexpr int64_t kWalkFoldMax = 1440;

template <typename VT, typename XT, typename AT, typename Epi>
cudaError_t launch_walk(const merbit_plan_s* p, const VT* vals, const XT* x, const Epi& epi, cudaStream_t st) {
  auto kern = merbit_spmv_walk_kernel<VT, XT, AT, Epi, kWalkCtas<AT>>;
  const void* kp = reinterpret_cast<const void*>(kern);
  const size_t smem = kWalkWarps * walk_warp_bytes<VT, AT>(p->sigma) + kWalkTail;
  int grid = persistent_grid(kp, kWalkThreads, smem, kWalkWarps * walk_warp_bytes<VT, AT>(kSigmaMax) + kWalkTail, p->num_sms);
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  Geometry g = p->geom();
  g.unit = walk_unit(p->tile_num, (int64_t)grid * kWalkWarps, p->tiles_per_block);
  const int64_t units = (p->tile_num + g.unit - 1) / g.unit;
  g.fold = units + 1 <= kWalkFoldMax;
  // A small product spreads its units over the SMs, one CTA each, before it gives a CTA's
  // warps more of them: every CTA is one arrival more before the second pass (100 PageRank
  // updates at R-MAT scale 14, 546 tiles: 1.80 ms on 152 CTAs, 2.23 ms on 546).
  const int64_t few = std::max<int64_t>((units + kWalkWarps - 1) / kWalkWarps, std::min<int64_t>(units, p->num_sms));
  if (grid > few) grid = (int)few;
  if (grid > kMaxParts) grid = kMaxParts;
  kern<<<grid, kWalkThreads, smem, st>>>(g, vals, x, epi);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || g.fold) return e;
  const int fgrid = (int)std::min<int64_t>((units + 1 + 255) / 256, (int64_t)p->num_sms * 4);
  merbit_walk_finalize_kernel<Epi><<<fgrid, 256, 0, st>>>(g, epi, Epi::kReduce ? grid : 0);
  return cudaGetLastError();
}

}  // namespace merbit

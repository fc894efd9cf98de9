// Kernels of the differentiation extension.
//
// * EpiAdjoint: the transposed PageRank fixed point.  With M = A + (1/n) 1 d^T the
//   PageRank operator (A = P^T, d the dangling indicator), pi = alpha M pi + (1-alpha)/n 1,
//   and a loss L(pi), the adjoint lambda of (I - alpha M)^T lambda = dL/dpi is the fixed
//   point of lambda' = alpha A^T lambda + alpha (sum(lambda) / n) d + dL/dpi, iterated here
//   by SpMVs on a plan of A^T (the rows of A^T that are empty are exactly the dangling
//   vertices, so every row is written).  dL/dA_ij = alpha lambda_i pi_j.
// * sddmm: out[k] = scale * g[row(k)] * x[col(k)] for every nonzero, walking the
//   plan's lanes (Sec. 4.1.1 descriptors): the value gradient of y = A x is g[row] x[col].
#include "extensions.cuh"
#include "spmv_kernel.cuh"

namespace merbit {

namespace {

template <typename T>
struct EpiAdjoint {
  static constexpr bool kReduce = true;
  AdjParams p;
  const T* xold;
  T a, c;
  __device__ __forceinline__ void init() {
    a = static_cast<T>(p.alpha);
    c = static_cast<T>(p.alpha * (*p.s_in) * p.inv_n);
  }
  __device__ __forceinline__ bool skip(const RedState* red) const {
    return *reinterpret_cast<const volatile int*>(&red->done) != 0;
  }
  __device__ __forceinline__ void put(int r, T v, double& p0, double& p1) const {
    if (is_dangling(p.dang, r)) v += c;
    static_cast<T*>(p.out)[r] = v;
    p0 += fabs(static_cast<double>(v) - static_cast<double>(xold[r]));
    p1 += static_cast<double>(v);
  }
  __device__ __forceinline__ void row(int r, T s, double& p0, double& p1) const {
    put(r, a * s + static_cast<const T*>(p.w)[r], p0, p1);
  }
  __device__ __forceinline__ void row64(int r, double s, double& p0, double& p1) const {
    put(r, static_cast<T>(p.alpha * s + static_cast<double>(static_cast<const T*>(p.w)[r])), p0, p1);
  }
  __device__ __forceinline__ void finish(double A, double B, RedState* red) const {
    p.s_out[0] = A;
    p.s_out[1] = B;
    ++red->launches;
    if (p.tol > 0.0 && A <= p.tol * (*p.wnorm)) {
      red->iters = p.iter + 1;
      red->done = 1;
    }
  }
};

// out[k] = (scale g[row(k)]) x[col(k)], a warp per tile.  The tile's columns are read, x is
// gathered and out is written in the order of the nonzeros, 32 consecutive ones at a time (one
// thread per lane of the schedule, each walking 14 consecutive nonzeros, spread every access of a
// warp over 32 lines).  Row values come from shared memory: the tile's scaled g values are read
// once, in row order, and each lane of the schedule writes them out along its steps while the
// gathers are in flight.  R-MAT scale 20 (16.1 M nonzeros), f32: 124 us before, 62 us; the
// gathers alone take about 63 us (the SpMV's time on this matrix).
constexpr int kSddmmWarps = 8;

template <typename T>
__global__ void __launch_bounds__(kSddmmWarps * 32, sizeof(T) == 8 ? 3 : 4)
    sddmm_kernel(const Geometry g, const T* __restrict__ gv, const T* __restrict__ x, T scale,
                 T* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  constexpr int U = kSigmaMax;                  // nonzeros in flight per lane
  const int lane = threadIdx.x & 31;
  const int per = kOmega * g.sigma + 2;         // a tile's rows (the open one included) and nonzeros
  T* const sg = reinterpret_cast<T*>(sm_raw) + (size_t)(threadIdx.x >> 5) * per;
  const uint64_t pol_stream = policy_evict_first(), pol_x = policy_evict_last();
  const int stride = gridDim.x * kSddmmWarps;
  for (int ti = blockIdx.x * kSddmmWarps + (int)(threadIdx.x >> 5); ti < g.tile_num; ti += stride) {
    const int xs = (int)__ldg(g.tile_x + ti), m = (int)__ldg(g.tile_x + ti + 1) - xs;
    const uint32_t tys = __ldg(g.tile_y + ti);
    const int y_ws = (int)(tys & ~kMsb);
    const int n_t = (int)(__ldg(g.tile_y + ti + 1) & ~kMsb) - y_ws;
    const int j = ti * kOmega + lane;
    const LaneDesc d = j < g.lane_num ? decode_lane(g, load_desc(g, j)) : LaneDesc{0, 0, 0};
    int c[U];
    T xv[U];
    auto columns = [&](int base) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = base + lane + 32 * u;
        c[u] = k < m ? (int)ld_stream(reinterpret_cast<const uint32_t*>(g.col) + xs + k, pol_stream) : -1;
      }
    };
    auto gathers = [&]() {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        xv[u] = T(0);
        if (c[u] >= 0) xv[u] = ld_x(x + c[u], pol_x);
      }
    };
    columns(0);
    // the rows' scaled values; the row open at the tile's end may be past the last row
    for (int r = lane; r <= n_t; r += 32) sg[r] = y_ws + r < g.n_rows ? scale * gv[y_ws + r] : T(0);
    gathers();
    __syncwarp();
    T* const sk = sg + n_t + 1;                 // a value per nonzero
    if (!(tys & kMsb)) {
      const int left = g.steps - j * g.sigma;   // steps of this lane (none past the last lane)
      const int len = j < g.lane_num ? (left < g.sigma ? left : g.sigma) : 0;
      int xk = d.xo, r = d.yo;
      for (int k = 0; k < len; ++k) {
        if ((d.flags >> k) & 1u) ++r;
        else sk[xk++] = sg[r];
      }
    }
    __syncwarp();
    const T one_row = sg[0];
    for (int base = 0; base < m; base += 32 * U) {
      if (base > 0) {                           // sigma > 14: more nonzeros than one batch
        columns(base);
        gathers();
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = base + lane + 32 * u;
        if (k < m) __stcs(out + xs + k, (tys & kMsb ? one_row : sk[k]) * xv[u]);
      }
    }
    __syncwarp();                               // the next tile writes the shared values anew
  }
}

// The same with a thread per lane of the schedule, for sigma below kSddmmTileSigma: a tile is then too
// little for a warp (sigma 1: 32 steps), and a lane's nonzeros hardly spread.  R-MAT scale 20, this
// and a warp per tile: f32, sigma 1 105 us (227), 2 70 (107), 3 69 (80), 4 76 (69); f64, sigma 1 115
// (237), 2 87 (123), 3 94 (92).
template <typename T>
constexpr int kSddmmTileSigma = sizeof(T) == 8 ? 3 : 4;

template <typename T>
__global__ void __launch_bounds__(256)
    sddmm_lanes_kernel(const Geometry g, const T* __restrict__ gv, const T* __restrict__ x, T scale,
                       T* __restrict__ out) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < g.lane_num; j += stride) {
    const int ti = (int)(j / kOmega);
    const LaneDesc d = decode_lane(g, load_desc(g, j));
    int xk = (int)__ldg(g.tile_x + ti) + d.xo;
    int row = (int)(__ldg(g.tile_y + ti) & ~kMsb) + d.yo;
    const int64_t left = (int64_t)g.steps - j * g.sigma;
    const int len = left < g.sigma ? (int)left : g.sigma;
    T gr = row < g.n_rows ? scale * gv[row] : T(0);
    for (int k = 0; k < len; ++k) {
      if ((d.flags >> k) & 1u) {
        ++row;
        gr = row < g.n_rows ? scale * gv[row] : T(0);
      } else {
        out[xk] = gr * x[__ldg(g.col + xk)];
        ++xk;
      }
    }
  }
}

template <typename T>
cudaError_t sddmm_typed(const merbit_plan_s* p, const T* g, const T* x, T scale, T* out, cudaStream_t st) {
  if (p->sigma < kSddmmTileSigma<T>) {
    const int grid = (int)std::min<int64_t>((p->lane_num + 255) / 256, (int64_t)p->num_sms * 16);
    sddmm_lanes_kernel<T><<<grid, 256, 0, st>>>(p->geom(), g, x, scale, out);
    return cudaGetLastError();
  }
  const size_t smem = kSddmmWarps * ((size_t)kOmega * p->sigma + 2) * sizeof(T);
  const size_t most = kSddmmWarps * ((size_t)kOmega * kSigmaMax64 + 2) * sizeof(T);
  int grid = persistent_grid(reinterpret_cast<const void*>(sddmm_kernel<T>), kSddmmWarps * 32, smem, most, p->num_sms);
  if (grid <= 0) return cudaErrorInvalidConfiguration;
  grid = (int)std::min<int64_t>(grid, (p->tile_num + kSddmmWarps - 1) / kSddmmWarps);
  sddmm_kernel<T><<<grid, kSddmmWarps * 32, smem, st>>>(p->geom(), g, x, scale, out);
  return cudaGetLastError();
}

template <typename T, bool ABS>
__global__ void vec_sum_kernel(const T* __restrict__ x, int64_t n, double* out) {
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    s += ABS ? fabs(static_cast<double>(x[i])) : static_cast<double>(x[i]);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, s);
}

}  // namespace

cudaError_t spmv_adj_f32(const merbit_plan_s* p, const float* vals, const float* x,
                         const AdjParams& prm, cudaStream_t st) {
  EpiAdjoint<float> epi{};
  epi.p = prm;
  epi.xold = x;
  return launch_spmv<float, float, float>(p, vals, x, epi, st);
}

cudaError_t spmv_adj_f64(const merbit_plan_s* p, const double* vals, const double* x,
                         const AdjParams& prm, cudaStream_t st) {
  EpiAdjoint<double> epi{};
  epi.p = prm;
  epi.xold = x;
  return launch_spmv<double, double, double>(p, vals, x, epi, st);
}

cudaError_t sddmm(const merbit_plan_s* p, merbit_dtype dt, const void* g, const void* x,
                  double scale, void* out, cudaStream_t st) {
  if (p->lane_num == 0) return cudaSuccess;
  if (dt == MERBIT_F64)
    return sddmm_typed<double>(p, static_cast<const double*>(g), static_cast<const double*>(x), scale,
                               static_cast<double*>(out), st);
  return sddmm_typed<float>(p, static_cast<const float*>(g), static_cast<const float*>(x), static_cast<float>(scale),
                            static_cast<float*>(out), st);
}

cudaError_t vec_sum(const void* x, merbit_dtype dt, int64_t n, double* out, bool absolute,
                    int num_sms, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), st);
  if (e != cudaSuccess || n == 0) return e;
  const int grid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 8);
  const double* xd = static_cast<const double*>(x);
  const float* xf = static_cast<const float*>(x);
  if (dt == MERBIT_F64 && absolute) vec_sum_kernel<double, true><<<grid, 256, 0, st>>>(xd, n, out);
  else if (dt == MERBIT_F64) vec_sum_kernel<double, false><<<grid, 256, 0, st>>>(xd, n, out);
  else if (absolute) vec_sum_kernel<float, true><<<grid, 256, 0, st>>>(xf, n, out);
  else vec_sum_kernel<float, false><<<grid, 256, 0, st>>>(xf, n, out);
  return cudaGetLastError();
}

}  // namespace merbit

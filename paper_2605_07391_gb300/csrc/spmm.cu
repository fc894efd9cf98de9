// Host side of the batched product Y = scale * A X (row-major X and Y, f32): column
// chunks of 32, 16, 8 or 4 through merbit_spmm_kernel.
//
// Slices of 4 columns (16 bytes) need rows of X on 16-byte boundaries, a whole number of slices
// wide.  Other X (an odd k, say) are copied into padded rows first, a chunk of columns at a time
// in a buffer the plan keeps, when the matrix has at least three nonzeros per row of X: the copy
// reads and writes a row once, while the product gathers it once per nonzero, and a one-column
// slice costs 2 to 4 times as much per nonzero (R-MAT, 1,000,003 rows, 11.6 M nonzeros, k = 13:
// 0.316 ms with one-column slices, 0.156 ms with the copy; k = 2: 0.097 and 0.079 ms).
#include "spmm_kernel.cuh"

namespace merbit {

namespace {

// P[r, 0..kp) = X[r, 0..kc) and zeros, kp = 4, 8, 16 or 32: a thread writes 16 bytes.
__global__ void __launch_bounds__(256) spmm_pack_kernel(const float* __restrict__ X, int64_t ldx, int64_t n, int kc,
                                                        int log_slices, float4* __restrict__ P) {
  const int64_t total = n << log_slices;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i >> log_slices;
    const int c = (int)(i & ((1 << log_slices) - 1)) * 4;
    const float* x = X + r * ldx + c;
    P[i] = make_float4(c < kc ? __ldg(x) : 0.f, c + 1 < kc ? __ldg(x + 1) : 0.f, c + 2 < kc ? __ldg(x + 2) : 0.f,
                       c + 3 < kc ? __ldg(x + 3) : 0.f);
  }
}

template <int VW, bool YVEC, bool SCALED>
cudaError_t spmm_chunk(const merbit_plan_s* p, const float* vals, const float* X, int64_t ldx, int kc,
                       const SpmmOut& out, double* acc, cudaStream_t st) {
  if (kc == 32) return launch_spmm<32, VW, YVEC, SCALED>(p, vals, X, ldx, out, acc, st);
  if (kc == 16) return launch_spmm<16, VW, YVEC, SCALED>(p, vals, X, ldx, out, acc, st);
  if (kc == 8) return launch_spmm<8, VW, YVEC, SCALED>(p, vals, X, ldx, out, acc, st);
  return launch_spmm<4, VW, YVEC, SCALED>(p, vals, X, ldx, out, acc, st);
}

// The plan's buffer of n_cols rows of kc floats (or of a wider chunk's), or null: too few nonzeros to
// pay for the copy, or no memory.  A wider buffer takes the place of the narrower ones, except of
// those that a captured launch keeps using.  In a capture the copy is as worthwhile as elsewhere
// (R-MAT, 1,000,003 rows, k = 13: 0.150 ms a replay, 0.320 with one-column slices).
float* pack_buffer(merbit_plan_s* p, int kc, cudaStream_t st) {
  if (p->nnz < 3 * p->n_cols) return nullptr;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  const bool recorded = cs != cudaStreamCaptureStatusNone;
  int width = 0;
  while ((4 << width) < kc) ++width;
  int w = width;
  while (w < 4 && !p->spmm_pack[w]) ++w;
  if (w == 4) {
    w = width;
    for (int i = 0; i < width && !recorded; ++i) {
      if (!p->spmm_pack[i] || ((p->spmm_pack_recorded >> i) & 1u)) continue;
      dev_free(p->device, {p->spmm_pack[i]});
      p->spmm_pack[i] = nullptr;
    }
    const RelaxedCalls relaxed;
    if (dev_alloc(&p->spmm_pack[w], sizeof(float) * (size_t)kc * (size_t)p->n_cols, st) != cudaSuccess) {
      cudaGetLastError();
      p->spmm_pack[w] = nullptr;
      return nullptr;
    }
  }
  if (recorded) p->spmm_pack_recorded |= 1u << w;
  return static_cast<float*>(p->spmm_pack[w]);
}

template <bool SCALED>
cudaError_t spmm_dispatch(merbit_plan_s* p, const float* vals, const float* X, int64_t k,
                          int64_t ldx, float* Y, int64_t ldy, float scale, bool gated, double* acc,
                          cudaStream_t st) {
  const bool xvec = k % 4 == 0 && ldx % 4 == 0 && ldx < ((int64_t)1 << 30) && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  const bool yvec = k % 4 == 0 && ldy % 4 == 0 && (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
  for (int64_t c0 = 0; c0 < k;) {
    const int64_t left = k - c0;
    const int kc = left >= 32 ? 32 : left > 8 ? 16 : left > 4 ? 8 : 4;
    const SpmmOut out{Y + c0, ldy, scale, (int)std::min<int64_t>(left, kc), gated};
    cudaError_t e = cudaSuccess;
    const float* xs = X + c0;
    int64_t ld = ldx;
    if (!xvec) {
      float* pack = pack_buffer(p, kc, st);
      if (pack) {
        const int64_t vecs = p->n_cols * (kc / 4);
        const int grid = (int)std::min<int64_t>((vecs + 255) / 256, (int64_t)p->num_sms * 16);
        const int log_slices = kc == 32 ? 3 : kc == 16 ? 2 : kc == 8 ? 1 : 0;
        spmm_pack_kernel<<<grid, 256, 0, st>>>(xs, ldx, p->n_cols, out.kc, log_slices, reinterpret_cast<float4*>(pack));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
      }
      xs = pack ? pack : xs;
      ld = pack ? kc : ldx;
      e = !pack ? spmm_chunk<1, false, SCALED>(p, vals, xs, ld, kc, out, acc, st)
          : yvec ? spmm_chunk<4, true, SCALED>(p, vals, xs, ld, kc, out, acc, st)
                 : spmm_chunk<4, false, SCALED>(p, vals, xs, ld, kc, out, acc, st);
    } else {
      e = yvec ? spmm_chunk<4, true, SCALED>(p, vals, xs, ld, kc, out, acc, st)
               : spmm_chunk<4, false, SCALED>(p, vals, xs, ld, kc, out, acc, st);
    }
    if (e != cudaSuccess) return e;
    c0 += out.kc;
  }
  return cudaSuccess;
}

}  // namespace

int64_t spmm_acc_sets(const merbit_plan_s* p) { return spmm_sets(p); }

cudaError_t spmm_plain_f32(merbit_plan_s* p, const float* vals, const float* X, int64_t k,
                           int64_t ldx, float* Y, int64_t ldy, double* acc, cudaStream_t st) {
  return spmm_dispatch<false>(p, vals, X, k, ldx, Y, ldy, 1.f, false, acc, st);
}

cudaError_t spmm_scaled_f32(merbit_plan_s* p, const float* vals, const float* X, int64_t k,
                            int64_t ldx, float* Y, int64_t ldy, float scale, double* acc,
                            cudaStream_t st) {
  return spmm_dispatch<true>(p, vals, X, k, ldx, Y, ldy, scale, true, acc, st);
}

}  // namespace merbit

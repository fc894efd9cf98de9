// Transpose of a CSR pattern on the GPU, for the backward product A^T g.
//
// A stable least-significant-digit radix sort orders the nonzeros of A by column; stability keeps
// each column's nonzeros in row order, so the result is the row-sorted CSR of A^T and does not
// depend on thread timing.  Digits have up to 11 bits, as few passes as the column indices need
// and the bits spread evenly over them.  Per pass: a digit histogram per tile of 6,144 nonzeros, a
// scan over the tiles for every digit (and one over the digits), and a scatter that ranks equal
// digits inside a warp by ballots and across the warps of a tile through shared counters, brings
// the tile into digit order in shared memory and writes it out in runs.  The first pass also
// finds each nonzero's row, which travels with its position: the sorted columns give A^T's row
// pointer, the rows its column indices, and the positions are the permutation that carries values
// over.
//
// The cost is passes, the instructions of the ranks (ten ballots a nonzero and pass) and how whole
// the scattered sectors are: two passes of 10 bits instead of three of 8 at 2^20 columns, runs of
// six nonzeros on average instead of one element per thread store, and rows carried along instead
// of expanded and gathered at the end.  R-MAT scale 20 (16.1 M nonzeros): 0.86 ms of kernels
// before, 0.46 ms.  Ranks by match instructions took 0.21 ms a pass, by ballots 0.17; 16 or 8
// nonzeros per thread 5 % more.
#include <algorithm>
#include <cstdio>

#include "extensions.cuh"

namespace merbit {
void set_last_error(const char* msg);
}  // namespace merbit

using namespace merbit;

namespace {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 12;                       // nonzeros per thread
constexpr int kTile = kSortThreads * kSortItems;     // nonzeros per CTA
constexpr int kDigitBits = 11;                       // largest digit
constexpr int kScanThreads = 256;
// Rows that start inside a tile are walked by its CTA, 512 at a time, up to this many; beyond that
// (runs of empty rows) each nonzero searches its row: 15 ms for 2^24 empty rows in one tile, walked;
// the search takes some 25 steps.
constexpr int kRowsWalked = 2 * kTile;

// Exclusive scan of one value per thread over the CTA (whole warps); *total gets the sum.
__device__ __forceinline__ uint32_t cta_exclusive_scan(uint32_t v, uint32_t* warp_tot, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < warps ? warp_tot[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < warps) warp_tot[lane] = wi - w;
    if (lane == 31) warp_tot[32] = wi;
  }
  __syncthreads();
  const uint32_t r = warp_tot[warp] + inc - v;
  *total = warp_tot[32];
  __syncthreads();
  return r;
}

// hist[d][tile] = nonzeros of the tile with digit d.  Two copies of the counters (even and odd
// warps) halve the contention on frequent digits.  When row_ptr is given (the first pass),
// tile_row[tile] = the row of the tile's first nonzero.
__global__ void __launch_bounds__(kSortThreads)
    radix_hist_kernel(const int32_t* __restrict__ keys, int64_t n, int shift, int bits, int num_tiles,
                      uint32_t* __restrict__ hist, const int32_t* __restrict__ row_ptr, int64_t n_rows,
                      int32_t* __restrict__ tile_row) {
  extern __shared__ uint32_t cnt[];                  // [2][bins]
  const int bins = 1 << bits;
  const uint32_t mask = (uint32_t)bins - 1u;
  for (int i = threadIdx.x; i < 2 * bins; i += kSortThreads) cnt[i] = 0;
  const int64_t base = (int64_t)blockIdx.x * kTile;
  int32_t key[kSortItems];
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const int64_t e = base + threadIdx.x + i * kSortThreads;
    key[i] = e < n ? __ldg(keys + e) : -1;
  }
  __syncthreads();
  uint32_t* const mine = cnt + ((threadIdx.x >> 5) & 1) * bins;
#pragma unroll
  for (int i = 0; i < kSortItems; ++i)
    if (key[i] >= 0) atomicAdd(&mine[((uint32_t)key[i] >> shift) & mask], 1u);
  if (row_ptr && threadIdx.x < 32) {
    // the last row that starts at or before nonzero `base`: a search 32 ways a round (row 0 starts
    // at nonzero 0)
    int64_t lo = 0, hi = n_rows - 1;
    while (lo < hi) {
      const int64_t step = (hi - lo + 31) / 32;
      const int64_t probe = lo + (int64_t)(threadIdx.x + 1) * step;
      const bool le = probe <= hi && (int64_t)__ldg(row_ptr + probe) <= base;
      lo += (int64_t)__popc(__ballot_sync(0xffffffffu, le)) * step;
      hi = lo + step - 1 < hi ? lo + step - 1 : hi;
    }
    if (threadIdx.x == 0) tile_row[blockIdx.x] = (int32_t)lo;
  }
  __syncthreads();
  for (int d = threadIdx.x; d < bins; d += kSortThreads)
    hist[(size_t)d * num_tiles + blockIdx.x] = cnt[d] + cnt[bins + d];
}

// One CTA per digit: exclusive scan of the digit's counts over the tiles, in place, and its total.
__global__ void __launch_bounds__(kScanThreads)
    radix_scan_kernel(uint32_t* __restrict__ hist, int num_tiles, uint32_t* __restrict__ totals) {
  __shared__ uint32_t warp_tot[33];
  uint32_t* const h = hist + (size_t)blockIdx.x * num_tiles;
  uint32_t carry = 0;
  for (int c0 = 0; c0 < num_tiles; c0 += kScanThreads) {
    const int i = c0 + threadIdx.x;
    uint32_t total;
    const uint32_t off = cta_exclusive_scan(i < num_tiles ? h[i] : 0u, warp_tot, &total);
    if (i < num_tiles) h[i] = carry + off;
    carry += total;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// One CTA: exclusive scan of the digits' totals in place (at most 2,048).
__global__ void __launch_bounds__(1024) radix_base_kernel(uint32_t* __restrict__ totals, int bins) {
  __shared__ uint32_t warp_tot[33];
  const int i = 2 * threadIdx.x;
  const uint32_t a = i < bins ? totals[i] : 0u, b = i + 1 < bins ? totals[i + 1] : 0u;
  uint32_t total;
  const uint32_t off = cta_exclusive_scan(a + b, warp_tot, &total);
  if (i < bins) totals[i] = off;
  if (i + 1 < bins) totals[i + 1] = off + a;
}

// Shared memory of the scatter: the tile in digit order (8 bytes a nonzero), the digits' local
// starts and global offsets, and per-warp counters.
__host__ __device__ constexpr size_t scatter_smem(int bits) {
  return sizeof(uint2) * kTile + (2 * sizeof(uint32_t) + (size_t)kSortWarps * sizeof(uint16_t)) * ((size_t)1 << bits);
}

// One pass's scatter.  BITS: at least the digit's bits.  FIRST: positions are the nonzeros' own
// indices and rows come from the row pointer; otherwise (position, row) pairs are read.  LAST:
// positions and rows are written to the results instead of pairs.
template <int BITS, bool FIRST, bool LAST>
__global__ void __launch_bounds__(kSortThreads, 2)
    radix_scatter_kernel(const int32_t* __restrict__ keys_in, const uint2* __restrict__ pair_in,
                         int32_t* __restrict__ keys_out, uint2* __restrict__ pair_out, int32_t* __restrict__ pos_out,
                         int32_t* __restrict__ row_out, int64_t n, int shift, int bits, int num_tiles,
                         const uint32_t* __restrict__ offs, const uint32_t* __restrict__ base,
                         const int32_t* __restrict__ row_ptr, int64_t n_rows, const int32_t* __restrict__ tile_row) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ uint32_t warp_tot[33];
  constexpr int H = kSortItems / 2;                  // pairs in flight per thread
  const int bins = 1 << bits;
  const uint32_t mask = (uint32_t)bins - 1u;
  uint2* const stage2 = reinterpret_cast<uint2*>(sm_raw);              // [kTile]
  uint32_t* const stage = reinterpret_cast<uint32_t*>(sm_raw);         // [kTile], at another time
  uint32_t* const start = reinterpret_cast<uint32_t*>(stage2 + kTile); // [bins]
  uint32_t* const goff = start + bins;                                 // [bins]: global place of local place 0
  uint32_t* const wz = goff + bins;                                    // [warps][bins / 2]: two digits a word
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t t0 = (int64_t)blockIdx.x * kTile;
  const int count = (int)(n - t0 < kTile ? n - t0 : kTile);
  const int w0 = warp * (32 * kSortItems) + lane;    // item it of this thread is nonzero w0 + 32 it
  int32_t key[kSortItems];
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) key[it] = w0 + it * 32 < count ? __ldcs(keys_in + t0 + w0 + it * 32) : -1;
  for (int i = tid; i < kSortWarps * bins / 2; i += kSortThreads) wz[i] = 0u;
  uint32_t row[FIRST ? kSortItems : 1];
  if constexpr (FIRST) {
    const int r0 = __ldg(tile_row + blockIdx.x);
    const int r1 = (int)blockIdx.x + 1 < num_tiles ? __ldg(tile_row + blockIdx.x + 1) : (int)n_rows - 1;
    if (r1 - r0 > kRowsWalked) {
      // a long run of empty rows: a search for every nonzero, a step of all of a thread's at a time
#pragma unroll
      for (int it = 0; it < kSortItems; ++it) row[it] = (uint32_t)r0;
      for (uint32_t s = 1u << (31 - __clz(r1 - r0)); s > 0u; s >>= 1) {
#pragma unroll
        for (int it = 0; it < kSortItems; ++it) {
          const uint32_t r = row[it] + s;              // rows stay below 2^31, steps below 2^31
          if (r <= (uint32_t)r1 && (int64_t)__ldg(row_ptr + r) <= t0 + w0 + it * 32) row[it] = r;
        }
      }
    } else {
      // rows of the tile's nonzeros: every row that starts inside the tile marks its first nonzero
      // (the last of several rows that start there wins: the others are empty), then a running maximum
      for (int i = tid; i < kTile; i += kSortThreads) stage[i] = 0u;
      __syncthreads();
      for (int64_t r = (int64_t)r0 + 1 + tid; r < n_rows; r += kSortThreads) {
        const int64_t p = (int64_t)__ldg(row_ptr + r) - t0;
        if (p >= count) break;
        atomicMax(&stage[p], (uint32_t)(r - r0));
      }
      __syncthreads();
      // a warp takes its own 384 nonzeros, 32 at a time, after the maxima of the warps before
      uint32_t m = 0;
#pragma unroll
      for (int it = 0; it < kSortItems; ++it) {
        row[it] = stage[w0 + it * 32];
        m = max(m, row[it]);
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) warp_tot[warp] = m;
      __syncthreads();
      uint32_t run = 0;
      for (int w = 0; w < warp; ++w) run = max(run, warp_tot[w]);
#pragma unroll
      for (int it = 0; it < kSortItems; ++it) {
        uint32_t inc = row[it];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc = max(inc, y);
        }
        inc = max(inc, run);
        run = __shfl_sync(0xffffffffu, inc, 31);
        row[it] = inc + (uint32_t)r0;
      }
    }
  }
  __syncthreads();
  // ranks inside the warp, in the order of the nonzeros; two a register
  uint16_t* const mine = reinterpret_cast<uint16_t*>(wz) + warp * bins;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t packed[H];
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    const bool ok = key[it] >= 0;
    const uint32_t d = ((uint32_t)key[it] >> shift) & mask;
    uint32_t peers = __ballot_sync(0xffffffffu, ok);   // lanes with the same digit
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
      const uint32_t one = (uint32_t)((int32_t)(d << (31 - b)) >> 31);   // all ones if bit b is set
      peers &= ~(__ballot_sync(0xffffffffu, one != 0u) ^ one);
    }
    const uint32_t before = ok ? mine[d] : 0u;
    const uint32_t rank = before + __popc(peers & lt);
    packed[it / 2] = it & 1 ? packed[it / 2] | (rank << 16) : rank;
    __syncwarp();
    if (ok && (peers & lt) == 0u) mine[d] = (uint16_t)(before + __popc(peers));
    __syncwarp();
  }
  uint2 pr[H];
  auto load_pairs = [&](int h) {
#pragma unroll
    for (int q = 0; q < H; ++q) {
      const int it = h * H + q;
      if constexpr (FIRST) pr[q] = make_uint2((uint32_t)(t0 + w0 + it * 32), row[it]);
      else pr[q] = w0 + it * 32 < count ? __ldcs(pair_in + t0 + w0 + it * 32) : make_uint2(0u, 0u);
    }
  };
  if constexpr (!FIRST) load_pairs(0);
  __syncthreads();
  // per digit: offsets of the warps in order, the digit's local start and its global offset (two
  // digits a word: the halves stay below 2^13, so no carry passes between them)
  {
    uint32_t pair[2], sum = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int w2 = 2 * tid + q;                     // digits 4 tid + 2 q and the next
      uint32_t run = 0;
      if (2 * w2 < bins)
#pragma unroll 4
        for (int w = 0; w < kSortWarps; ++w) {
          const uint32_t c = wz[w * (bins >> 1) + w2];
          wz[w * (bins >> 1) + w2] = run;
          run += c;
        }
      pair[q] = run;
      sum += (run & 0xffffu) + (run >> 16);
    }
    uint32_t total;
    uint32_t off = cta_exclusive_scan(sum, warp_tot, &total);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int d = 4 * tid + q;
      if (d < bins) {
        start[d] = off;
        goff[d] = __ldg(base + d) + __ldg(offs + (size_t)d * num_tiles + blockIdx.x) - off;
      }
      off += q & 1 ? pair[q / 2] >> 16 : pair[q / 2] & 0xffffu;
    }
  }
  __syncthreads();
  // places in the tile's digit order
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    uint32_t place = 0;
    if (key[it] >= 0) {
      const uint32_t d = ((uint32_t)key[it] >> shift) & mask;
      place = (it & 1 ? packed[it / 2] >> 16 : packed[it / 2] & 0xffffu) + start[d] + mine[d];
      stage[place] = (uint32_t)key[it];
    }
    packed[it / 2] = it & 1 ? (packed[it / 2] & 0xffffu) | (place << 16) : (packed[it / 2] & 0xffff0000u) | place;
  }
  __syncthreads();
  uint32_t dst[kSortItems];                           // of local places tid + 512 it
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    const int i = tid + it * kSortThreads;
    dst[it] = 0u;
    if (i < count) {
      const uint32_t k = stage[i];
      dst[it] = goff[(k >> shift) & mask] + (uint32_t)i;
      keys_out[dst[it]] = (int32_t)k;
    }
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (FIRST || h > 0) load_pairs(h);
#pragma unroll
    for (int q = 0; q < H; ++q) {
      const int it = h * H + q;
      if (w0 + it * 32 < count) stage2[it & 1 ? packed[it / 2] >> 16 : packed[it / 2] & 0xffffu] = pr[q];
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    const int i = tid + it * kSortThreads;
    if (i < count) {
      const uint2 v = stage2[i];
      if constexpr (LAST) {
        pos_out[dst[it]] = (int32_t)v.x;
        row_out[dst[it]] = (int32_t)v.y;
      } else {
        pair_out[dst[it]] = v;
      }
    }
  }
}

template <int BITS>
cudaError_t launch_scatter(bool first, bool last, unsigned tiles, size_t smem, cudaStream_t st, const int32_t* keys_in,
                           const uint2* pair_in, int32_t* keys_out, uint2* pair_out, int32_t* pos_out, int32_t* row_out,
                           int64_t n, int shift, int bits, const uint32_t* offs, const uint32_t* base,
                           const int32_t* row_ptr, int64_t n_rows, const int32_t* tile_row) {
  auto kern = first ? (last ? radix_scatter_kernel<BITS, true, true> : radix_scatter_kernel<BITS, true, false>)
                    : (last ? radix_scatter_kernel<BITS, false, true> : radix_scatter_kernel<BITS, false, false>);
  if (persistent_grid(reinterpret_cast<const void*>(kern), kSortThreads, smem, scatter_smem(BITS), 1) <= 0)
    return cudaErrorInvalidConfiguration;
  kern<<<tiles, kSortThreads, smem, st>>>(keys_in, pair_in, keys_out, pair_out, pos_out, row_out, n, shift, bits,
                                          (int)tiles, offs, base, row_ptr, n_rows, tile_row);
  return cudaGetLastError();
}

// row_ptr_t[c] = first position of column c in the sorted column list, c in [0, n_cols].
__global__ void boundaries_kernel(const int32_t* __restrict__ sorted, int64_t nnz, int64_t n_cols,
                                  int32_t* __restrict__ row_ptr_t) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p <= nnz;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cur = p < nnz ? sorted[p] : n_cols;
    const int64_t prev = p > 0 ? sorted[p - 1] : -1;
    for (int64_t c = prev + 1; c <= cur; ++c) row_ptr_t[c] = (int32_t)p;
  }
}

template <typename T>
__global__ void gather_kernel(const T* __restrict__ src, const int32_t* __restrict__ idx,
                              T* __restrict__ dst, int64_t count) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = src[idx[i]];
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

int grid_of(int64_t work, int threads) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((work + threads - 1) / threads,
                                                     (int64_t)sm_count() * 16));
}

cudaError_t build_transpose(merbit_transpose_s* t, const int32_t* row_ptr, const int32_t* col,
                            cudaStream_t st) {
  const int64_t nnz = t->nnz;
  if (nnz == 0) {
    cudaError_t e = cudaMemsetAsync(t->row_ptr_t, 0, sizeof(int32_t) * (size_t)(t->n_cols + 1), st);
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
  }
  int bits = 1;
  while (bits < 31 && ((int64_t)1 << bits) < t->n_cols) ++bits;
  const int passes = (bits + kDigitBits - 1) / kDigitBits;
  const int digit = (bits + passes - 1) / passes;      // bits of a pass's digit
  const int bins = 1 << digit;
  const int64_t num_tiles = (nnz + kTile - 1) / kTile;
  // keys and (position, row) pairs between passes, the last pass's keys, the histograms, the
  // digits' totals and the tiles' rows, in one allocation
  const auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t nb = up(sizeof(int32_t) * (size_t)nnz), pb = up(sizeof(uint2) * (size_t)nnz);
  const size_t hb = up(sizeof(uint32_t) * (size_t)bins * (size_t)num_tiles);
  const size_t tb = up(sizeof(uint32_t) * (size_t)bins);
  const int sets = passes > 2 ? 2 : passes - 1;
  void* mem = nullptr;
  cudaError_t e = dev_alloc(&mem, (size_t)sets * (nb + pb) + nb + hb + tb + up(sizeof(int32_t) * (size_t)num_tiles), st);
  if (e != cudaSuccess) return e;
  char* m = static_cast<char*>(mem);
  const auto take = [&](size_t b) {
    char* r = m;
    m += b;
    return r;
  };
  int32_t* keys[2] = {nullptr, nullptr};
  uint2* pairs[2] = {nullptr, nullptr};
  for (int s = 0; s < sets; ++s) {
    keys[s] = reinterpret_cast<int32_t*>(take(nb));
    pairs[s] = reinterpret_cast<uint2*>(take(pb));
  }
  int32_t* const last_keys = reinterpret_cast<int32_t*>(take(nb));
  uint32_t* const hist = reinterpret_cast<uint32_t*>(take(hb));
  uint32_t* const totals = reinterpret_cast<uint32_t*>(take(tb));
  int32_t* const tile_row = reinterpret_cast<int32_t*>(m);
  const size_t smem = scatter_smem(digit);
  const int32_t* kin = col;
  const uint2* pin = nullptr;
  const unsigned tiles = (unsigned)num_tiles;
  for (int pass = 0; pass < passes && e == cudaSuccess; ++pass) {
    const bool first = pass == 0, last = pass == passes - 1;
    const int shift = digit * pass;
    int32_t* const kout = last ? last_keys : keys[pass & 1];
    uint2* const pout = last ? nullptr : pairs[pass & 1];
    radix_hist_kernel<<<tiles, kSortThreads, 2 * sizeof(uint32_t) * (size_t)bins, st>>>(
        kin, nnz, shift, digit, (int)num_tiles, hist, first ? row_ptr : nullptr, t->n_rows, tile_row);
    radix_scan_kernel<<<bins, kScanThreads, 0, st>>>(hist, (int)num_tiles, totals);
    radix_base_kernel<<<1, 1024, 0, st>>>(totals, bins);
    auto go = digit <= 8 ? launch_scatter<8> : digit == 9 ? launch_scatter<9> : digit == 10 ? launch_scatter<10>
                                                                              : launch_scatter<11>;
    e = go(first, last, tiles, smem, st, kin, pin, kout, pout, t->perm, t->col_t, nnz, shift, digit, hist, totals, row_ptr,
           t->n_rows, tile_row);
    kin = kout;
    pin = pout;
  }
  if (e == cudaSuccess) {
    boundaries_kernel<<<grid_of(nnz + 1, 256), 256, 0, st>>>(kin, nnz, t->n_cols, t->row_ptr_t);
    e = cudaGetLastError();
  }
  const cudaError_t es = cudaStreamSynchronize(st);
  cudaFree(mem);
  return e == cudaSuccess ? es : e;
}

void free_transpose(merbit_transpose_s* t) {
  if (!t) return;
  dev_free(t->device, {t->row_ptr_t});    // the three arrays' block
  delete t;
}

merbit_status tfail(merbit_status s, const char* msg) {
  set_last_error(msg);
  return s;
}

}  // namespace

namespace merbit {

cudaError_t gather(const void* src, const int32_t* idx, void* dst, int64_t count, size_t elem,
                   cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  if (elem == 8)
    gather_kernel<double><<<grid_of(count, 256), 256, 0, st>>>(
        static_cast<const double*>(src), idx, static_cast<double*>(dst), count);
  else
    gather_kernel<float><<<grid_of(count, 256), 256, 0, st>>>(
        static_cast<const float*>(src), idx, static_cast<float*>(dst), count);
  return cudaGetLastError();
}

}  // namespace merbit

extern "C" {

merbit_status merbit_transpose(const int32_t* row_ptr, const int32_t* col_idx, int64_t n_rows,
                               int64_t n_cols, int64_t nnz, void* stream, merbit_transpose_t* out) {
  set_last_error("");
  if (!out) return tfail(MERBIT_EINVAL, "out is NULL");
  *out = nullptr;
  if (n_rows < 0 || n_cols < 0 || nnz < 0) return tfail(MERBIT_EINVAL, "negative size");
  if (!row_ptr || (nnz > 0 && !col_idx)) return tfail(MERBIT_EINVAL, "row_ptr or col_idx is NULL");
  if (n_rows >= INT32_MAX || n_cols >= INT32_MAX || nnz >= INT32_MAX)
    return tfail(MERBIT_EOVERFLOW, "sizes must fit int32");
  auto* t = new merbit_transpose_s();
  t->n_rows = n_rows;
  t->n_cols = n_cols;
  t->nnz = nnz;
  cudaGetDevice(&t->device);
  const size_t pb = (sizeof(int32_t) * (size_t)(n_cols + 1) + 255) & ~size_t(255);
  const size_t nb = (sizeof(int32_t) * (size_t)std::max<int64_t>(nnz, 1) + 255) & ~size_t(255);
  void* mem = nullptr;
  cudaError_t e = dev_alloc(&mem, pb + 2 * nb, static_cast<cudaStream_t>(stream));
  if (e == cudaSuccess) {
    t->row_ptr_t = static_cast<int32_t*>(mem);
    t->col_t = reinterpret_cast<int32_t*>(static_cast<char*>(mem) + pb);
    t->perm = reinterpret_cast<int32_t*>(static_cast<char*>(mem) + pb + nb);
  }
  if (e == cudaSuccess) e = build_transpose(t, row_ptr, col_idx, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    free_transpose(t);
    char msg[256];
    std::snprintf(msg, sizeof(msg), "merbit_transpose: %s", cudaGetErrorString(e));
    return tfail(e == cudaErrorMemoryAllocation ? MERBIT_ENOMEM : MERBIT_ECUDA, msg);
  }
  *out = t;
  return MERBIT_OK;
}

merbit_status merbit_transpose_get(merbit_transpose_t t, const int32_t** row_ptr_t,
                                   const int32_t** col_t, const int32_t** perm) {
  set_last_error("");
  if (!t) return tfail(MERBIT_EINVAL, "transpose is NULL");
  if (row_ptr_t) *row_ptr_t = t->row_ptr_t;
  if (col_t) *col_t = t->col_t;
  if (perm) *perm = t->perm;
  return MERBIT_OK;
}

void merbit_transpose_destroy(merbit_transpose_t t) { free_transpose(t); }

merbit_status merbit_gather(merbit_dtype dtype, const void* src, const int32_t* idx, void* dst,
                            int64_t count, void* stream) {
  set_last_error("");
  if (count < 0) return tfail(MERBIT_EINVAL, "negative count");
  if (count > 0 && (!src || !idx || !dst)) return tfail(MERBIT_EINVAL, "NULL pointer");
  if (dtype != MERBIT_F32 && dtype != MERBIT_F64) return tfail(MERBIT_EINVAL, "dtype must be F32 or F64");
  cudaError_t e = gather(src, idx, dst, count, dtype == MERBIT_F64 ? 8 : 4,
                         static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return tfail(MERBIT_ECUDA, cudaGetErrorString(e));
  return MERBIT_OK;
}

}  // extern "C"

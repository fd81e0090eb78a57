// Few query rows against the resident panel, on the integer pipe.
//
// One to kFewRows rows leave the tensor-core kernel with almost nothing but the
// panel's operand planes to read, 2 bytes per genotype.  The pair counts need
// only the two code bits: of a panel sample's words (L, H) of 32 markers and
// a row's V (present), hom (homozygous) and H,
//   N    = popc(V_p & V),
//   IBS0 = popc((H_p ^ H) & hom_p & hom)     (both homozygous, not the same),
//   IBS1 = popc((hom_p ^ hom) & V_p & V),
// four logic operations and three population counts per pair and 32 markers
// (codes 0 hom A1, 1 missing, 2 het, 3 hom A2: V = H | ~L, hom = ~(H ^ L)).  The
// panel's words, [32-marker column][sample], are a second copy of the panel made
// at load (an eighth of the operand planes' size).
//
// Thread = two panel samples (one load of 8 bytes each per column, coalesced over
// the warp), kQ rows at a time from shared memory; the marker axis is split over
// blockIdx.y, each split's counts go to parts of their own, and a second kernel
// adds them.  One row is bound by HBM (0.25 B per genotype), 8 rows by
// population counts (16 per clock and SM).  Measured, one row
// against 20,000 samples x 100,000 markers: 84 us, 6.0 TB/s, and 7 us for the
// sums (the tensor-core kernel, which reads the operand planes: 990 us).
#include <algorithm>

#include "ibs_device.cuh"
#include "ibs_internal.h"

namespace ibs {

namespace {

constexpr int kFewThreads = 256;
constexpr int kFewSpan = 2 * kFewThreads;  // panel samples per CTA
constexpr int kFewCols = 64;               // columns of the rows' words staged at a time

// The rows' words from their requests' packed bytes: thread = column c of row r,
// {V, hom, H, 0}; rows past the last and markers past m count as missing.
template <int kQ>
__global__ void __launch_bounds__(256) few_words_kernel(const FewTables tab, int64_t n_rows, int64_t m, int64_t n_cols,
                                                        uint4* __restrict__ words) {
  const int64_t c = (int64_t)blockIdx.x * 256 + threadIdx.x, r = blockIdx.y;
  if (c >= n_cols) return;
  uint32_t H = 0, L = ~0u;
  if (r < n_rows) {
    const RowSrc src = tab.rows[r];
    const int64_t stride = src.n_half, left = m - c * 32;
    const uint8_t* p = reinterpret_cast<const uint8_t*>(src.planes) + c * 32 * stride + (src.row >> 2);
    const int sh = 2 * (int)(src.row & 3);
    uint32_t byte[32];
#pragma unroll
    for (int k = 0; k < 32; ++k, p += stride) byte[k] = k < left ? __ldg(p) : 0x55u;
    H = L = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const uint32_t code = (byte[k] >> sh) & 3u;
      H |= (code >> 1) << k;
      L |= (code & 1u) << k;
    }
  }
  words[((r / kQ) * n_cols + c) * kQ + r % kQ] = make_uint4(H | ~L, ~(H ^ L), H, 0);
}

struct FewArgs {
  const uint2* panel;  // [n_cols][n]{L, H}
  const uint4* rows;   // [row group][n_cols][kQ]
  int64_t n, n_cols, split_cols;
  int64_t s0, n0, s1, count;  // panel samples s0 .. s0 + n0 - 1, then from s1, `count` together
  int32_t* part;              // [split][row][3][count]
  int32_t n_rows;
};
__device__ __forceinline__ int64_t few_sample(const FewArgs& a, int64_t i) { return i < a.n0 ? a.s0 + i : a.s1 + (i - a.n0); }

template <int kQ>
__global__ void __launch_bounds__(kFewThreads) few_pairs_kernel(const FewArgs a) {
  __shared__ uint4 sq[kFewCols * kQ];
  const int64_t i0 = (int64_t)blockIdx.x * kFewSpan + threadIdx.x, i1 = i0 + kFewThreads;
  const uint2* p0 = a.panel + few_sample(a, min(i0, a.count - 1));
  const uint2* p1 = a.panel + few_sample(a, min(i1, a.count - 1));
  const uint4* rows = a.rows + (int64_t)blockIdx.z * a.n_cols * kQ;
  int acc[2][kQ][3] = {};
  const int64_t end = min(a.n_cols, (int64_t)(blockIdx.y + 1) * a.split_cols);
  for (int64_t c = (int64_t)blockIdx.y * a.split_cols; c < end; c += kFewCols) {
    const int cols = (int)min((int64_t)kFewCols, end - c);
    __syncthreads();
    for (int i = threadIdx.x; i < cols * kQ; i += kFewThreads) sq[i] = __ldg(rows + c * kQ + i);
    __syncthreads();
#pragma unroll 4
    for (int j = 0; j < cols; ++j) {
      const int64_t off = (c + j) * a.n;
      const uint2 w[2] = {__ldg(p0 + off), __ldg(p1 + off)};
#pragma unroll
      for (int q = 0; q < kQ; ++q) {
        const uint4 r = sq[j * kQ + q];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const uint32_t L = w[t].x, H = w[t].y, V = (H | ~L) & r.x, hom = ~(H ^ L);
          acc[t][q][0] += __popc((H ^ r.z) & hom & r.y);
          acc[t][q][1] += __popc((hom ^ r.y) & V);
          acc[t][q][2] += __popc(V);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const int64_t r = (int64_t)blockIdx.z * kQ + q;
    if (r >= a.n_rows) break;
    int32_t* out = a.part + ((int64_t)blockIdx.y * a.n_rows + r) * 3 * a.count;
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      if (i0 < a.count) out[v * a.count + i0] = acc[0][q][v];
      if (i1 < a.count) out[v * a.count + i1] = acc[1][q][v];
    }
  }
}

__global__ void __launch_bounds__(256) few_sum_kernel(const FewArgs a, int splits, const FewTables tab) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x, r = blockIdx.y;
  if (i >= a.count) return;
  int32_t sum[3] = {0, 0, 0};
#pragma unroll 4
  for (int s = 0; s < splits; ++s) {
    const int32_t* p = a.part + ((int64_t)s * a.n_rows + r) * 3 * a.count + i;
#pragma unroll
    for (int v = 0; v < 3; ++v) sum[v] += p[v * a.count];
  }
  reinterpret_cast<int4*>(tab.out[r])[few_sample(a, i)] = make_int4(sum[0], sum[1], sum[2] - sum[0] - sum[1], sum[2]);
}

template <int kQ>
cudaError_t few(const FewTables& tab, int64_t m, uint4* words, int splits, const FewArgs& a, cudaStream_t st) {
  const unsigned groups = (unsigned)((a.n_rows + kQ - 1) / kQ);
  few_words_kernel<kQ><<<dim3((unsigned)((a.n_cols + 255) / 256), groups * kQ), 256, 0, st>>>(tab, a.n_rows, m,
                                                                                             a.n_cols, words);
  if (cudaError_t e = cudaGetLastError()) return e;
  few_pairs_kernel<kQ><<<dim3((unsigned)((a.count + kFewSpan - 1) / kFewSpan), (unsigned)splits, groups), kFewThreads, 0,
                         st>>>(a);
  if (cudaError_t e = cudaGetLastError()) return e;
  few_sum_kernel<<<dim3((unsigned)((a.count + 255) / 256), (unsigned)a.n_rows), 256, 0, st>>>(a, splits, tab);
  return cudaGetLastError();
}

}  // namespace

size_t few_rows_bytes(int64_t n_cols) { return (size_t)kFewRows * n_cols * sizeof(uint4); }

cudaError_t launch_few_rows(const FewTables& tab, int64_t n_rows, const uint32_t* panel_words, int64_t n_panel, int64_t m,
                            const int64_t (&samples)[2][2], void* words, void* part, size_t part_bytes, int num_sms,
                            cudaStream_t st) {
  FewArgs a;
  a.panel = reinterpret_cast<const uint2*>(panel_words);
  a.rows = static_cast<const uint4*>(words);
  a.n = n_panel;
  a.n_cols = (m + 31) / 32;
  a.s0 = samples[0][0];
  a.n0 = samples[0][1] - samples[0][0];
  a.s1 = samples[1][0];
  a.count = a.n0 + samples[1][1] - samples[1][0];
  a.part = static_cast<int32_t*>(part);
  a.n_rows = (int32_t)n_rows;
  if (n_rows < 1 || n_rows > kFewRows || a.count < 1) return cudaErrorInvalidValue;
  // about four CTAs of the pair kernel per SM, as far as the parts have room
  const int64_t groups = (a.count + kFewSpan - 1) / kFewSpan * ((n_rows + 7) / 8);
  int64_t splits = std::max<int64_t>(1, (4 * (int64_t)num_sms + groups - 1) / groups);
  splits = std::min(splits, (int64_t)(part_bytes / ((size_t)n_rows * a.count * 12)));
  splits = std::min<int64_t>(splits, (a.n_cols + kFewCols - 1) / kFewCols);
  if (splits < 1) return cudaErrorInvalidValue;
  a.split_cols = (a.n_cols + splits - 1) / splits;
  splits = (a.n_cols + a.split_cols - 1) / a.split_cols;
  if (n_rows > 4) return few<8>(tab, m, static_cast<uint4*>(words), (int)splits, a, st);
  if (n_rows > 2) return few<4>(tab, m, static_cast<uint4*>(words), (int)splits, a, st);
  if (n_rows > 1) return few<2>(tab, m, static_cast<uint4*>(words), (int)splits, a, st);
  return few<1>(tab, m, static_cast<uint4*>(words), (int)splits, a, st);
}

}  // namespace ibs

// Complete-linkage clustering of the samples under the IBS distance matrix.
//
// The paper's identity-by-state section ("Identity-by-state matrices, complete
// linkage clustering") runs complete linkage on the IBS matrix and brings the
// clustering from O(n^3) down to O(n^2 log n).  The same merges come from the
// textbook greedy rule: merge the two active clusters at the smallest
// complete-linkage distance D(A, B) = max over members, maintained by
// D(A u B, C) = max(D(A, C), D(B, C)).  Ties: a cluster is represented by its
// smallest member, and among equal distances the smallest (representative A,
// representative B) pair merges first; NaN distances (no common non-missing
// marker) count as +infinity.
//
// Here every active row i keeps its minimum (D[i][j], j) over active j > i,
// compared lexicographically.  Each step is then O(n) parallel work:
//   1. the global minimum over the row minima, (value, row), lexicographic,
//      gives the pair (i, j) to merge;
//   2. the rows whose minimum may be gone are listed: it pointed at j, which
//      disappears, or at i, whose distance may grow (distances only grow, so
//      every other row's minimum stays);
//   3. row and column i become the elementwise max of rows i and j, the same
//      pass finds row i's new minimum, and the listed rows rescan their row,
//      the CTA's warps divided evenly among them (3.2 rows per merge on 4,096
//      unrelated samples).  A rescan needs nothing of the update: by symmetry
//      row r holds both D[r][i] and D[r][j], whose max it takes in column i's
//      place.  So a merge waits for memory once, for both together.
// The steps form one CTA of 1,024 threads (32 warps), launched again each time a
// quarter of the rows and columns has been merged away and dropped; phases are
// separated by block barriers, which also order the memory updates.  Up to
// kClSmemRows samples the row minima and flags sit in shared memory.  The
// working matrix is square and symmetric in HBM.  It holds order-preserving
// 64-bit keys of the distances (8 bytes per entry), so that comparisons and
// warp-wide minima run on the integer pipes: GB300's FP64 rate is 1/64 of
// its FP32 rate, and redux.sync takes three instructions where a shuffle tree
// over (double, index) pairs takes fifteen.
//
// What bounds it: latency.  The merges are a serial chain, each one round of
// loads (700 cycles from L2, more from HBM) and four block barriers.
// Measured, n = 4,096 unrelated samples: 24.2 ms, 5.9 us per merge; 31.4 ms over
// all columns to the end (see cl_next); 34.3 ms with the rescans after the
// update; 125.1 ms with one warp per rescanned row, a check of every flag before
// the next load of a row, FP64 shuffle trees and rescans after the update.
#include <cstdint>
#include <type_traits>

#include "ibs_device.cuh"
#include "ibs_internal.h"

namespace ibs {

namespace {

constexpr int kClThreads = 1024;

// Order-preserving key of a distance: a < b as doubles <=> key(a) < key(b).
// NaN counts as +infinity, -0 as 0; kNoKey is above every key.
constexpr uint64_t kNoKey = ~0ull;
constexpr uint32_t kNoIdx = ~0u;
__device__ __forceinline__ uint64_t cl_key(double d) {
  const uint64_t inf = 0x7ff0000000000000ull;
  uint64_t b = d != d ? inf : (uint64_t)__double_as_longlong(d);
  if ((b << 1) == 0) b = 0;  // -0
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double cl_value(uint64_t k) {
  return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

// An entry that one thread of the CTA may read while another replaces it: either
// the old or the new value is read.
__device__ __forceinline__ uint64_t ld_shared_entry(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.cta.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_shared_entry(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.cta.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Smallest (key, index), lexicographic, over the warp's lanes (in every lane).
__device__ __forceinline__ void warp_best(uint64_t& key, uint32_t& idx) {
  const uint32_t hi = (uint32_t)(key >> 32);
  const uint32_t mh = __reduce_min_sync(0xffffffffu, hi);
  const uint32_t lo = hi == mh ? (uint32_t)key : kNoIdx;
  const uint32_t ml = __reduce_min_sync(0xffffffffu, lo);
  idx = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? idx : kNoIdx);
  key = (uint64_t)mh << 32 | ml;
}

// Triangle (upper, with diagonal, as ibs_compute writes it) -> square keys.
// One 32 x 32 tile (I <= J) per CTA, its mirror image written through shared
// memory so that both halves are stored in whole rows.
__global__ void __launch_bounds__(256) cl_init_kernel(const double* __restrict__ tri, int64_t n,
                                                      uint64_t* __restrict__ D) {
  __shared__ uint64_t tile[32][33];
  const int64_t I = blockIdx.y, J = blockIdx.x;
  if (I > J) return;
  const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
  for (int r = r0; r < 32; r += 8) {
    const int64_t i = I * 32 + r, j = J * 32 + c;
    uint64_t k = kNoKey;
    if (i <= j && j < n) {
      k = cl_key(tri[tri_index(i, j, n)]);
      D[i * n + j] = k;
    }
    tile[r][c] = k;
  }
  __syncthreads();
  for (int r = r0; r < 32; r += 8) {
    const int64_t i = J * 32 + r, j = I * 32 + c;  // row i of the lower half, column j < i
    if (i < n && j < i) D[i * n + j] = tile[c][r];
  }
}

// Row minimum of row r over all columns j > r: one warp.
__global__ void cl_rowmin_kernel(const uint64_t* __restrict__ D, int64_t n, uint64_t* __restrict__ rk,
                                 uint32_t* __restrict__ rj) {
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
  const int lane = threadIdx.x & 31;
  for (int64_t r = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); r < n; r += warps) {
    uint64_t k = kNoKey;
    uint32_t j = kNoIdx;
#pragma unroll 8
    for (int64_t c = r + 1 + lane; c < n; c += 32) {
      const uint64_t d = D[r * n + c];
      if (d < k) {  // columns visited in increasing order per lane
        k = d;
        j = (uint32_t)c;
      }
    }
    warp_best(k, j);
    if (lane == 0) {
      rk[r] = k;
      rj[r] = j;
    }
  }
}

struct ClArgs {
  uint64_t* D;
  int64_t ld;     // row stride: the samples of the call
  int64_t n;      // rows and columns still there
  int32_t step0, steps;  // merges before this launch, and of it
  uint64_t* rk;   // row minima: key (kNoKey: merged away, or no active column to the right)
  uint32_t* rj;   // and column
  uint8_t* active;
  uint32_t* list;  // rows to rescan after a merge (not kSmem)
  uint16_t* phys;  // kSmem: row r of the n is row phys[r] of D
  int32_t* id;
  int32_t* size;
  double* Z;  // [n-1][4]
};

// Row minima, activity flags, the rescan list and the rows' places live in
// shared memory when they fit (17 bytes per sample, up to kClSmemRows samples),
// so that the per-step argmin and the rescan checks touch no global memory.
constexpr int64_t kClSmemRows = 12000;
constexpr size_t cl_smem_bytes(int64_t n) { return n <= kClSmemRows ? (size_t)n * 17 + 16 : 0; }

// Loads in flight per thread: a row of 4,096 is one batch of 4 for the whole
// CTA, or two batches of 8 for an eighth of it.
constexpr int kClUpd = 4, kClScan = 8;

template <bool kSmem>
__global__ void __launch_bounds__(kClThreads, 1) cl_main_kernel(ClArgs a) {
  extern __shared__ __align__(16) uint8_t cl_smem[];
  constexpr int kWarps = kClThreads / 32;
  __shared__ uint64_t s_k[kWarps], s_uk[kWarps], s_sk[kWarps];
  __shared__ uint32_t s_i[kWarps], s_ui[kWarps], s_si[kWarps];
  __shared__ uint32_t s_cnt[2];
  const int n = (int)a.n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  using List = std::conditional_t<kSmem, uint16_t, uint32_t>;
  uint64_t* rk;
  uint32_t* rj;
  List* list;
  uint16_t* phys = nullptr;
  uint8_t* active;
  if constexpr (kSmem) {
    rk = reinterpret_cast<uint64_t*>(cl_smem);
    rj = reinterpret_cast<uint32_t*>(cl_smem + (size_t)n * 8);
    list = reinterpret_cast<uint16_t*>(cl_smem + (size_t)n * 12);
    phys = reinterpret_cast<uint16_t*>(cl_smem + (size_t)n * 14);
    active = cl_smem + (size_t)n * 16;
    for (int r = tid; r < n; r += kClThreads) {
      rk[r] = a.rk[r];
      rj[r] = a.rj[r];
      phys[r] = a.phys[r];
      active[r] = a.active[r];
    }
  } else {
    rk = a.rk;
    rj = a.rj;
    list = a.list;
    active = a.active;
  }
  auto row_of = [&](int r) { return a.D + (size_t)(kSmem ? (int)phys[r] : r) * a.ld; };
  if (tid < 2) s_cnt[tid] = 0;
  __syncthreads();
  for (int step = 0; step < a.steps; ++step) {
    // 1. global minimum over the row minima: (value, row) lexicographic
    uint64_t k = kNoKey;
    uint32_t b = kNoIdx;
#pragma unroll 4
    for (int r = tid; r < n; r += kClThreads) {
      const uint64_t v = rk[r];
      if (v < k) {
        k = v;
        b = (uint32_t)r;
      }
    }
    warp_best(k, b);
    if (lane == 0) {
      s_k[warp] = k;
      s_i[warp] = b;
    }
    __syncthreads();
    k = s_k[lane];
    b = s_i[lane];
    warp_best(k, b);  // every warp has the result
    const int i0 = (int)b, j0 = (int)rj[b];
    uint64_t* Di = row_of(i0);
    const uint64_t* Dj = row_of(j0);
    // the update's first loads, in flight while the list is made
    uint64_t di[kClUpd], dj[kClUpd];
    auto load_update = [&](int c0) {
#pragma unroll
      for (int q = 0; q < kClUpd; ++q) {
        const int c = c0 + q * kClThreads;
        di[q] = dj[q] = kNoKey;
        if (c < n && c != i0 && c != j0 && active[c]) {
          di[q] = Di[c];
          dj[q] = Dj[c];
        }
      }
    };
    load_update(tid);
    // 2. rows that may have lost their minimum
    uint32_t* cnt = &s_cnt[step & 1];
#pragma unroll 4
    for (int c = tid; c < n; c += kClThreads) {
      const int cj = (int)rj[c];
      if ((cj == j0 && c != i0) || cj == i0) list[atomicAdd(cnt, 1u)] = (List)c;
    }
    __syncthreads();
    const uint32_t L = *cnt;
    if (tid == 0) s_cnt[(step + 1) & 1] = 0;
    // 3a. rescan the listed rows: 8, 4, 2 or 1 warps each
    const int gw = L <= 4 ? 8 : (L <= 8 ? 4 : (L <= 16 ? 2 : 1));
    for (uint32_t t = (uint32_t)(warp / gw); t < L; t += kWarps / gw) {
      const int r = (int)list[t];
      const uint64_t* Dr = row_of(r);
      const int stride = 32 * gw;
      uint64_t sk = kNoKey;
      uint32_t si = kNoIdx;
      if (r < i0 && warp % gw == 0 && lane == 0) {  // column i0 takes the max of columns i0 and j0
        const uint64_t x = ld_shared_entry(Dr + i0), y = Dr[j0];
        sk = x > y ? x : y;
        si = (uint32_t)i0;
      }
      for (int c0 = r + 1 + lane + 32 * (warp % gw); c0 < n; c0 += kClScan * stride) {
        uint64_t d[kClScan];
#pragma unroll
        for (int q = 0; q < kClScan; ++q) {
          const int c = c0 + q * stride;
          d[q] = c < n && c != i0 && c != j0 && active[c] ? Dr[c] : kNoKey;
        }
#pragma unroll
        for (int q = 0; q < kClScan; ++q) {
          const int c = c0 + q * stride;
          if (d[q] < sk || (d[q] == sk && (uint32_t)c < si && sk != kNoKey)) {
            sk = d[q];
            si = (uint32_t)c;
          }
        }
      }
      warp_best(sk, si);
      if (lane == 0) {
        if (gw == 1) {
          rk[r] = sk;
          rj[r] = si;
        } else {  // one row per group of warps
          s_sk[warp] = sk;
          s_si[warp] = si;
        }
      }
    }
    // 3b. the merged cluster's distances: elementwise max of the two rows, and
    // its new minimum.  (A rescan reads its row's entry in column i0 before or
    // after it is replaced here: the max with column j0's is the same.)
    uint64_t uk = kNoKey;
    uint32_t ui = kNoIdx;
    for (int c0 = tid;;) {
#pragma unroll
      for (int q = 0; q < kClUpd; ++q) {
        if (di[q] == kNoKey) continue;
        const int c = c0 + q * kClThreads;
        const uint64_t d = di[q] > dj[q] ? di[q] : dj[q];
        if (d != di[q]) {
          Di[c] = d;
          st_shared_entry(row_of(c) + i0, d);
        }
        if (c > i0 && d < uk) {
          uk = d;
          ui = (uint32_t)c;
        }
      }
      c0 += kClUpd * kClThreads;
      if (c0 - tid >= n) break;
      load_update(c0);
    }
    warp_best(uk, ui);
    if (lane == 0) {
      s_uk[warp] = uk;
      s_ui[warp] = ui;
    }
    __syncthreads();
    // 4. the new minima
    if (gw > 1 && (uint32_t)tid < L) {
      uint64_t sk = s_sk[tid * gw];
      uint32_t si = s_si[tid * gw];
      for (int w = 1; w < gw; ++w) {
        const uint64_t ok = s_sk[tid * gw + w];
        const uint32_t oi = s_si[tid * gw + w];
        if (ok < sk || (ok == sk && oi < si)) {
          sk = ok;
          si = oi;
        }
      }
      const uint32_t r = list[tid];
      rk[r] = sk;
      rj[r] = si;
    }
    if (warp == kWarps - 1) {
      uk = s_uk[lane];
      ui = s_ui[lane];
      warp_best(uk, ui);
      if (lane == 0) {
        rk[i0] = uk;
        rj[i0] = ui;
        rk[j0] = kNoKey;
        rj[j0] = kNoIdx;
        active[j0] = 0;
      }
    }
    if (tid == kClThreads - 64) {  // the merge itself, off the critical path
      const int32_t ia = a.id[i0], ib = a.id[j0], sz = a.size[i0] + a.size[j0];
      double* z = a.Z + (size_t)(a.step0 + step) * 4;
      z[0] = (double)(ia < ib ? ia : ib);
      z[1] = (double)(ia < ib ? ib : ia);
      z[2] = cl_value(k);
      z[3] = (double)sz;
      a.id[i0] = (int32_t)(a.ld + a.step0 + step);
      a.size[i0] = sz;
    }
    __syncthreads();
  }
  if constexpr (kSmem) {  // for cl_compact_kernel
    for (int r = tid; r < n; r += kClThreads) {
      a.rk[r] = rk[r];
      a.rj[r] = rj[r];
      a.active[r] = active[r];
    }
  }
}

// Between launches of the main kernel: rows and columns merged away are dropped
// (in order, so ties fall as before).  The arrays move down in place, a chunk at
// a time: an entry never moves up, so a chunk is read before anything is written
// over it.  act[c] = old column of new column c.
__global__ void __launch_bounds__(kClThreads, 1) cl_compact_kernel(ClArgs a, uint16_t* __restrict__ act) {
  extern __shared__ __align__(16) uint8_t cl_smem[];
  uint16_t* to = reinterpret_cast<uint16_t*>(cl_smem);  // new index of an old one
  __shared__ uint32_t s_sum[kClThreads / 32];
  const int n = (int)a.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t before = 0;
  for (int r0 = 0; r0 < n; r0 += kClThreads) {
    const int r = r0 + tid;
    const bool on = r < n && a.active[r] != 0;
    const uint32_t ballot = __ballot_sync(0xffffffffu, on);
    if (lane == 0) s_sum[warp] = __popc(ballot);
    __syncthreads();
    uint32_t at = before;
    for (int w = 0; w < kClThreads / 32; ++w) {
      if (w < warp) at += s_sum[w];
      before += s_sum[w];
    }
    at += __popc(ballot & ((1u << lane) - 1u));
    if (on) {
      to[r] = (uint16_t)at;
      act[at] = (uint16_t)r;
    }
    __syncthreads();
  }
  for (int r0 = 0; r0 < n; r0 += kClThreads) {
    const int r = r0 + tid;
    const bool on = r < n && a.active[r] != 0;
    uint64_t k = 0;
    uint32_t j = 0;
    int32_t id = 0, size = 0;
    uint16_t phys = 0;
    if (on) {
      k = a.rk[r];
      j = a.rj[r];
      id = a.id[r];
      size = a.size[r];
      phys = a.phys[r];
    }
    __syncthreads();
    if (on) {
      const int t = to[r];
      a.rk[t] = k;
      a.rj[t] = j < (uint32_t)n ? to[j] : j;
      a.id[t] = id;
      a.size[t] = size;
      a.phys[t] = phys;
    }
    __syncthreads();
  }
  for (int r = tid; r < (int)before; r += kClThreads) a.active[r] = 1;
}

// ... and the columns of the `left` rows that stay, CTA = row.
__global__ void __launch_bounds__(256) cl_compact_rows_kernel(ClArgs a, const uint16_t* __restrict__ act, int left) {
  uint64_t* row = a.D + (size_t)a.phys[blockIdx.x] * a.ld;
  constexpr int kPer = 8;
  for (int c0 = threadIdx.x; c0 - (int)threadIdx.x < left; c0 += kPer * 256) {
    uint64_t v[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int c = c0 + q * 256;
      if (c < left) v[q] = row[act[c]];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int c = c0 + q * 256;
      if (c < left) row[c] = v[q];
    }
    __syncthreads();
  }
}

// Rows and columns after the next compaction: three quarters, down to 512 (and
// only where the main kernel's state is in shared memory).  A merge costs 2.9
// us on average from 256 columns down, 3.7 from 1,024 and 7.7 from 4,096 when
// none are dropped.  4,096 samples: 24.2 ms against 31.4 (halves: 26.0; seven
// eighths: 23.7, but more launches for the smaller matrices).
int64_t cl_next(int64_t n) { return n <= 512 || n > kClSmemRows ? 1 : n * 3 / 4; }

__global__ void cl_state_init_kernel(int64_t n, uint8_t* active, int32_t* id, int32_t* size, uint16_t* phys) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    active[i] = 1;
    id[i] = (int32_t)i;
    size[i] = 1;
    if (phys != nullptr) phys[i] = (uint16_t)i;
  }
}

}  // namespace

size_t cluster_workspace_bytes(int64_t n) {
  return (size_t)n * (size_t)n * 8 + (size_t)n * (8 + 4 + 4 + 4 + 4 + 1) + 4096;
}

cudaError_t launch_cluster_complete(const double* tri, int64_t n, double* Z, void* work, int num_sms,
                                    cudaStream_t st) {
  if (n <= 1) return cudaSuccess;
  uint8_t* w = static_cast<uint8_t*>(work);
  uint64_t* D = reinterpret_cast<uint64_t*>(w);
  w += (size_t)n * n * 8;
  uint64_t* rk = reinterpret_cast<uint64_t*>(w);
  w += (size_t)n * 8;
  uint32_t* rj = reinterpret_cast<uint32_t*>(w);
  w += (size_t)n * 4;
  uint32_t* list = reinterpret_cast<uint32_t*>(w);
  w += (size_t)n * 4;
  int32_t* id = reinterpret_cast<int32_t*>(w);
  w += (size_t)n * 4;
  int32_t* size = reinterpret_cast<int32_t*>(w);
  w += (size_t)n * 4;
  uint8_t* active = w;
  const int grid = num_sms * 8;
  const unsigned T = (unsigned)((n + 31) / 32);  // at most 4,096 (n <= 131,072)
  cl_init_kernel<<<dim3(T, T), 256, 0, st>>>(tri, n, D);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // (kSmem does not use the list in global memory)
  const bool small = n <= kClSmemRows;
  uint16_t *phys = small ? reinterpret_cast<uint16_t*>(list) : nullptr, *act = small ? phys + n : nullptr;
  cl_state_init_kernel<<<grid, 256, 0, st>>>(n, active, id, size, phys);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  cl_rowmin_kernel<<<grid, 256, 0, st>>>(D, n, rk, rj);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  auto kern = small ? cl_main_kernel<true> : cl_main_kernel<false>;
  if (cl_smem_bytes(n) > 48 * 1024 &&
      (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cl_smem_bytes(n))) != cudaSuccess)
    return e;
  for (int64_t left = n; left > 1;) {
    const int64_t next = cl_next(left);
    const ClArgs args{D, n, left, (int32_t)(n - left), (int32_t)(left - next), rk, rj, active, list, phys, id, size, Z};
    kern<<<1, kClThreads, cl_smem_bytes(left), st>>>(args);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (next > 1) {
      cl_compact_kernel<<<1, kClThreads, (size_t)left * 2, st>>>(args, act);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      cl_compact_rows_kernel<<<(unsigned)next, 256, 0, st>>>(args, act, (int)next);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    left = next;
  }
  return cudaSuccess;
}

// Kernel launches of a call.
int cluster_launches(int64_t n) {
  int k = 3;
  for (int64_t left = n; left > 1; left = cl_next(left)) k += cl_next(left) > 1 ? 3 : 1;
  return k;
}

}  // namespace ibs

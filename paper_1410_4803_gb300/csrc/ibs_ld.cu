// Linkage disequilibrium: the correlation r of marker pairs within a window,
// on the tensor cores.
//
// The paper's example of bit population counts beyond identity-by-state
// ("Improvements in PLINK 1.9 / Bitwise parallelism") is the correlation
// coefficient r between two markers x and y with missing calls: x_i = +1 for
// a homozygous major call, -1 for a homozygous minor call, 0 for a
// heterozygous or missing call; with S_xy the samples where neither call is
// missing and N = |S_xy|, the paper's form with means over S_xy multiplied
// through by N^2 is
//   r = (N Sxy - Sx Sy) / sqrt((N Sxx - Sx^2) (N Syy - Sy^2)),
// Sx, Sxx, Sy, Syy, Sxy being sums over S_xy.  All six sums are products over
// the sample axis of per-marker indicator rows:
//   V = 1 present,  X = +1 hom A1 / -1 hom A2 / 0,  H = X^2 = 1 homozygous;
//   N = V_a V_b^T,  Sx = X_a V_b^T,  Sy = V_a X_b^T,  Sxx = H_a V_b^T,
//   Syy = V_a H_b^T,  Sxy = X_a X_b^T.
// They are computed relative to A1 and oriented afterwards:
// r_major = s_a s_b r_A1, with s = +1 when A1 is the major allele (#hom A1 >=
// #hom A2 over the marker's calls), which is the same as flipping x.
//
// Markers are the MMA rows (128 per block for A, 64 per half-block for B) and
// samples the K axis (64 per E2M1 chunk).  The variant-major .bed rows already
// have this orientation, so the operand builder only expands 2-bit codes into
// E2M1 values.  Every value is 0 or +-1 and every partial sum an integer of
// magnitude at most the sample count (kept below 2^24), so FP32 accumulation
// is exact.  The numerator and variance terms are formed in int64.  Only the
// reciprocal square root and the products are rounded, in float-float
// arithmetic on the FP32 pipe (see ld_r_value).
//
// One persistent CTA per SM, 20 warps: the copy warp claims (A block, B
// half-block) items of the band |b - a| <= window from a counter and streams
// each item's sample chunks through a ring of 3 stages x 3 chunks (one copy of
// the A block's 3 planes x 4 KiB per chunk, one tensor copy of the B
// half-block's 3 x 2 KiB per chunk out of the same planes: a second copy of
// them laid out for B took as long to write as the first); three
// MMA warps issue 3 MMAs (M = 128, N = 192, 128 and 64, K = 64) per chunk into
// six FP32 accumulators (64 tensor-memory columns each; unit scale factors at
// 384..511); warps 4..19 read the accumulators back (four warps per lane
// quarter, 16 columns each) and store r.  Every wait is bounded (2 s of
// %globaltimer), as in the IBS kernels.
#include <algorithm>
#include <vector>

#include "ibs_tc_common.cuh"

namespace ibs {

namespace {

constexpr int kLdPlanes = 3;                         // X, V, H
constexpr int kLdChunkBytes = kLdPlanes * kTileBytes;  // 12 KiB per (marker block, sample chunk)
constexpr int kLdHalfBytes = kTileBytes / 2;         // 64 rows of a plane tile
constexpr int kLdHalfChunkBytes = kLdPlanes * kLdHalfBytes;  // 6 KiB per (half-block, sample chunk)
// A ring stage holds kLdPer chunks of the A block and of the B half-block, one
// bulk copy each (the copy engine spends a fixed time per copy).  Beside the
// ring, each epilogue warp has a piece of 32 rows x 8 columns of r and N to
// transpose.
constexpr int kLdPer = 3;
constexpr int kLdStageBytes = kLdPer * (kLdChunkBytes + kLdHalfChunkBytes);  // 54 KiB
constexpr int kLdStages = 3;
constexpr int kLdEpiWarps = 16;
constexpr int kLdTransBytes = 32 * 9 * 12;
constexpr size_t kLdSmem = (size_t)kLdStages * kLdStageBytes + kLdEpiWarps * kLdTransBytes + 1024;
static_assert(kLdSmem <= 227 * 1024, "ring exceeds shared memory");
constexpr int kLdN = 64;                             // B rows (markers) per item
// Accumulator columns.  A chunk's X, V and H rows of B are contiguous, so one MMA
// multiplies a plane of A by two or three of them (N = 128 or 192): 3 MMAs per
// chunk; 6 of N = 64, one per sum, took 1.79 ms a call against 1.74
// (4,096 samples x 100,000 markers, window 1,000).
constexpr uint32_t kLdSy = 0, kLdCnt = 64, kLdSyy = 128, kLdSxy = 192, kLdSx = 256, kLdSxx = 320;
constexpr int kLdQueue = 8;
// warps 0 (copies), 1, 2 and 3 (MMAs), 4..19 epilogue: four warps per TMEM
// lane quarter, each reading 16 of the item's 64 accumulator columns
constexpr int kLdThreads = (4 + kLdEpiWarps) * 32;

// Even bits of a 64-bit word packed into 32 bits (bit 2i -> bit i).
__device__ __forceinline__ uint32_t even_bits(uint64_t x) {
  x &= 0x5555555555555555ull;
  x = (x | (x >> 1)) & 0x3333333333333333ull;
  x = (x | (x >> 2)) & 0x0F0F0F0F0F0F0F0Full;
  x = (x | (x >> 4)) & 0x00FF00FF00FF00FFull;
  x = (x | (x >> 8)) & 0x0000FFFF0000FFFFull;
  x = (x | (x >> 16)) & 0x00000000FFFFFFFFull;
  return (uint32_t)x;
}

// Operand rows: CTA = (sample chunk c, marker block b), thread (row r, half):
// marker b*128 + r, samples c*64 + 32*half .. +31 (8 bytes of the .bed row).
// Writes 16 bytes of each of X, V, H (E2M1: +1 = 0x2, -1 = 0xA) into
// [block][chunk][plane][128 rows]; adds the marker's #hom A1 - #hom A2 over
// these samples to diff.
__global__ void __launch_bounds__(256) ld_planes_kernel(const uint8_t* __restrict__ packed, int64_t row_bytes,
                                                        int64_t n, int64_t m, uint8_t* __restrict__ planes,
                                                        int64_t n_chunks,
                                                        int32_t* __restrict__ diff) {
  const int64_t c = blockIdx.x, b = blockIdx.y;
  const int r = threadIdx.x >> 1, half = threadIdx.x & 1;
  const int64_t k = b * kTB + r;
  const int64_t s0 = c * 64 + 32 * half;
  uint32_t a1 = 0, a2 = 0, pres = 0;
  int d = 0;
  if (k < m && s0 < n) {
    const uint8_t* row = packed + k * row_bytes + (s0 >> 2);
    const int64_t left = row_bytes - (s0 >> 2);
    uint64_t w = 0;
    if (left >= 8 && (reinterpret_cast<uintptr_t>(row) & 7) == 0) {
      w = __ldg(reinterpret_cast<const unsigned long long*>(row));
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) w |= (uint64_t)(q < left ? __ldg(row + q) : 0x55u) << (8 * q);
    }
    const uint32_t lo = even_bits(w), hi = even_bits(w >> 1);  // code bit 0, code bit 1 of 32 samples
    const uint32_t valid = n - s0 >= 32 ? 0xFFFFFFFFu : ((1u << (uint32_t)(n - s0)) - 1u);
    pres = (hi | ~lo) & valid;   // code != 1
    a1 = ~hi & ~lo & valid;      // code 0, homozygous A1
    a2 = hi & lo & valid;        // code 3, homozygous A2
    d = __popc(a1) - __popc(a2);
  }
  d += __shfl_xor_sync(0xffffffffu, d, 1);  // the row's two halves (all lanes converged here)
  if (half == 0 && k < m && d != 0) atomicAdd(diff + k, d);
  uint32_t wx[4], wv[4], wh[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const uint32_t s1 = nib8(a1 >> (8 * g)), s2 = nib8(a2 >> (8 * g)), sv = nib8(pres >> (8 * g));
    wx[g] = ((s1 | s2) << 1) | (s2 << 3);
    wv[g] = sv << 1;
    wh[g] = (s1 | s2) << 1;
  }
  uint8_t* base = planes + (size_t)(b * n_chunks + c) * kLdChunkBytes + tile_off(r, 16 * half);
  *reinterpret_cast<uint4*>(base + 0 * kTileBytes) = make_uint4(wx[0], wx[1], wx[2], wx[3]);
  *reinterpret_cast<uint4*>(base + 1 * kTileBytes) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
  *reinterpret_cast<uint4*>(base + 2 * kTileBytes) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
}

// r from the six exact sums, oriented by the two markers' signs; NaN when N = 0
// or a variance term is 0.  The numerator and the variance terms are exact
// int64 values below 2^48 (N < 2^24); they are split exactly into float-float
// pairs, and r = num / sqrt(va vb) is formed in float-float arithmetic on the
// FP32 pipe (GB300 runs FP32 at 64x its FP64 rate): the product va vb, an
// rsqrtf seed (relative error near 2^-22) refined by one Newton step whose
// residual 1 - P y^2 is taken in float-float, and the product with the
// numerator.  Error: about 1.5 * 2^-44 from the Newton step plus a few 2^-46
// from the float-float operations, well under 1e-12 relative.
struct FF {
  float hi, lo;
};

// Error-free sum (Knuth): s + e == a + b.
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

// x (|x| < 2^48) as an exact float-float: x = h 2^24 + l with 0 <= l < 2^24.
__device__ __forceinline__ FF ff_from_i48(long long x) {
  const long long h = x >> 24;  // floor: |h| < 2^24
  const int l = (int)(x - (h << 24));
  return ff_two_sum(__fmul_rn((float)(int)h, 16777216.0f), (float)l);
}

// a * b in float-float (products exact by FMA, cross terms added once).
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  const float s = __fadd_rn(p, e);
  return {s, __fsub_rn(e, __fsub_rn(s, p))};
}

// The double hi + lo (2^-70 < |hi| < 2^70, |lo| at most half an ulp of hi),
// rounded to 53 bits: lo is scaled to units of the last bit (half as large where
// lo takes a power of two below itself) and added to hi's bit pattern.  Two
// conversions of FP32 to FP64 and an FP64 addition would hold the FP64 pipe for
// 12,000 cycles per 128 x 64 pairs, as long as their MMAs.
__device__ __forceinline__ double ff_to_double(FF r) {
  const int hb = __float_as_int(r.hi), lb = __float_as_int(r.lo), e = (hb >> 23) & 0xFF;
  const int below = (hb & 0x7FFFFF) == 0 && (hb ^ lb) < 0;
  const int k = __float2int_rn(__fmul_rn(r.lo, __int_as_float((306 - e + below) << 23)));
  const long long mag =
      ((long long)(e - 127 + 1023) << 52) + ((long long)(hb & 0x7FFFFF) << 29) + (hb < 0 ? -k : k);
  return __longlong_as_double(mag | ((long long)hb & (long long)0x8000000000000000ull));
}

// r = num / sqrt(va vb) from exact float-float operands, va and vb positive.
__device__ __forceinline__ double ld_r_quotient(FF num, FF va, FF vb) {
  if (num.hi == 0.0f) return 0.0;
  const FF P = ff_mul(va, vb);
  const float y0 = rsqrtf(P.hi);
  const float q = __fmul_rn(y0, y0);
  const FF w = ff_mul(P, FF{q, __fmaf_rn(y0, y0, -q)});  // P y0^2, near 1
  const float t = __fsub_rn(__fsub_rn(1.0f, w.hi), w.lo);  // 1 - P y0^2 (the first difference is exact)
  const FF y = ff_two_sum(y0, __fmul_rn(__fmul_rn(y0, t), 0.5f));  // one Newton step
  return ff_to_double(ff_mul(num, y));
}

// x (|x| < 2^30) as an exact float-float, without conversions (they issue at a
// quarter of the rate): x = h 2^15 + l, both made floats by their bit patterns.
__device__ __forceinline__ FF ff_from_i30(int x) {
  const float h = __fsub_rn(__int_as_float(0x4B400000 + (x >> 15)), 12582912.0f);
  const float l = __fsub_rn(__int_as_float(0x4B000000 | (x & 0x7FFF)), 8388608.0f);
  const float s = __fmaf_rn(h, 32768.0f, l);
  return {s, __fadd_rn(__fmaf_rn(h, 32768.0f, -s), l)};
}

// The six sums of a pair, each below 2^15 in magnitude (fewer than 2^15
// samples), in three words.
struct LdSums {
  uint32_t a, b, c;
};
__device__ __forceinline__ uint32_t ld_pack(uint32_t lo, uint32_t hi) {
  // adding 1.5 * 2^23 leaves the integer in the low bits of the pattern
  return __byte_perm(__float_as_uint(__fadd_rn(__uint_as_float(lo), 12582912.0f)),
                     __float_as_uint(__fadd_rn(__uint_as_float(hi), 12582912.0f)), 0x5410);
}
__device__ __forceinline__ double ld_r_small(const LdSums& p, int sign) {
  const int N = (int)(p.a & 0xFFFF), sxx = (int)(p.a >> 16), syy = (int)(p.b & 0xFFFF);
  const int sx = (int)p.b >> 16, sy = (int)(p.c << 16) >> 16, sxy = (int)p.c >> 16;
  const int va = N * sxx - sx * sx, vb = N * syy - sy * sy;  // 0 <= . < 2^30
  if (va == 0 || vb == 0) return __longlong_as_double(0x7ff8000000000000LL);
  const int num = N * sxy - sx * sy;
  return ld_r_quotient(ff_from_i30(sign < 0 ? -num : num), ff_from_i30(va), ff_from_i30(vb));
}

__device__ __forceinline__ double ld_r_value(int32_t N, int32_t sx, int32_t sy, int32_t sxx, int32_t syy,
                                             int32_t sxy, int sign) {
  const long long n = N;
  const long long va = n * sxx - (long long)sx * sx, vb = n * syy - (long long)sy * sy;
  if (N == 0 || va == 0 || vb == 0) return __longlong_as_double(0x7ff8000000000000LL);
  const long long num = n * sxy - (long long)sx * sy;
  return ld_r_quotient(ff_from_i48(sign * num), ff_from_i48(va), ff_from_i48(vb));
}

struct LdArgs {
  const uint8_t* planes;    // A layout
  int64_t n_chunks, m, window;
  const int2* items;  // (A marker block, B half-block)
  int64_t n_items;
  const int32_t* diff;
  double* out_r;
  int32_t* out_n;
  int* counter;
  int* status;
};

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x0, int x1, int x2, int x3,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(smem_addr(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// kSmall: fewer than 2^15 samples.  The epilogue then packs the six sums of its
// 32 rows x 16 columns into registers and hands tensor memory back before it
// computes, so that the next item's MMAs run beside the arithmetic; with more
// samples the accumulators are held while the first half is computed.  The
// arithmetic is integer and FP32 only, and the stores go through shared memory.
// With FP64 arithmetic on held accumulators and one lane per marker row the
// call took 2.33 ms (4,096 samples x 100,000 markers, window 1,000); 1.74 with
// 8 epilogue warps, 1.67 with 16 (and 1.58 with three MMA warps instead of two).
template <bool kSmall>
__global__ void __launch_bounds__(kLdThreads, 1) tc_ld_kernel(const __grid_constant__ CUtensorMap bmap, const LdArgs args) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full[kLdStages], empty[kLdStages], tfull, tempty, drain;
  __shared__ __align__(8) uint64_t qfull[kLdQueue], qempty[kLdQueue];
  __shared__ int64_t q_item[kLdQueue];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* status = args.status;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kLdStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 3);  // the MMA warps' commits
    }
    for (int s = 0; s < kLdQueue; ++s) {
      mbar_init(&qfull[s], 1);
      mbar_init(&qempty[s], 3 + kLdEpiWarps);  // the MMA warps and the epilogue warps
    }
    mbar_init(&tfull, 3);
    mbar_init(&tempty, kLdEpiWarps);
    mbar_init(&drain, 3);
    mbar_fence_init();
    abort_flag = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (warp >= 4 && warp < 8) tmem_fill_unit_scales(tmem, warp - 4);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  auto fail = [&] {  // one thread
    if (*(volatile int*)&abort_flag == 0) {
      atomicExch(status, kDevTimeout);
      atomicExch(&abort_flag, 1);
    }
  };
  // one thread's next item: false after a failed wait
  auto queue_get = [&](uint32_t e, int64_t& it) {
    const int qs = (int)(e % kLdQueue);
    if (!ring_wait(&qfull[qs], (e / kLdQueue) & 1u, kWaitLimitNs, &abort_flag)) return false;
    it = *(volatile int64_t*)&q_item[qs];
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&qempty[qs])) : "memory");
    return true;
  };
  const int64_t nk = args.n_chunks;  // whole stages

  if (warp == 0) {
    if (lane == 0) {
      uint32_t g = 0, s = 0, ph = 1;  // stages issued, ring slot, parity of the slot's previous release
      bool ok = true;
      for (uint32_t e = 0; ok; ++e) {
        int64_t it = atomicAdd(args.counter, 1);
        if (it >= args.n_items) it = -1;
        const int qs = (int)(e % kLdQueue);
        if (e >= (uint32_t)kLdQueue && !ring_wait(&qempty[qs], ((e / kLdQueue) - 1) & 1u, kWaitLimitNs, &abort_flag)) {
          ok = false;
          break;
        }
        q_item[qs] = it;
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&qfull[qs])) : "memory");
        if (it < 0) break;
        const int2 item = args.items[it];
        const uint8_t* a = args.planes + (size_t)item.x * nk * kLdChunkBytes;
        int b = (int)((item.y >> 1) * nk);  // chunk of the B half-block's block
        for (int64_t k = 0; k < nk; k += kLdPer, a += kLdPer * kLdChunkBytes, b += kLdPer) {
          if (g >= (uint32_t)kLdStages && !ring_wait(&empty[s], ph, kWaitLimitNs, &abort_flag)) {
            ok = false;
            break;
          }
          uint8_t* dst = ring + (size_t)s * kLdStageBytes;
          mbar_arrive_expect_tx(&full[s], kLdStageBytes);
          bulk_g2s(dst, a, kLdPer * kLdChunkBytes, &full[s]);
          tma_load_4d(dst + kLdPer * kLdChunkBytes, &bmap, 0, item.y & 1, 0, b, &full[s]);
          ++g;
          if (++s == kLdStages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) fail();
      // (after a stop: the copies in flight land before the CTA may exit)
      for (uint32_t j = g > (uint32_t)kLdStages ? g - kLdStages : 0; j < g && !ok; ++j)
        mbar_wait_bounded(&full[j % kLdStages], (j / kLdStages) & 1u);
    }
    __syncwarp();
  } else if (warp < 4) {
    // Three MMA warps with accumulators and products of their own: V_a times the
    // three planes of B, X_a times two, H_a times one.  One warp's MMAs run while
    // another commits a stage and waits for the next (the tensor core queues hardly more than the MMA it runs).  Each waits
    // (bounded), at an item's start, until the epilogue has read the previous
    // item's accumulators, and for each stage until its operands have landed;
    // after a failed wait or another role's abort nothing more is issued.
    if (lane == 0) {
      uint32_t s = 0, ph = 0;
      const uint32_t sf = tmem + kSfCol, ring0 = smem_addr(ring);
      bool ok = true;
      for (uint32_t e = 0; ok; ++e) {
        int64_t it = -1;
        ok = queue_get(e, it);
        if (!ok || it < 0) break;
        if (e > 0) ok = mbar_wait_bounded(&tempty, (e - 1) & 1u);
        for (int64_t k0 = 0; k0 < nk && ok; k0 += kLdPer) {
          if (!ring_wait(&full[s], ph, kWaitLimitNs, &abort_flag)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st0 = ring0 + s * kLdStageBytes;
#pragma unroll
          for (int c = 0; c < kLdPer; ++c) {
            // X, V and H of a chunk, 4 KiB each of A and 2 KiB each of B
            const uint32_t a0 = st0 + c * kLdChunkBytes, b0 = st0 + kLdPer * kLdChunkBytes + c * kLdHalfChunkBytes;
            const uint32_t acc = k0 + c > 0 ? 1u : 0u;
            if (warp == 1) {
              umma<kTcFp4, 3 * kLdN>(tmem + kLdSy, umma_desc(a0 + kTileBytes), umma_desc(b0), acc, sf);
            } else if (warp == 2) {
              umma<kTcFp4, 2 * kLdN>(tmem + kLdSxy, umma_desc(a0), umma_desc(b0), acc, sf);
            } else {
              umma<kTcFp4, kLdN>(tmem + kLdSxx, umma_desc(a0 + 2 * kTileBytes), umma_desc(b0 + kLdHalfBytes), acc, sf);
            }
          }
          umma_commit(&empty[s]);
          if (++s == kLdStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        umma_commit(&tfull);
      }
      if (!ok) fail();
      umma_commit(&drain);
    }
    __syncwarp();
    const bool drained = mbar_wait_bounded(&drain, 0);
    if (lane == 0 && !drained) atomicExch(status, kDevTimeout);
  } else if (warp >= 4) {
    const int quarter = warp & 3, colq = (warp - 4) >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + 16 * colq;
    uint8_t* trans = ring + (size_t)kLdStages * kLdStageBytes + (size_t)(warp - 4) * kLdTransBytes;
    double* sr = reinterpret_cast<double*>(trans);
    int32_t* sn = reinterpret_cast<int32_t*>(trans + 32 * 9 * 8);
    for (uint32_t e = 0;; ++e) {
      int64_t it = -1;
      bool ok = true;
      if (lane == 0) ok = queue_get(e, it);
      it = __shfl_sync(0xffffffffu, it, 0);
      if (ok && it >= 0) ok = mbar_wait_bounded(&tfull, e & 1u) && *(volatile int*)&abort_flag == 0;
      if (__any_sync(0xffffffffu, !ok)) {
        if (lane == 0) fail();
        break;
      }
      if (it < 0) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int2 item = args.items[it];
      const int64_t a0 = (int64_t)item.x * kTB + quarter * 32, b0 = (int64_t)item.y * kLdN + 16 * colq;
      // markers whose major allele is A2: this thread's row, the warp's 16 columns
      const bool minus = a0 + lane < args.m && args.diff[a0 + lane] < 0;
      const uint32_t bminus = __ballot_sync(0xffffffffu, lane < 16 && b0 + lane < args.m && args.diff[b0 + lane] < 0);
      auto hand_back = [&] {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&tempty)) : "memory");
      };
      // Columns u0 .. u0 + 7 of the warp's: r of (row, column u) from value(u), N
      // from count(u); transposed through shared memory, so that 8 lanes store 8
      // consecutive pairs of a marker.
      auto put = [&](int u0, auto&& value, auto&& count) {
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          sr[lane * 9 + u] = value(u, ((bminus >> (u0 + u)) & 1u) != (minus ? 1u : 0u) ? -1 : 1);
          sn[lane * 9 + u] = count(u);
        }
        __syncwarp();
        const int64_t b = b0 + u0 + (lane & 7), a1 = a0 + (lane >> 3);
        int64_t d = b - a1 - 1, at = a1 * args.window + d;
#pragma unroll
        for (int r = 0; r < 32; r += 4, d -= 4, at += 4 * args.window - 4) {
          if (d < 0 || d >= args.window || b >= args.m) continue;  // (b > the row's marker: that is below m too)
          const int from = (r + (lane >> 3)) * 9 + (lane & 7);
          args.out_r[at] = sr[from];
          if (args.out_n) args.out_n[at] = sn[from];
        }
      };
      if constexpr (kSmall) {
        LdSums p[16];
        uint32_t lo[16], hi[16];
        auto pair = [&](uint32_t ql, uint32_t qh) {
          tmem_ld16(lane_base + ql, lo);
          tmem_ld16(lane_base + qh, hi);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        };
        pair(kLdCnt, kLdSxx);
#pragma unroll
        for (int u = 0; u < 16; ++u) p[u].a = ld_pack(lo[u], hi[u]);
        pair(kLdSyy, kLdSx);
#pragma unroll
        for (int u = 0; u < 16; ++u) p[u].b = ld_pack(lo[u], hi[u]);
        pair(kLdSy, kLdSxy);
        hand_back();
#pragma unroll
        for (int u = 0; u < 16; ++u) p[u].c = ld_pack(lo[u], hi[u]);
#pragma unroll
        for (int u0 = 0; u0 < 16; u0 += 8)
          put(u0, [&](int u, int sign) { return ld_r_small(p[u0 + u], sign); },
              [&](int u) { return (int)(p[u0 + u].a & 0xFFFF); });
      } else {
#pragma unroll 1
        for (int u0 = 0; u0 < 16; u0 += 8) {
          constexpr uint32_t col[6] = {kLdCnt, kLdSx, kLdSy, kLdSxx, kLdSyy, kLdSxy};
          uint32_t v[6][8];
#pragma unroll
          for (int q = 0; q < 6; ++q) tmem_ld8(lane_base + col[q] + u0, v[q]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (u0 == 8) hand_back();
          auto sum = [&](int q, int u) { return __float2int_rn(__uint_as_float(v[q][u])); };
          put(u0,
              [&](int u, int sign) {
                return ld_r_value(sum(0, u), sum(1, u), sum(2, u), sum(3, u), sum(4, u), sum(5, u), sign);
              },
              [&](int u) { return sum(0, u); });
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// Slots whose second marker lies past the last one: r = NaN, N = 0.
__global__ void ld_fill_tail_kernel(int64_t m, int64_t window, double* __restrict__ out_r,
                                    int32_t* __restrict__ out_n) {
  const int64_t a0 = m > window ? m - window : 0;
  const int64_t total = (m - a0) * window;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = a0 + t / window, d = t % window;
    if (a + 1 + d < m) continue;
    out_r[a * window + d] = __longlong_as_double(0x7ff8000000000000LL);
    if (out_n) out_n[a * window + d] = 0;
  }
}

// The planes as 64-bit elements, [block x chunk][plane][half-block][256]: a box is
// one half-block's rows of kLdPer chunks.
bool encode_ld_map(CUtensorMap* map, const void* planes, int64_t chunks) {
  const EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {256, 2, kLdPlanes, (cuuint64_t)chunks};
  const cuuint64_t strides[3] = {(cuuint64_t)kLdHalfBytes, (cuuint64_t)kTileBytes, (cuuint64_t)kLdChunkBytes};
  const cuuint32_t box[4] = {256, 1, kLdPlanes, kLdPer};
  const cuuint32_t elem[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<void*>(planes), dims, strides, box, elem,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Sample chunks: ceil(n / 64), padded to a multiple of kLdPer with zero chunks.
static int64_t ld_chunks(int64_t n) { return ((n + 63) / 64 + kLdPer - 1) / kLdPer * kLdPer; }

size_t ld_planes_bytes(int64_t n, int64_t m) {
  return (size_t)((m + kTB - 1) / kTB) * (size_t)ld_chunks(n) * kLdChunkBytes;
}

// Items of the band: (A block I of 128 markers, B half-block j of 64 markers)
// holding at least one pair a < b <= a + window, in order of I then j.
void ld_items(int64_t m, int64_t window, std::vector<int2>& items) {
  items.clear();
  const int64_t nb = (m + kTB - 1) / kTB, nh = (m + kLdN - 1) / kLdN;
  for (int64_t I = 0; I < nb; ++I) {
    const int64_t a_min = I * kTB, a_max = std::min<int64_t>(a_min + kTB - 1, m - 1);
    const int64_t j0 = std::max<int64_t>(0, (a_min + 1) / kLdN);
    const int64_t j1 = std::min<int64_t>(nh - 1, (a_max + window) / kLdN);
    for (int64_t j = j0; j <= j1; ++j) items.push_back(make_int2((int)I, (int)j));
  }
}

cudaError_t launch_ld(const uint8_t* packed, int64_t n, int64_t m, int64_t window, uint8_t* planes, int32_t* diff,
                      const int2* items, int64_t n_items, int* counter, double* out_r, int32_t* out_n,
                      int* status, int num_sms, cudaStream_t st) {
  const int64_t nc = ld_chunks(n), nb = (m + kTB - 1) / kTB;
  if (nc > 2147483647LL || nb > 65535 || nb * nc > 2147483647LL || n_items > 2147483647LL - num_sms) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(diff, 0, (size_t)m * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  ld_planes_kernel<<<dim3((unsigned)nc, (unsigned)nb), 256, 0, st>>>(packed, (n + 3) / 4, n, m, planes, nc, diff);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(counter, 0, sizeof(int), st)) != cudaSuccess) return e;
  auto kern = n < (1 << 15) ? tc_ld_kernel<true> : tc_ld_kernel<false>;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLdSmem)) != cudaSuccess)
    return e;
  LdArgs args{planes, nc, m, window, items, n_items, diff, out_r, out_n, counter, status};
  if (n_items > 0) {
    CUtensorMap bmap;
    if (!encode_ld_map(&bmap, planes, nb * nc)) return cudaErrorInvalidValue;
    kern<<<(int)std::min<int64_t>(num_sms, n_items), kLdThreads, kLdSmem, st>>>(bmap, args);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  ld_fill_tail_kernel<<<64, 256, 0, st>>>(m, window, out_r, out_n);
  return cudaGetLastError();
}

}  // namespace ibs

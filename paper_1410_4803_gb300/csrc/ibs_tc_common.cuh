// Building blocks of the tensor-core kernels (tcgen05): operand-tile layout,
// shared-memory and instruction descriptors, the MMA, commit and
// tensor-memory load wrappers, the unit scale factors of the block-scaled E2M1
// kind, and the bit-to-operand expansions.  Included by ibs_tc.cu (IBS pair
// counts) and ibs_ld.cu (LD correlation); each translation unit gets its own
// copy of these inline definitions.
//
// Operand tiles: 128 rows x 32 bytes (one MMA K step: 64 E2M1 or 32 E4M3
// values per row) in the canonical K-major layout without swizzle: 8-row x
// 16-byte core matrices, the two core matrices of a row group 128 bytes apart
// (leading byte offset), row groups 256 bytes apart (stride byte offset).
// Rows 64..127 of a tile are its second contiguous 2 KiB, so a 64-row operand
// is half a tile.
#pragma once

#include <cstdint>

#include <cuda.h>

#include "ibs_device.cuh"
#include "ibs_internal.h"

namespace ibs {
namespace {

constexpr int kTB = 128;                          // samples per block (tile edge)
constexpr int kTileBytes = kTB * 32;              // one plane of one chunk: 128 rows x 32 bytes
constexpr uint32_t kTmemCols = 512;               // accumulators at 0/128/256, FP4 scale factors at 384..511
constexpr uint32_t kSfCol = 384;                  // scale factors of A at 384, of B at 448
constexpr uint8_t kFp8One = 0x38;                 // E4M3 1.0 (sign bit 0x80 makes -1.0)

// markers per chunk: one MMA K step
template <int F>
constexpr int kMarkers = F == kTcFp4 ? 64 : 32;

__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(128 >> 4) << 16;   // leading byte offset: next core matrix along K
  d |= (uint64_t)(256 >> 4) << 32;   // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;            // descriptor version
  return d;                          // no swizzle
}

// Instruction descriptors, K-major A and B, M = 128.
// E4M3 x E4M3 -> F32 (kind::f8f6f4): D format F32 (bit 4), A and B formats
// E4M3 (0 at bits 7 and 10), N >> 3 at bit 17, M >> 4 at bit 24.
template <int N>
constexpr uint32_t kIdescFp8 = (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(N >> 3) << 17) |
                               ((uint32_t)(128 >> 4) << 24);
// Block-scaled E2M1 x E2M1 -> F32 (kind::mxf4): scale-factor ids 0 (bits 4
// and 29), A and B formats E2M1 (1 at bits 7 and 10), N >> 3 at bit 17, scale
// format UE8M0 (bit 23), M >> 4 at bit 24, K = 64.
template <int N>
constexpr uint32_t kIdescFp4 = (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) |
                               ((uint32_t)(128 >> 4) << 24);

// One MMA of the operand kind F, M = 128 and N columns; sf = the TMEM address
// of the scale factors (E2M1 only).
template <int F, int N = 128>
__device__ __forceinline__ void umma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc, uint32_t sf) {
  if constexpr (F == kTcFp4) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(
            tmem),
        "l"(a), "l"(b), "r"(kIdescFp4<N>), "r"(acc), "r"(sf), "r"(sf + 64u)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(a), "l"(b), "r"(kIdescFp8<N>), "r"(acc)
        : "memory");
  }
}

// FP4: every scale factor the MMAs can read is 1.0.  The calling warp fills
// its 32 TMEM lanes (quarter = warp % 4) at columns 384..511 with UE8M0 127
// bytes, so the factors read are 1.0 whichever byte and column of that range
// the hardware picks for a row.
__device__ __forceinline__ void tmem_fill_unit_scales(uint32_t tmem, int quarter) {
  const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + kSfCol;
  const uint32_t one = 0x7F7F7F7Fu;
#pragma unroll
  for (int c = 0; c < 128; c += 32)
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,"
        "%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(base + c),
        "r"(one)
        : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
      "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// Byte offset of (sample row r, byte column k) inside one 128 x 32-byte
// canonical tile (FP8: k is the marker; FP4: marker pair k holds markers 2k, 2k+1).
__device__ __forceinline__ int tile_off(int r, int k) {
  return (r >> 3) * 256 + (k >> 4) * 128 + (r & 7) * 16 + (k & 15);
}

// ---------------------------------------------------------------------------
// Indicator bits -> operand bytes.  FP8: 4 bits become 4 bytes with a
// multiply, (x * 0x204081) & 0x01010101, and a second multiply makes each 1
// the E4M3 value.  FP4: 8 bits become 8 nibbles (bit t to bit 4t) by three
// shift-or-mask steps; E2M1 1.0 is 0b0010 and -1.0 is 0b1010.
__device__ __forceinline__ uint32_t spread4(uint32_t x) { return (x * 0x00204081u) & 0x01010101u; }

__device__ __forceinline__ uint32_t nib8(uint32_t x) {
  x &= 0xFFu;
  x = (x | (x << 12)) & 0x000F000Fu;
  x = (x | (x << 6)) & 0x03030303u;
  x = (x | (x << 3)) & 0x11111111u;
  return x;
}

// 32 x 32 bit transpose across a warp: lane i's bit j becomes lane j's bit i.
__device__ __forceinline__ uint32_t tc_transpose32(uint32_t x, int lane) {
  constexpr uint32_t kMask[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    const int j = 16 >> r;
    const uint32_t m = kMask[r];
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) == 0 ? ((x & m) | ((y & m) << j)) : ((x & ~m) | ((y & ~m) >> j));
  }
  return x;
}

// A ring barrier's wait: non-blocking probes on the usual path (a thread that
// has suspended in try_wait wakes late: 76.6 ms against 73.8 for 20,000 samples
// x 500,000 markers); past a few hundred, bounded by limit_ns and ended by
// another role's abort.
__device__ __noinline__ bool ring_wait_slow(uint64_t* bar, uint32_t parity, unsigned long long limit_ns,
                                             const int* abort_flag) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    if (limit_ns < 1000000ull) {  // short bounds (tests): a blocking probe could outlast them
      if (mbar_test_wait(bar, parity)) return true;
    } else {
      for (int i = 0; i < 64; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    }
    if (*(volatile const int*)abort_flag != 0 || globaltimer_ns() - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ bool ring_wait(uint64_t* bar, uint32_t parity, unsigned long long limit_ns,
                                           const int* abort_flag) {
  if (limit_ns >= 1000000ull) {
    for (int i = 0; i < 400; ++i)
      if (mbar_test_wait(bar, parity)) return true;
  }
  return ring_wait_slow(bar, parity, limit_ns, abort_flag);
}

// ---------------------------------------------------------------------------
// Clusters of two CTAs (the two-SM kernels).
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_index() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_total() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// Every thread of both CTAs: release this CTA's prior writes, acquire the peer's.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared variable in cluster CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Waits on a barrier that the peer CTA also arrives on (acquire at cluster scope).
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint64_t* bar, uint32_t parity,
                                                          unsigned long long limit_ns = kWaitLimitNs) {
  if (limit_ns < 1000000ull) {  // short bounds (tests): non-blocking probes, clock read after each
    const unsigned long long t0 = globaltimer_ns();
    for (;;) {
      uint32_t ok;
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(ok)
          : "r"(smem_addr(bar)), "r"(parity)
          : "memory");
      if (ok) return true;
      if (globaltimer_ns() - t0 > limit_ns) return false;
    }
  }
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait_cluster(bar, parity)) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}
// A box copy issued by either CTA of the pair, completing on the barrier at
// `bar` (a shared::cluster address: the even CTA's barrier), so the even CTA's
// MMA warp sees both CTAs' operands land on one barrier.
__device__ __forceinline__ void tma_load_4d_pair(void* dst, const CUtensorMap* map, int x0, int x1, int x2, int x3,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, "
      "%3, %4, %5}], [%6];" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(bar)
      : "memory");
}

// Arrives on the barrier at this offset in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void umma_commit_both(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_addr(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void umma_commit_local2(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
// Wait until *counter >= need (a counter that other CTAs advance; bounded).
__device__ __forceinline__ bool wait_ready(const int* counter, int need, unsigned long long limit_ns) {
  const unsigned long long t0 = globaltimer_ns();
  for (unsigned ns = 32;; ns = ns < 1024 ? 2 * ns : ns) {
    int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if (v >= need) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
    __nanosleep(ns);
  }
}

// cuTensorMapEncodeTiled, from the driver through the runtime (no link-time
// dependency on libcuda).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return (EncodeTiledFn) nullptr;
    }
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

}  // namespace
}  // namespace ibs

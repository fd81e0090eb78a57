// Pair counts in marker sweeps: the two-SM tensor-core kernel of ibs_compute.
//
// The indicator products are those of ibs_tc.cu: per sample and marker V = 1
// present, U = +1 homozygous / -1 heterozygous, Q = 1 homozygous A2, R = 1
// homozygous A1 (0 when missing), N = V V^T, IBS1 = (N - U U^T) / 2,
// IBS0 = Q R^T + R Q^T, all exact integers in FP32.  That kernel streams all
// four planes of a tile together into three accumulators of 128 columns.  Here
// a tile is swept over the marker axis once per product, one plane pair at a
// time: V V^T, then U U^T, then Q R^T and R Q^T in turn, ring stage by ring stage
// (so that the second finds its planes in L2: one after the other they took a
// third more HBM reads, 3.5 GB against 2.4 for 6,000 samples x 60,000 markers),
// and the 384 accumulator columns of tensor memory hold one product of a tile
// three times as wide: a cluster of two CTAs computes 256 x 384 pairs.  Per SM
// and 96 markers of one product that is 6 KiB of A and 9 KiB of B for three
// 128 x 128 results, 13.3 KiB per result, plane set and 64 markers against 24
// KiB for 256 x 128 tiles with all planes together.  Between sweeps the
// accumulators go to a scratch buffer (three values per pair, in L2).
//
// The MMAs are kind::mxf4 with K = 96 (sm_103a; bit 31 of the instruction
// descriptor), M = 256, N = 192 over the CTA pair.  Measured back to back from
// shared memory on all SMs: 96 cycles each, 14.5 PFLOP/s; N = 256: 128 cycles,
// the same rate; N = 128: 76 cycles, 12.2 PFLOP/s; K = 64: 9.7 PFLOP/s for
// every N.  One CTA's MMAs (cta_group::1) reach 9.7 at K = 96, N = 128 and
// 12.9 at N = 256.
//
// Operand planes: [plane][64-sample half-block][32-marker column][64 rows][16
// bytes], E2M1, so a column of a half-block is 1 KiB in the canonical K-major
// layout without swizzle (8-row x 16-byte core matrices 128 bytes apart), and
// a K step of 96 markers is three columns.  One tensor map box copies any
// number of half-blocks over kSwCols columns into [column][half-block][1 KiB],
// an operand whose rows are one contiguous run per column.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <utility>
#include <vector>

#include "ibs_tc_common.cuh"

namespace ibs {

namespace {

// A ring stage is kSwCols columns (three K steps): 18 KiB of A and up to 27
// KiB of B.  With one copying thread a stage costs about 500 cycles whatever its
// size (barrier wait, two copies, release; copies alone: 31, 62 and 95 B/clk per
// SM for stages of 3, 6 and 9 columns, 95 B/clk also for 12), and the MMAs of
// three K steps take 576.  As built (a copying thread per operand), 4,096 x
// 100,000 takes 1,033 us with 4 stages of 9 columns, 1,089 with 6 of 6 and 1,065
// with 3 of 12.
constexpr int kSwCols = 9;
constexpr int kSwMarkers = 32 * kSwCols;  // 288
constexpr int kSwStages = 4;
constexpr int kSwABytes = kSwCols * 2048, kSwBBytes = kSwCols * 3072;
constexpr int kSwStageBytes = kSwABytes + kSwBBytes;
constexpr int kSwEpiWarps = 8;  // two per tensor-memory lane quarter
constexpr int kSwThreads = 128 + 32 * kSwEpiWarps;
constexpr int kSwTransBytes = 32 * 17 * 8;  // per epilogue warp: the counts of 32 x 16 pairs, packed
constexpr size_t kSwSmem = (size_t)kSwStages * kSwStageBytes + kSwEpiWarps * kSwTransBytes + 1024;
static_assert(kSwSmem <= 227 * 1024, "ring exceeds shared memory");
constexpr int kSwTileCols = 384;
constexpr size_t kSwHalfTile = (size_t)kSwTileCols * kTB;  // values of one product of one CTA's 128 x 384 tile
constexpr int kSwEpiBar = 1;  // hardware barrier of the epilogue warps

// kind::mxf4, E2M1 x E2M1 -> F32, UE8M0 scale factors, K = 96, M = 256.
template <int N>
constexpr uint32_t kIdescSweep = (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) |
                                 ((uint32_t)(256 >> 4) << 24) | (1u << 31);

template <int N>
__device__ __forceinline__ void umma_sweep(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc, uint32_t sf) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(kIdescSweep<N>), "r"(acc), "r"(sf), "r"(sf + 64u)
      : "memory");
}

// Operand of rows 16 bytes apart in columns `col` bytes apart (K core matrices).
__device__ __forceinline__ uint64_t sweep_desc(uint32_t saddr, uint32_t col) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | (uint64_t)(col >> 4) << 16 | (uint64_t)(128 >> 4) << 32 |
         (uint64_t)1 << 46;
}

// Programmatic dependent launch: the operand builder, the sweeps and the sums of
// a call follow each other without draining the machine in between; each starts
// its set-up when the one before lets it and waits here until that one's results
// are complete.  256 samples x 4,096 markers: 47 -> 42 us from Python, 1,501 x
// 30,011 101 -> 98.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The 16 bytes (64 samples) from byte0 on of marker row `marker` of `m`: any
// alignment; beyond the row or the matrix, missing.
__device__ __forceinline__ void sweep_row64(const uint8_t* __restrict__ packed, int64_t row_bytes, int64_t marker,
                                            int64_t m, int64_t byte0, uint32_t (&w)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) w[i] = 0x55555555u;  // missing
  if (marker >= m) return;
  const uint8_t* p = packed + marker * row_bytes + byte0;
  const int64_t left = row_bytes - byte0;  // bytes of the row from here on
  const uintptr_t at = reinterpret_cast<uintptr_t>(p);
  if (left >= 16 && (at & 15) == 0) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
  } else if (left >= 16 && marker > 0 && marker + 1 < m) {
    // five aligned words, all inside the matrix (the row is neither its first
    // nor its last), shifted into place
    const uint32_t* q = reinterpret_cast<const uint32_t*>(at & ~(uintptr_t)3);
    const int sh = 8 * (int)(at & 3);
    uint32_t v[5];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __ldg(q + i);
    v[4] = sh ? __ldg(q + 4) : 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(v[i], v[i + 1], sh);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t v = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b)
        v |= (uint32_t)(4 * i + b < left ? __ldg(p + 4 * i + b) : (uint8_t)0x55) << (8 * b);
      w[i] = v;
    }
  }
}

// ---------------------------------------------------------------------------
// Packed .bed rows -> operand planes.  Warp = one column of one half-block: lane
// t reads the 16 bytes (64 samples) of marker row t, and each of the four
// 16-sample words is transposed by warp shuffles; then lanes 2s and 2s + 1
// hold the low and the high code bits of sample s at the 32 markers, exchange
// them, and write 16 bytes of V and U (even lanes) or Q and R (odd lanes).  The
// eight warps of a CTA take neighbouring half-blocks, so the CTA reads whole
// 128-byte lines of the rows, and every store of a warp is 256 contiguous bytes
// per plane.  HBM-bound: 0.25 B read and 2 B written per genotype.
__global__ void __launch_bounds__(256) sweep_planes_kernel(const uint8_t* __restrict__ packed, int64_t row_bytes,
                                                           int64_t n, int64_t m, uint8_t* __restrict__ planes,
                                                           int64_t n_half, int64_t n_cols) {
  let_next_start();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t c = blockIdx.x, h = (int64_t)blockIdx.y * 8 + warp;
  if (h >= n_half) return;
  const int64_t marker = c * 32 + lane;
  uint32_t w[4];
  sweep_row64(packed, row_bytes, marker, m, h * 16, w);
  const bool odd = (lane & 1) != 0;
  const size_t plane_stride = (size_t)n_half * n_cols * 1024;
  uint8_t* base = planes + (size_t)(odd ? 2 : 0) * plane_stride + ((size_t)h * n_cols + c) * 1024;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t x = tc_transpose32(w[i], lane);
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, 1);
    const uint32_t L = odd ? y : x, H = odd ? x : y;
    const int s = i * 16 + (lane >> 1);
    const uint32_t mask = h * 64 + s < n ? 0xFFFFFFFFu : 0u;
    const uint32_t a = (odd ? H & L : H | ~L) & mask;    // Q, or V
    const uint32_t b = (odd ? ~H & ~L : H & ~L) & mask;  // R, or heterozygous
    uint32_t wa[4], wb[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const uint32_t na = nib8(a >> (8 * g)) << 1, nb = nib8(b >> (8 * g));
      wa[g] = na;
      wb[g] = odd ? nb << 1 : na | (nb << 3);  // R, or U with the sign bit of heterozygous calls
    }
    *reinterpret_cast<uint4*>(base + s * 16) = make_uint4(wa[0], wa[1], wa[2], wa[3]);
    *reinterpret_cast<uint4*>(base + plane_stride + s * 16) = make_uint4(wb[0], wb[1], wb[2], wb[3]);
  }
}

// ---------------------------------------------------------------------------
// Outputs of a tile.

// Counts of one pair, packed (N, IBS0, IBS1, each below 2^21).
struct SweepCounts {
  int32_t i0, i1, n;
};
__device__ __forceinline__ uint64_t sweep_pack(float vn, float vu, float vz) {
  const uint32_t nn = (uint32_t)__float2int_rn(vn), i0 = (uint32_t)__float2int_rn(vz);
  const uint32_t i1 = (nn - (uint32_t)__float2int_rn(vu)) >> 1;
  return (uint64_t)nn << 42 | (uint64_t)i0 << 21 | i1;
}
__device__ __forceinline__ SweepCounts sweep_unpack(uint64_t v) {
  return {(int32_t)(v >> 21 & 0x1FFFFF), (int32_t)(v & 0x1FFFFF), (int32_t)(v >> 42)};
}

// Where the counts go: the triangle or the full square of n samples.
struct SweepOut {
  int64_t n;
  int32_t* counts;
  double* dist;
  int32_t square;
  __device__ bool none(int64_t gi0, int64_t gj0, int cols) const {
    return gi0 >= n || gj0 >= n || gj0 + cols <= gi0;
  }
  __device__ bool has(int64_t gi, int64_t gj) const { return gi < n && gj < n && gj >= gi; }
  __device__ bool mirrored() const { return square != 0; }
  __device__ void store(int64_t p, uint64_t v) const {
    const SweepCounts c = sweep_unpack(v);
    reinterpret_cast<int4*>(counts)[p] = make_int4(c.i0, c.i1, c.n - c.i0 - c.i1, c.n);
    if (dist) dist[p] = ibs_dist(c.i0, c.i1, c.n);
  }
  __device__ void put(int64_t gi, int64_t gj, uint64_t v) const {
    store(square ? gi * n + gj : tri_index(gi, gj, n), v);
  }
  __device__ void put_mirror(int64_t gi, int64_t gj, uint64_t v) const { store(gj * n + gi, v); }
};

// Serving: counts only, step row r through its own output row [n_cols][4].
struct SweepRows {
  int32_t* const* row_out;
  int64_t n_rows, n_cols;
  __device__ bool none(int64_t gi0, int64_t gj0, int) const { return gi0 >= n_rows || gj0 >= n_cols; }
  __device__ bool has(int64_t gi, int64_t gj) const { return gi < n_rows && gj < n_cols; }
  __device__ bool mirrored() const { return false; }
  __device__ void put(int64_t gi, int64_t gj, uint64_t v) const {
    const SweepCounts c = sweep_unpack(v);
    reinterpret_cast<int4*>(row_out[gi])[gj] = make_int4(c.i0, c.i1, c.n - c.i0 - c.i1, c.n);
  }
  __device__ void put_mirror(int64_t, int64_t, uint64_t) const {}
};

// Write one piece of a tile, 32 rows from gi0 by 16 columns from gj0, from its
// three products: load(pr, v) sets v[j] to product pr of (row gi0 + lane, column
// gj0 + j).  The packed counts are transposed through `sm`, so that a half-warp
// stores 16 consecutive pairs of a row (256 bytes of counts) at a time; a
// square's mirror image is contiguous down the column as it is loaded.
template <class Out, class Load>
__device__ __forceinline__ void sweep_store(const Out& o, int64_t gi0, int64_t gj0, const Load& load, uint64_t* sm) {
  const int lane = threadIdx.x & 31;
  if (o.none(gi0, gj0, 16)) return;
  float vn[16], vu[16], vz[16];
  load(0, vn);
  load(1, vu);
  load(2, vz);
  __syncwarp();  // the warp's previous piece has been read
#pragma unroll
  for (int j = 0; j < 16; ++j) sm[lane * 17 + j] = sweep_pack(vn[j], vu[j], vz[j]);
  __syncwarp();
  const int64_t gj = gj0 + (lane & 15);
#pragma unroll 4
  for (int r = lane >> 4; r < 32; r += 2)
    if (o.has(gi0 + r, gj)) o.put(gi0 + r, gj, sm[r * 17 + (lane & 15)]);
  if (o.mirrored()) {
    const int64_t gi = gi0 + lane;
#pragma unroll 4
    for (int j = 0; j < 16; ++j)
      if (gj0 + j > gi && o.has(gi, gj0 + j)) o.put_mirror(gi, gj0 + j, sm[lane * 17 + j]);
  }
}

// ---------------------------------------------------------------------------
// The kernel.

// Views of one matrix's operand planes, boxes of 1, 2 and 3 half-blocks.
struct SweepMaps {
  CUtensorMap half1, half2, half3;
  __device__ const CUtensorMap* of(int w) const { return w == 3 ? &half3 : (w == 2 ? &half2 : &half1); }
};
static_assert(sizeof(SweepMaps) == kSweepMapsBytes, "the host sizes arrays of them");

// What a launch computes.  One matrix:
struct SweepOne {
  SweepMaps maps;
  SweepOut result;
  int32_t n_stages;
  __device__ const CUtensorMap* a(const SweepItem&) const { return &maps.half2; }
  __device__ const CUtensorMap* b(const SweepItem& it) const { return maps.of(it.w); }
  __device__ int stages(int) const { return n_stages; }
  __device__ SweepOut out(int) const { return result; }
};
// the subsets of a batch (SubsetDev::n_chunks counts ring stages here):
struct SweepBatch {
  const SweepMaps* maps;
  const SubsetDev* subs;
  __device__ const CUtensorMap* a(const SweepItem& it) const { return &maps[it.subset].half2; }
  __device__ const CUtensorMap* b(const SweepItem& it) const { return maps[it.subset].of(it.w); }
  __device__ int stages(int subset) const { return (int)subs[subset].n_chunks; }
  __device__ SweepOut out(int subset) const {
    return {subs[subset].n, subs[subset].out_counts, subs[subset].out_dist, 0};
  }
};
// the rows of a serving step against a panel.
struct SweepCross {
  SweepMaps maps;      // the panel's planes
  CUtensorMap rows;    // the step rows' planes, boxes of 2
  SweepRows result;
  int32_t n_stages;
  __device__ const CUtensorMap* a(const SweepItem&) const { return &rows; }
  __device__ const CUtensorMap* b(const SweepItem& it) const { return maps.of(it.w); }
  __device__ int stages(int) const { return n_stages; }
  __device__ SweepRows out(int) const { return result; }
};

struct SweepArgs {
  const SweepItem* items;
  const int32_t* first;  // items of cluster c: first[c] .. first[c + 1] - 1
  float* scratch;        // [CTA][3][384][128]: products of the CTA's whole item
  float* part;           // [slot][2][384][128]: products of split items
  int* status;
  unsigned long long wait_ns;
  SweepSync sync;
};

// Warps: 0 and 3 copies of A and of B, 1 and 2 MMAs (even CTA), 4..11 epilogue.
// Roles and barriers as in ibs_tc.cu's two-SM kernel: both CTAs' copies complete
// on the even CTA's `full`; its MMA warps commit each stage to both CTAs' `empty`
// and each finished product to both CTAs' `tfull`; the epilogue warps of both
// arrive on the even CTA's `tempty` once the product is read.  Every wait is
// bounded.
//
// An item is a tile and a range [q0, q1) of the 4 * stages ring stages of its
// sweeps.  A whole tile (slot < 0) keeps its products in the CTA's scratch and
// is written after its last sweep, while the next item's first sweep runs; a
// piece writes each product it has a part of to a slot of its own, which the
// finalisation adds up.
template <class W>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSwThreads, 1)
    sweep_kernel(const __grid_constant__ W work, const SweepArgs args) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full[kSwStages], empty[kSwStages], tfull, tempty, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t issued[2];  // ring stages this CTA's copy warps issued
  __shared__ int abort_flag;
  __shared__ int s_ok[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const uint32_t cid = cluster_index();
  int* status = args.status;
  const unsigned long long wait_ns = args.wait_ns;
  const int it0 = args.first[cid], it1 = args.first[cid + 1];
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSwStages; ++s) {
      mbar_init(&full[s], 1);  // the even CTA's: both CTAs' copies complete on it
      mbar_init(&empty[s], 2);  // both MMA warps' commits
    }
    mbar_init(&tfull, 2);
    mbar_init(&tempty, 2 * kSwEpiWarps);
    mbar_init(&drain, 2);
    mbar_fence_init();
    abort_flag = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (warp >= 4 && warp < 8) tmem_fill_unit_scales(tmem, warp - 4);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();  // both CTAs' barriers initialised and scale factors stored
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  wait_for_previous();

  // S stages of V V^T, S of U U^T, 2 S of Q R^T + R Q^T: the end of stage q's
  // product, or of the item
  auto product_end = [](int S, int q, int q1) { return min(q1, q < S ? S : (q < 2 * S ? 2 * S : 4 * S)); };

  if (warp == 0 || warp == 3) {
    // Copies: lane 0 of warp 0 streams the A operand, lane 0 of warp 3 the B
    // operand, one box per ring stage each.
    if (lane == 0) {
      const bool is_b = warp == 3;
      const uint32_t full0 = cluster_addr(&full[0], 0);  // the even CTA's ring barriers
      uint8_t* dst0 = ring + (is_b ? kSwABytes : 0);
      uint32_t g = 0, s = 0, ph = 1;  // stages issued, ring slot, parity of the slot's previous release
      int lag = args.sync.lag;
      bool stop = false;
      for (int e = it0; e < it1 && !stop; ++e) {
        const SweepItem it = args.items[e];
        const int h = is_b ? 2 * it.J + it.w * (int)rank : 2 * (it.I + (int)rank);
        const CUtensorMap* map = is_b ? work.b(it) : work.a(it);
        const int S = work.stages(it.subset);
        const uint32_t bytes = 2u * (uint32_t)(kSwABytes + kSwCols * 1024 * it.w);
        // lockstep: warp 0 announces every segment and holds back until the
        // whole wave has started the segment `lag` back (warp 3 follows
        // through the ring).  That only saves traffic: where the wave does not
        // come within a quarter of the bound that the other roles wait with
        // (another kernel holds an SM, as the clustering of a large matrix does
        // for seconds), the CTA goes on alone.
        int* ctr = !is_b && args.sync.seg > 0 && it.wave >= 0 ? args.sync.ctr + (int64_t)it.wave * args.sync.n_seg : nullptr;
        int left = 0, sg = 0;
        int q = it.q0;
        while (q < it.q1 && !stop) {
          // V V^T, then U U^T, then Q R^T and R Q^T in turn over the same markers
          const int pr = q < S ? 0 : (q < 2 * S ? 1 : 2), q0 = pr * S, end = product_end(S, q, it.q1);
          for (; q < end; ++q) {
            const int odd = (q - q0) & 1;
            const int plane = pr < 2 ? pr : (is_b ? 3 - odd : 2 + odd);
            const int col = (pr < 2 ? q - q0 : (q - q0) >> 1) * kSwCols;
            if (ctr != nullptr && left-- == 0) {
              left = args.sync.seg - 1;
              atomicAdd(ctr + sg, 1);
              if (sg >= lag && !wait_ready(ctr + sg - lag, 2 * (int)cluster_total(), wait_ns / 4)) lag = INT_MAX;
              ++sg;
            }
            if (g >= (uint32_t)kSwStages && !ring_wait(&empty[s], ph, wait_ns, &abort_flag)) {
              stop = true;
              break;
            }
            const uint32_t bar = full0 + s * 8u;
            if (!is_b && rank == 0) mbar_arrive_expect_tx(&full[s], bytes);
            tma_load_4d_pair(dst0 + s * kSwStageBytes, map, 0, h, col, plane, bar);
            ++g;
            if (++s == kSwStages) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
      }
      if (stop && *(volatile int*)&abort_flag == 0) {
        atomicExch(status, kDevTimeout);
        atomicExch(&abort_flag, 1);
      }
      // the last stages' releases (commits of the even CTA) have landed here
      for (uint32_t j = g > (uint32_t)kSwStages ? g - kSwStages : 0; j < g && !stop; ++j)
        if (!mbar_wait_bounded(&empty[j % kSwStages], (j / kSwStages) & 1u)) {
          atomicExch(status, kDevTimeout);
          atomicExch(&abort_flag, 1);
          break;
        }
      issued[is_b ? 1 : 0] = g;
    }
    __syncwarp();
  } else if ((warp == 1 || warp == 2) && rank == 0) {
    // Two MMA warps, each with its own half of the accumulator columns.  The
    // tensor core queues hardly more than the MMA it runs, so whatever a warp
    // does between two stages (commit, the next stage's wait) leaves it idle
    // unless another warp's MMAs follow: with one MMA warp, released through a
    // hardware barrier by a warp that waits on memory, a stage took 790 cycles
    // for 576 of MMAs (20,000 samples x 500,000 markers: 81.4 ms against 76.9;
    // 4,096 x 100,000: 1,074 us against 1,033).
    if (lane == 0) {
      uint32_t s = 0, ph = 0, p = 0;  // ring slot and its parity, products
      const uint32_t half = warp - 1, sf = tmem + kSfCol, ring0 = smem_addr(ring);
      bool ok = true;
      // `stages` stages of one product; W > 1: N = 64 W columns from column
      // 64 W half on; W = 1 has no halves, the first warp takes it all
      auto product = [&](auto width, int stages) {
        constexpr int w = decltype(width)::value;
        constexpr int kN = w == 3 ? 192 : 128;
        uint32_t acc = 0;  // the first K step overwrites
        for (int k = 0; k < stages; ++k) {
          if (!ring_wait(&full[s], ph, wait_ns, &abort_flag)) {
            ok = false;
            return;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st0 = ring0 + s * kSwStageBytes;
          const uint64_t a = sweep_desc(st0, 2048), b = sweep_desc(st0 + kSwABytes + half * (kN / 2 * 16), 1024 * w);
          if (w > 1 || half == 0) {
#pragma unroll
            for (int t = 0; t < kSwCols / 3; ++t) {
              umma_sweep<kN>(tmem + kN * half, a + t * (3 * 2048 / 16), b + t * (3 * 1024 * w / 16), acc, sf);
              acc = 1;
            }
          }
          umma_commit_both(&empty[s]);
          if (++s == kSwStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        umma_commit_both(&tfull);
      };
      for (int e = it0; e < it1 && ok; ++e) {
        const SweepItem it = args.items[e];
        const int S = work.stages(it.subset);
        for (int q = it.q0; q < it.q1 && ok; ++p) {
          const int end = product_end(S, q, it.q1);
          if (p > 0) ok = mbar_wait_cluster_bounded(&tempty, (p - 1) & 1u, wait_ns);
          if (!ok) break;
          if (it.w == 3)
            product(std::integral_constant<int, 3>{}, end - q);
          else if (it.w == 2)
            product(std::integral_constant<int, 2>{}, end - q);
          else
            product(std::integral_constant<int, 1>{}, end - q);
          q = end;
        }
      }
      if (!ok && *(volatile int*)&abort_flag == 0) {
        // nothing more is issued: the other roles of both CTAs stop at this
        // flag or come to the end of their own bounds
        atomicExch(status, kDevTimeout);
        atomicExch(&abort_flag, 1);
      }
      umma_commit_local2(&drain);
    }
    __syncwarp();
    const bool drained = mbar_wait_bounded(&drain, 0);
    if (lane == 0 && !drained) atomicExch(status, kDevTimeout);
  } else if (warp >= 4) {
    const int quarter = warp & 3, part = (warp - 4) >> 2, row = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t tempty_addr = cluster_addr(&tempty, 0);
    float* scratch = args.scratch + (size_t)(2 * cid + rank) * 3 * kSwHalfTile;
    uint64_t* sm = reinterpret_cast<uint64_t*>(ring + (size_t)kSwStages * kSwStageBytes + (warp - 4) * kSwTransBytes);
    uint32_t p = 0;
    bool stop = false;
    for (int e = it0; e < it1 && !stop; ++e) {
      const SweepItem it = args.items[e];
      const int S = work.stages(it.subset);
      int slot = it.slot;
      for (int q = it.q0; q < it.q1;) {
        const int pr = q < S ? 0 : (q < 2 * S ? 1 : 2);
        const int end = pr == 2 ? 4 * S : (pr + 1) * S;
        q = end < it.q1 ? end : it.q1;
        // one thread waits for the product and decides for all eight warps
        // (alternating slots: a warp that is late still reads its own decision)
        if (threadIdx.x == 128)
          s_ok[p & 1] = mbar_wait_bounded(&tfull, p & 1u, wait_ns) && *(volatile int*)&abort_flag == 0;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("bar.sync %0, %1;" ::"n"(kSwEpiBar), "n"(32 * kSwEpiWarps) : "memory");
        if (*(volatile int*)&s_ok[p & 1] == 0) {
          if (threadIdx.x == 128 && *(volatile int*)&abort_flag == 0) {
            atomicExch(status, kDevTimeout);
            atomicExch(&abort_flag, 1);
          }
          stop = true;
          break;
        }
        ++p;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float* dst = it.slot < 0 ? scratch + pr * kSwHalfTile : args.part + (size_t)(2 * slot + (int)rank) * kSwHalfTile;
        ++slot;
        // 32-column groups part, part + 2, ...; three in flight
        const int ng = 4 * it.w;
        for (int g0 = part; g0 < ng; g0 += 6) {
          uint32_t v[3][32];
#pragma unroll
          for (int u = 0; u < 3; ++u) tmem_ld32(lane_base + (g0 + 2 * u) * 32, v[u]);  // past ng: columns unused
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (g0 + 6 >= ng) {  // the last of this warp's columns are in registers: hand tensor memory back
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(tempty_addr);
          }
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            const int gr = g0 + 2 * u;
            if (gr < ng) {
              // w = 2 and 3: two MMAs of 64 w columns, each half of the even
              // CTA's B rows, then half of the odd CTA's
              const int r = gr % (2 * it.w), odd = r / it.w;
              const int c0 = it.w == 1 ? gr * 32 : odd * 64 * it.w + (gr / (2 * it.w) * it.w + r % it.w) * 32;
#pragma unroll
              for (int j = 0; j < 32; ++j) dst[(size_t)(c0 + j) * kTB + row] = __uint_as_float(v[u][j]);
            }
          }
        }
      }
      if (stop || it.slot >= 0) continue;
      // whole tile: every product is in the scratch; 32 x 16 pieces by warps
      asm volatile("bar.sync %0, %1;" ::"n"(kSwEpiBar), "n"(32 * kSwEpiWarps) : "memory");
      const auto out = work.out(it.subset);
      const int64_t gi0 = (int64_t)(it.I + (int)rank) * kTB + quarter * 32;
      for (int ct = part; ct < 8 * it.w; ct += 2) {
        const float* src = scratch + (size_t)ct * 16 * kTB + row;
        sweep_store(out, gi0, (int64_t)it.J * kTB + ct * 16,
                    [&](int pr, float (&v)[16]) {
#pragma unroll
                      for (int j = 0; j < 16; ++j) v[j] = __ldcg(src + pr * kSwHalfTile + (size_t)j * kTB);
                    },
                    sm);
      }
    }
  }
  let_next_start();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();  // both CTAs have issued their last copy and the even CTA's MMAs are drained
  if (rank == 0 && warp == 0) {
    // Every copy of either CTA completes on the even CTA's `full`.  After a
    // stop some issued stages were never consumed, so wait (bounded) for the
    // last ring's worth that either CTA issued before either CTA may exit.
    uint32_t p0 = 0, p1 = 0;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(p0) : "r"(cluster_addr(&issued[0], 1)) : "memory");
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(p1) : "r"(cluster_addr(&issued[1], 1)) : "memory");
    const uint32_t gmax = max(max(issued[0], issued[1]), max(p0, p1));
    for (uint32_t j = gmax > (uint32_t)kSwStages ? gmax - kSwStages : 0; j < gmax; ++j) {
      const bool ok = mbar_wait_bounded(&full[j % kSwStages], (j / kSwStages) & 1u);
      if (__any_sync(0xffffffffu, !ok)) {
        if (lane == 0) atomicExch(status, kDevTimeout);
        break;
      }
    }
  }
  __syncthreads();
  cluster_sync_all();  // no copy into either CTA and no arrival on either CTA's barriers is outstanding
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// Split tiles: the parts of each product added up and written.  Warp = one 32 x
// 16 piece of a tile, 32 loads of parts in flight per thread.
template <class W>
__global__ void __launch_bounds__(128) sweep_finalize_kernel(const SweepGroup* __restrict__ groups,
                                                             const float* __restrict__ part,
                                                             const __grid_constant__ W work) {
  __shared__ uint64_t sm[4][32 * 17];
  const SweepGroup gr = groups[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.y * 4 + warp;  // 2 CTAs x 4 row quarters x 24 column pieces
  const int ct = t % 24, quarter = (t / 24) & 3, rank = t / 96;
  wait_for_previous();
  if (ct >= 8 * gr.w) return;
  const float* src = part + (size_t)(2 * gr.slot + rank) * kSwHalfTile + (size_t)ct * 16 * kTB + quarter * 32 + lane;
  const int first[3] = {0, gr.pieces[0], gr.pieces[0] + gr.pieces[1]};
  sweep_store(work.out(gr.subset), (int64_t)(gr.I + rank) * kTB + quarter * 32, (int64_t)gr.J * kTB + ct * 16,
              [&](int pr, float (&v)[16]) {
                const float* p = src + (size_t)first[pr] * 2 * kSwHalfTile;
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = 0.0f;
#pragma unroll 2
                for (int k = 0; k < gr.pieces[pr]; ++k, p += 2 * kSwHalfTile)
#pragma unroll
                  for (int j = 0; j < 16; ++j) v[j] += __ldg(p + (size_t)j * kTB);  // whole numbers: exact
              },
              sm[warp]);
}

// Batched subsets, when they read a good part of the pool: the pool's rows
// [begin, end) regrouped by sample, words[c][sample] = the low and the high code
// bits of markers begin + 32 c ...  The gather below then reads 8 bytes per
// sample and column; out of the rows it reads single bytes of 32 lines, which
// took 1.8 ms of a 4 ms batch (24 subsets of 100 to 3,000 samples, 10,000 x
// 200,000 pool).  Warp = one column of 64 samples, transposed by shuffles;
// 512 neighbouring samples per CTA.  A fixed grid (the launch is in a graph and
// the window is known per call); HBM-bound: the pool read once and written once.
__device__ __forceinline__ void sweep_words(const SweepPool& p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_half = (p.n + 63) / 64, groups = (n_half + 7) / 8, total = p.cols * groups;
  for (int64_t i = blockIdx.x; i < total; i += gridDim.x) {
    const int64_t c = i / groups, h = (i % groups) * 8 + warp;
    if (h >= n_half) continue;
    uint32_t w[4];
    sweep_row64(p.packed, p.row_bytes, p.begin + c * 32 + lane, p.m, h * 16, w);
    uint32_t* out = p.words + ((size_t)c * p.n + (size_t)h * 64) * 2;
#pragma unroll
    for (int i4 = 0; i4 < 4; ++i4) {
      const uint32_t x = tc_transpose32(w[i4], lane);
      if (h * 64 + i4 * 16 + (lane >> 1) < p.n) out[i4 * 32 + lane] = x;
    }
  }
}

__global__ void __launch_bounds__(256) sweep_words_kernel(const SweepPool* __restrict__ pool) { sweep_words(*pool); }
__global__ void __launch_bounds__(256) panel_words_kernel(const SweepPool pool) { sweep_words(pool); }

// Batched subsets: sample sel[128 block + r] of the pool over 16 columns of the
// subset's window, thread r = sample r of the block; 16 bytes of each plane per
// column.  map[c] = {job, sample block, column group} of CTA c, in the order of
// the pool variant it starts at, so that subsets with overlapping windows share
// the pool through L2.  An index outside the pool is not read: the sample is
// all-missing and the status word reports it.  Without words the thread reads
// one byte of each of a column's 32 marker rows.
constexpr int kSwGatherCols = 16;
__device__ __forceinline__ void sweep_put_column(uint32_t H, uint32_t L, uint8_t* base, size_t plane) {
  const uint32_t V = H | ~L, P = H & ~L, Q = H & L, R = ~H & ~L;
  uint32_t wv[4], wu[4], wq[4], wr[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    wv[g] = nib8(V >> (8 * g)) << 1;
    wu[g] = wv[g] | (nib8(P >> (8 * g)) << 3);
    wq[g] = nib8(Q >> (8 * g)) << 1;
    wr[g] = nib8(R >> (8 * g)) << 1;
  }
  *reinterpret_cast<uint4*>(base) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
  *reinterpret_cast<uint4*>(base + plane) = make_uint4(wu[0], wu[1], wu[2], wu[3]);
  *reinterpret_cast<uint4*>(base + 2 * plane) = make_uint4(wq[0], wq[1], wq[2], wq[3]);
  *reinterpret_cast<uint4*>(base + 3 * plane) = make_uint4(wr[0], wr[1], wr[2], wr[3]);
}
__global__ void __launch_bounds__(kTB, 8) sweep_gather_kernel(const TcGatherJob* __restrict__ jobs,
                                                           const int4* __restrict__ map,
                                                           const SweepPool* __restrict__ pool, int* status) {
  const int4 e = map[blockIdx.x];
  const TcGatherJob& j = jobs[e.x];
  const int r = threadIdx.x;
  const int64_t s = (int64_t)e.y * kTB + r, nh = (j.n + 63) / 64, h = s >> 6;
  if (h >= nh) return;
  int64_t ps = -1;
  if (s < j.n) {
    ps = j.src.sel[s];
    if (ps < 0 || ps >= j.src.n_src) {
      atomicExch(status, 1);
      ps = -1;
    }
  }
  // (in registers: the stores below could alias the job)
  const int64_t row_bytes = j.src.row_bytes, nc = j.nc, m = j.m;
  uint8_t* const out = j.tc + (size_t)h * nc * 1024 + (size_t)(s & 63) * 16;
  const size_t plane = (size_t)nh * nc * 1024;
  const int64_t c0 = (int64_t)e.z * kSwGatherCols, c1 = min(nc, c0 + kSwGatherCols);
  const int64_t first = j.src.var_begin - pool->begin;
  if (pool->cols > 0 && ps >= 0) {
    // words of pool columns c + first / 32 and the next one, shifted; past the
    // last one the markers are outside the window
    const int64_t cols = pool->cols, stride = pool->n;
    const uint2* w = reinterpret_cast<const uint2*>(pool->words) + ps;
    const int sh = (int)(first & 31);
    int64_t pc = c0 + (first >> 5);
    const uint2 none = make_uint2(~0u, 0u);
    uint2 cur = pc < cols ? __ldg(w + pc * stride) : none;
#pragma unroll 4
    for (int64_t c = c0; c < c1; ++c, ++pc) {
      const uint2 next = pc + 1 < cols ? __ldg(w + (pc + 1) * stride) : none;
      uint32_t L = __funnelshift_r(cur.x, next.x, sh), H = __funnelshift_r(cur.y, next.y, sh);
      const int64_t kn = m - c * 32;  // markers of the column inside the window
      if (kn < 32) {
        const uint32_t in = kn > 0 ? (1u << kn) - 1u : 0u;
        H &= in;
        L |= ~in;
      }
      sweep_put_column(H, L, out + (size_t)c * 1024, plane);
      cur = next;
    }
    return;
  }
  const int sh = ps >= 0 ? 2 * (int)(ps & 3) : 0;
  const uint8_t* col = j.src.packed + j.src.var_begin * row_bytes + (ps >= 0 ? (ps >> 2) : 0);
#pragma unroll 1
  for (int64_t c = c0; c < c1; ++c) {
    const int64_t k0 = c * 32;
    const int kn = (int)(m - k0 < 32 ? m - k0 : 32);  // markers of the column inside the window
    uint32_t H = 0, L = ~0u;                              // all missing unless read
    if (ps >= 0 && kn > 0) {
      // the row stride is re-read in each column (an empty asm), or the
      // compiler keeps 32 row offsets in registers across columns and spills
      int64_t stride = row_bytes;
      asm volatile("" : "+l"(stride));
      const uint8_t* p = col + k0 * stride;
      uint32_t byte[32];
#pragma unroll
      for (int k = 0; k < 32; ++k, p += stride) byte[k] = k < kn ? __ldg(p) : 0x55u;
      H = 0;
      L = 0;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const uint32_t code = (byte[k] >> sh) & 3u;
        H |= (code >> 1) << k;
        L |= (code & 1u) << k;
      }
    }
    sweep_put_column(H, L, out + (size_t)c * 1024, plane);
  }
}

// Serving: rows of the requests' planes packed densely into the step's planes.
// CTA = (column, half-block); thread (row, plane).
__global__ void __launch_bounds__(256) sweep_gather_rows_kernel(const RowSrc* __restrict__ rows, int64_t n_rows,
                                                                int64_t n_cols, uint8_t* __restrict__ dst,
                                                                int64_t dst_half) {
  const int64_t c = blockIdx.x, h = blockIdx.y;
  const int r = threadIdx.x & 63, plane = threadIdx.x >> 6;
  const int64_t d = h * 64 + r;
  if (d >= n_rows) return;
  const RowSrc src = rows[d];
  const uint8_t* from = reinterpret_cast<const uint8_t*>(src.planes) +
                        (((size_t)plane * src.n_half + (src.row >> 6)) * n_cols + c) * 1024 + (src.row & 63) * 16;
  *reinterpret_cast<uint4*>(dst + (((size_t)plane * dst_half + h) * n_cols + c) * 1024 + r * 16) =
      *reinterpret_cast<const uint4*>(from);
}

// A view of the operand planes, a box `halves` half-blocks over kSwCols
// columns of one plane, landing as [column][half-block][1 KiB]; half-blocks
// past the last read as zeros.
bool encode_sweep_map(CUtensorMap* map, const void* planes, int64_t n_half, int64_t n_cols, int halves) {
  const EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {128, (cuuint64_t)n_half, (cuuint64_t)n_cols, 4};
  const cuuint64_t strides[3] = {(cuuint64_t)n_cols * 1024, 1024, (cuuint64_t)n_half * (cuuint64_t)n_cols * 1024};
  const cuuint32_t box[4] = {128, (cuuint32_t)halves, kSwCols, 1};
  const cuuint32_t elem[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<void*>(planes), dims, strides, box, elem,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool encode_sweep_maps(SweepMaps* m, const void* planes, int64_t n_half, int64_t n_cols) {
  return encode_sweep_map(&m->half1, planes, n_half, n_cols, 1) &&
         encode_sweep_map(&m->half2, planes, n_half, n_cols, 2) &&
         encode_sweep_map(&m->half3, planes, n_half, n_cols, 3);
}

// A tile before it is scheduled.
struct Tile {
  int I, J, w, subset, stages;
};

// The tiles of a triangle of n samples: two block rows by up to three block
// columns, in bands of 16 block rows, column by column in a band, so that the
// tiles in flight share operand blocks through L2.  The columns are grouped from
// the right edge, the same for every row, and the group that holds the
// diagonal starts at it.
void triangle_tiles(int64_t n, int stages, int subset, std::vector<Tile>& full, std::vector<Tile>& narrow) {
  const int T = (int)((n + kTB - 1) / kTB);
  constexpr int G = 16;
  for (int g0 = 0; g0 < T; g0 += G)
    for (int end = (T - g0 - 1) % 3 + 1 + g0; end <= T; end += 3)  // column groups end at T, T - 3, ...
      for (int I = g0; I < std::min(T, g0 + G) && I < end; I += 2) {
        const int J = std::max(I, end - 3);
        (end - J == 3 ? full : narrow).push_back({I, J, end - J, subset, stages});
      }
}

// Cost of a tile's ring stage in cycles: about 620 at full width with the operands
// in L2 (715 in a long lockstep wave), the fixed cost of a stage for the narrow
// tiles.
double stage_cost(int w) { return w == 3 ? 620.0 : (w == 2 ? 520.0 : 500.0); }
double tile_cost(const Tile& t) { return stage_cost(t.w) * 4 * t.stages; }

SweepItem whole_item(const Tile& t, int wave) {
  SweepItem it{};
  it.I = t.I;
  it.J = t.J;
  it.w = t.w;
  it.subset = t.subset;
  it.q1 = 4 * t.stages;
  it.slot = -1;
  it.wave = wave;
  return it;
}

constexpr int kPartsPerCluster = 6;

// Lay the tiles of `rest` end to end and cut them so that every cluster's load
// ends at the same time: each takes the next stretch, a few pieces of
// neighbouring tiles.  A stretch has at least a few stages (a piece costs about
// kMin stages of its own: pipeline fill, read-back, a part to add up) or a tile,
// so a small problem leaves clusters idle.  A tile that is not cut goes to parts
// too, as far as there are slots: two SMs take about 110 us to write the 256 x 384
// pairs of a whole tile, the sums' grid has all of them.  With few markers that
// is all there is: 300 x 50 42 us and 106 with whole tiles, 1,000 x 300 44 and 104,
// 3,000 x 1,000 77 and 297 (the last share held 80 of its 900 stages).
void cut_rest(const std::vector<Tile>& rest, std::vector<std::vector<SweepItem>>& own, std::vector<double>& load,
              SweepPlan& pl) {
  const int C = (int)own.size(), R = (int)rest.size();
  constexpr double kMin = 8 * 620.0;
  const bool parts = 3 * R + C <= sweep_max_slots(C);  // a cut adds at most one slot to its tile's three
  double total = 0;
  for (const Tile& t : rest) total += tile_cost(t);
  // the clusters that take part, the least loaded first, and the common end
  std::vector<int> by((size_t)C);
  for (int c = 0; c < C; ++c) by[(size_t)c] = c;
  std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return load[(size_t)a] < load[(size_t)b]; });
  int shares = 0;
  double held = 0, end = 0;
  for (int k = 1; k <= C; ++k) {
    held += load[(size_t)by[(size_t)k - 1]];
    const double e = (held + total) / k;  // if k clusters share the rest
    if (k > std::max(1, R) && e - load[(size_t)by[(size_t)k - 1]] < kMin) break;
    shares = k;
    end = e;
  }
  std::sort(by.begin(), by.begin() + shares);  // in order, so that neighbours work on neighbouring tiles
  int share = 0;
  double left = total;
  auto room = [&] { return end - load[(size_t)by[(size_t)share]]; };
  // (the end of those that are left, anew: what the rules on slivers gave or took
  // would otherwise all fall to the last one)
  auto next_share = [&] {
    ++share;
    end = left;
    for (int k = share; k < shares; ++k) end += load[(size_t)by[(size_t)k]];
    end /= shares - share;
  };
  for (const Tile& t : rest) {
    const int S = t.stages;
    const double cost = stage_cost(t.w);
    SweepGroup gr{};
    gr.I = t.I;
    gr.J = t.J;
    gr.w = t.w;
    gr.subset = t.subset;
    gr.slot = pl.slots;
    int q = 0;
    while (q < 4 * S) {
      const bool last = share == shares - 1;
      int k = last ? 4 * S - q : (int)std::max(0.0, std::min((double)(4 * S - q), room() / cost + 0.5));
      if (4 * S - q - k > 0 && 4 * S - q - k < 3) k = 4 * S - q;  // no sliver left behind
      if (k < 3 && k < 4 * S - q) {                               // nor one begun
        next_share();
        continue;
      }
      SweepItem it = whole_item(t, -1);
      it.q0 = q;
      it.q1 = q + k;
      if (parts || q != 0 || k != 4 * S) {
        it.slot = pl.slots;
        for (int pr = 0; pr < 3; ++pr) {
          const int a = pr == 0 ? 0 : pr * S, b = pr == 2 ? 4 * S : (pr + 1) * S;
          if (it.q0 < b && it.q1 > a) {
            ++gr.pieces[pr];
            ++pl.slots;
          }
        }
      }
      own[(size_t)by[(size_t)share]].push_back(it);
      load[(size_t)by[(size_t)share]] += cost * k;
      left -= cost * k;
      q += k;
      if (!last && room() < 0.5 * cost) next_share();
    }
    if (gr.pieces[0] + gr.pieces[1] + gr.pieces[2] > 0) pl.groups.push_back(gr);
  }
}

// The same in rounds: every tile of `rest` (one subset) is cut into 4 h equal
// pieces, h each of V V^T and U U^T and 2 h of the third product, and the
// clusters take the pieces in turn, all tiles' first pieces, then all second
// ones: the tiles of a round run over the same markers and share operand
// blocks through L2, which cut_rest's shares, each at a place of its own, do
// not.  The cheaper of the two by a model in cycles: 620 a stage, 4 stages to
// fill a piece's pipeline, 160 to write and add up a part; cut_rest's shares at
// least the time of their operands, 3.4 KB a cycle from HBM or, where the
// `operands` stay in L2, 5.7.  False where that is cut_rest.  Measured, rounds
// against shares: 1,501 samples x 30,011 markers 101 us and 111, 2,500 x 100,000
// 507 and 755, the square of 3,001 x 60,000 404 and 587, 6,000 x 200,000 3.46 ms
// and 3.91, 20 served requests of 3,003 rows 8.9 and 11.8.
bool cut_rounds(const std::vector<Tile>& rest, std::vector<std::vector<SweepItem>>& own, size_t operands,
                SweepPlan& pl) {
  const int64_t C = (int64_t)own.size(), R = (int64_t)rest.size();
  if (R < 4) return false;
  const int S = rest[0].stages;
  constexpr double kFill = 4, kPart = 160, kHbm = 3400, kL2 = 5700;
  constexpr size_t kL2Bytes = (size_t)129 << 20;
  double even = 0, bytes = 0;
  for (const Tile& t : rest) {
    even += tile_cost(t) / (double)C;
    bytes += 8.0 * t.stages * (kSwABytes + t.w * (kSwBBytes / 3));
  }
  double best = std::max(even, bytes / (operands > kL2Bytes ? kHbm : kL2)) + kPart * (double)(C + 2 * R);
  int h = 0;
  for (int k = 1; k <= 8 && S >= 8 * k && 4 * k * R <= kPartsPerCluster * C; ++k) {
    const double cost = (double)((4 * k * R + C - 1) / C) * ((double)S / k + kFill) * stage_cost(3) + kPart * (double)(4 * k * R);
    if (cost < best) {
      best = cost;
      h = k;
    }
  }
  if (h == 0) return false;
  for (int64_t t = 0; t < R; ++t) {
    SweepGroup gr{};
    gr.I = rest[(size_t)t].I;
    gr.J = rest[(size_t)t].J;
    gr.w = rest[(size_t)t].w;
    gr.subset = rest[(size_t)t].subset;
    gr.slot = pl.slots + (int)(4 * h * t);
    gr.pieces[0] = gr.pieces[1] = h;
    gr.pieces[2] = 2 * h;
    pl.groups.push_back(gr);
  }
  for (int k = 0; k < 4 * h; ++k)
    for (int64_t t = 0; t < R; ++t) {
      SweepItem it = whole_item(rest[(size_t)t], -1);
      it.q0 = (int)((int64_t)S * k / h);
      it.q1 = (int)((int64_t)S * (k + 1) / h);
      it.slot = pl.slots + (int)(4 * h * t) + k;
      own[(size_t)((k * R + t) % C)].push_back(it);
    }
  pl.slots += (int)(4 * h * R);
  return true;
}

// The clusters' lists, one after the other.
void lay_out(const std::vector<std::vector<SweepItem>>& own, SweepPlan& pl) {
  const int C = (int)own.size();
  pl.first.assign((size_t)C + 1, 0);
  for (int c = 0; c < C; ++c) {
    for (const SweepItem& it : own[(size_t)c]) {
      if (it.slot < 0) pl.scratch = true;
      pl.items.push_back(it);
    }
    pl.first[(size_t)c + 1] = (int32_t)pl.items.size();
  }
  // clusters without work are not launched
  pl.clusters = C;
  while (pl.clusters > 1 && pl.first[(size_t)pl.clusters - 1] == (int32_t)pl.items.size()) --pl.clusters;
}

// One matrix or one step: the full-width tiles run whole, one per cluster and
// wave, as many full waves as there are; the last partial wave and the
// narrower tiles are cut into pieces, in rounds or in equal shares.
SweepPlan schedule(std::vector<Tile>& full, const std::vector<Tile>& narrow, int clusters, size_t operands) {
  SweepPlan pl;
  const size_t C = (size_t)std::max(1, clusters), whole = full.size() / C * C;
  std::vector<std::vector<SweepItem>> own(C);
  std::vector<double> load(C, 0.0);
  for (size_t t = 0; t < whole; ++t) {
    own[t % C].push_back(whole_item(full[t], (int)(t / C)));
    load[t % C] += tile_cost(full[t]);
    pl.wave_stages = std::max(pl.wave_stages, 4 * full[t].stages);
  }
  pl.waves = (int)(whole / C);
  std::vector<Tile> rest(full.begin() + (long)whole, full.end());
  rest.insert(rest.end(), narrow.begin(), narrow.end());
  if (!cut_rounds(rest, own, operands, pl)) cut_rest(rest, own, load, pl);
  lay_out(own, pl);
  return pl;
}

template <class W>
cudaError_t launch_sweep_w(const W& work, const SweepLaunch& l, cudaStream_t st) {
  // function attributes are per device: set before every launch
  cudaError_t e = cudaFuncSetAttribute(sweep_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSwSmem);
  if (e != cudaSuccess) return e;
  const SweepArgs args{l.items, l.first, l.scratch, l.part, l.status, l.wait_ns, l.sync};
  cudaLaunchAttribute early = {};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * l.clusters));
  cfg.blockDim = dim3(kSwThreads);
  cfg.dynamicSmemBytes = kSwSmem;
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  if ((e = cudaLaunchKernelEx(&cfg, sweep_kernel<W>, work, args)) != cudaSuccess || l.n_groups <= 0) return e;
  if (l.between) {
    e = cudaEventRecord(l.between, st);
    if (e != cudaSuccess) return e;
  }
  cfg.gridDim = dim3((unsigned)l.n_groups, 48);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = 0;
  return cudaLaunchKernelEx(&cfg, sweep_finalize_kernel<W>, l.groups, l.part, work);
}

}  // namespace

int sweep_stages(int64_t m) { return (int)((m + kSwMarkers - 1) / kSwMarkers); }
int64_t sweep_cols(int64_t m) { return (int64_t)sweep_stages(m) * kSwCols; }

size_t sweep_planes_bytes(int64_t n, int64_t m) { return (size_t)((n + 63) / 64) * (size_t)sweep_cols(m) * 4096; }

size_t sweep_scratch_bytes(int clusters) { return (size_t)clusters * 2 * 3 * kSwHalfTile * sizeof(float); }
size_t sweep_slot_bytes() { return 2 * kSwHalfTile * sizeof(float); }
int sweep_max_slots(int clusters) { return kPartsPerCluster * std::max(1, clusters); }

// Lockstep of `waves` waves of whole tiles of at most `stages` ring stages, by
// the two-SM kernels' setting {chunks of 64 markers, lag}; off: no counters.
SweepSync sweep_sync(int waves, int stages, int2 ss) {
  SweepSync s;
  if (ss.x <= 0 || waves < 1) return s;
  s.seg = std::max(1, ss.x * 64 / kSwMarkers);
  s.lag = ss.y;
  s.n_seg = (stages + s.seg - 1) / s.seg;
  return s;
}

cudaError_t launch_sweep_planes(const uint8_t* packed, int64_t n, int64_t m, uint8_t* planes, cudaStream_t st) {
  const int64_t nh = (n + 63) / 64, nc = sweep_cols(m);
  if (nc > 2147483647LL || (nh + 7) / 8 > 65535) return cudaErrorInvalidValue;
  sweep_planes_kernel<<<dim3((unsigned)nc, (unsigned)((nh + 7) / 8)), 256, 0, st>>>(packed, (n + 3) / 4, n, m, planes,
                                                                                    nh, nc);
  return cudaGetLastError();
}

int64_t sweep_gather_ctas(int64_t n, int64_t n_cols) {
  return (n + kTB - 1) / kTB * ((n_cols + kSwGatherCols - 1) / kSwGatherCols);
}
int sweep_gather_cols() { return kSwGatherCols; }

// (ungraphed: a serving panel's words)
cudaError_t launch_sweep_words(const SweepPool& pool, int num_sms, cudaStream_t st) {
  panel_words_kernel<<<8 * num_sms, 256, 0, st>>>(pool);
  return cudaGetLastError();
}

// Regrouping costs about 0.12 ps per genotype of the pool's rows in use and
// saves 0.8 ps per gathered genotype.
bool sweep_words_pay(int64_t pool_genotypes, int64_t gathered) { return gathered >= pool_genotypes / 4; }

cudaError_t launch_sweep_gather(const TcGatherJob* jobs, const int4* map, int64_t ctas, const SweepPool* pool,
                                int num_sms, int* status, cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  if (ctas > 2147483647LL) return cudaErrorInvalidValue;
  sweep_words_kernel<<<8 * num_sms, 256, 0, st>>>(pool);
  if (cudaError_t e = cudaGetLastError()) return e;
  sweep_gather_kernel<<<(unsigned)ctas, kTB, 0, st>>>(jobs, map, pool, status);
  return cudaGetLastError();
}

cudaError_t launch_sweep_gather_rows(const RowSrc* rows, int64_t n_rows, int64_t n_cols, uint8_t* dst,
                                     int64_t dst_half, cudaStream_t st) {
  if (n_rows <= 0) return cudaSuccess;
  sweep_gather_rows_kernel<<<dim3((unsigned)n_cols, (unsigned)((n_rows + 63) / 64)), 256, 0, st>>>(rows, n_rows, n_cols,
                                                                                                 dst, dst_half);
  return cudaGetLastError();
}

// Clusters of two that fit at once, counted once per device ordinal.
int sweep_clusters() {
  constexpr int kDevs = 64;
  static std::atomic<int> cache[kDevs];  // 0 = not yet counted, else count + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) {
    cudaGetLastError();
    return 0;
  }
  if (const int c = cache[dev].load(std::memory_order_acquire)) return c - 1;
  int n = 0, sms = 0;
  auto kern = sweep_kernel<SweepOne>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSwSmem) == cudaSuccess &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::max(2, sms & ~1));
    cfg.blockDim = dim3(kSwThreads);
    cfg.dynamicSmemBytes = kSwSmem;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) n = 0;
  }
  cudaGetLastError();
  cache[dev].store(n + 1, std::memory_order_release);
  return n;
}

// E2M1 form; a tile's counts below 2^21 (exact FP32 sums, and their packing in
// sweep_store); the tensor map's coordinates.
bool sweep_usable(int64_t n, int64_t m) {
  if (m >= ((int64_t)1 << 21) || (n + 63) / 64 > 65535 * 8) return false;
  return encode_tiled_fn() != nullptr && sweep_clusters() > 0;
}

SweepPlan sweep_plan(int64_t n, int64_t m, int clusters) {
  std::vector<Tile> full, narrow;
  triangle_tiles(n, sweep_stages(m), 0, full, narrow);
  return schedule(full, narrow, clusters, sweep_planes_bytes(n, m));
}

// Batched subsets, by decreasing marker count.  First the whole waves of every
// subset that has any, one tile per cluster and in lockstep as for one matrix;
// then the other tiles, each in turn to the least loaded cluster, so that a
// subset's tiles run at about the same time and share some of its planes through
// L2 (in shares of tiles laid end to end the clusters ran all subsets at once,
// from HBM: 3.8 ms for 24 subsets of a 10,000 x 200,000 pool); the last tiles,
// about one per cluster, are cut to even out the end.  64 subsets of up to 8,000
// samples and 200,000 markers: 79 ms against 125 without the waves.
SweepPlan sweep_plan_batch(const std::vector<std::pair<int64_t, int64_t>>& shapes, int clusters) {
  std::vector<size_t> order(shapes.size());
  for (size_t k = 0; k < order.size(); ++k) order[k] = k;
  std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t b) { return shapes[a].second > shapes[b].second; });
  SweepPlan pl;
  const size_t C = (size_t)std::max(1, clusters);
  std::vector<std::vector<SweepItem>> own(C);
  std::vector<double> load(C, 0.0);
  std::vector<Tile> all;
  for (size_t k : order) {
    std::vector<Tile> full, narrow;
    triangle_tiles(shapes[k].first, sweep_stages(shapes[k].second), (int)k, full, narrow);
    const size_t whole = full.size() / C * C;
    for (size_t t = 0; t < whole; ++t) {
      own[t % C].push_back(whole_item(full[t], pl.waves + (int)(t / C)));
      load[t % C] += tile_cost(full[t]);
      pl.wave_stages = std::max(pl.wave_stages, 4 * full[t].stages);
    }
    pl.waves += (int)(whole / C);
    all.insert(all.end(), full.begin() + (long)whole, full.end());
    all.insert(all.end(), narrow.begin(), narrow.end());
  }
  const size_t lead = all.size() > C ? all.size() - C : 0;
  for (size_t t = 0; t < lead; ++t) {
    const size_t c = (size_t)(std::min_element(load.begin(), load.end()) - load.begin());
    own[c].push_back(whole_item(all[t], -1));
    load[c] += tile_cost(all[t]);
  }
  cut_rest(std::vector<Tile>(all.begin() + (long)lead, all.end()), own, load, pl);
  lay_out(own, pl);
  return pl;
}

// Panel blocks of a serving step of row_blocks blocks, of the `left` that the
// request furthest from its end still needs: one step where the rows are one or
// two blocks and the panel up to 16 blocks per cluster (155,000 samples), so that
// a lone request takes one; else about 8 blocks per cluster and row pair, short
// enough for new requests to join soon.  Steps over the same rows are of even
// length, in whole tiles (three blocks) up to the last.  Measured, one request
// against 100,000 samples x 200,000 markers: 17 to 256 rows 6.0 to 6.4 ms (6.0 to
// 6.3 on the unbatched path), 9.2 to 9.6 in two steps of 608 blocks of the 782; 20
// requests of 3,003 rows in all against 20,000 x 100,000: 7.3 ms, 7.5 with 5
// blocks per cluster and row pair, 7.2 to 7.4 with 14, 8.6 with lengths that are
// neither whole tiles nor bounded by what is left.
int64_t sweep_step_blocks(int64_t panel_blocks, int64_t row_blocks, int64_t left, int clusters) {
  const int64_t pairs = std::max<int64_t>(1, (row_blocks + 1) / 2), C = std::max(1, clusters);
  const int64_t most = pairs == 1 ? 16 * C : std::max((8 * C + pairs - 1) / pairs, (panel_blocks + 31) / 32);
  const int64_t steps = std::max<int64_t>(1, (left + most - 1) / most);
  return std::min(left, ((left + steps - 1) / steps + 2) / 3 * 3);
}

// Row pairs over two ranges of block columns [col0, col1) (the second may be
// empty): columns in groups of three, the row pairs of a group together.
SweepPlan sweep_plan_cross(int64_t row_blocks, const int64_t (&cols)[2][2], int64_t m, int clusters) {
  std::vector<Tile> full, narrow;
  const int S = sweep_stages(m);
  const int64_t blocks = cols[0][1] - cols[0][0] + cols[1][1] - cols[1][0];
  for (const auto& r : cols)
    for (int64_t J = r[0]; J < r[1]; J += 3) {
      const int w = (int)std::min<int64_t>(3, r[1] - J);
      for (int64_t I = 0; I < row_blocks; I += 2) (w == 3 ? full : narrow).push_back({(int)I, (int)J, w, 0, S});
    }
  return schedule(full, narrow, clusters, sweep_planes_bytes(kTB * (row_blocks + blocks), m));
}

bool sweep_encode_maps(void* maps, const void* planes, int64_t n, int64_t m) {
  return encode_sweep_maps(static_cast<SweepMaps*>(maps), planes, (n + 63) / 64, sweep_cols(m));
}

cudaError_t launch_sweep_one(const uint8_t* planes, int64_t n, int64_t m, int32_t* counts, double* dist, bool square,
                             const SweepLaunch& l, cudaStream_t st) {
  SweepOne w{};
  if (!encode_sweep_maps(&w.maps, planes, (n + 63) / 64, sweep_cols(m))) return cudaErrorInvalidValue;
  w.result = SweepOut{n, counts, dist, square ? 1 : 0};
  w.n_stages = sweep_stages(m);
  return launch_sweep_w(w, l, st);
}

cudaError_t launch_sweep_batch(const void* maps_dev, const SubsetDev* subs, const SweepLaunch& l, cudaStream_t st) {
  return launch_sweep_w(SweepBatch{static_cast<const SweepMaps*>(maps_dev), subs}, l, st);
}

cudaError_t launch_sweep_cross(const uint8_t* row_planes, int64_t row_half, const uint8_t* panel, int64_t n_panel,
                               int64_t m, int32_t* const* row_out, int64_t n_rows, const SweepLaunch& l,
                               cudaStream_t st) {
  SweepCross w{};
  if (!encode_sweep_maps(&w.maps, panel, (n_panel + 63) / 64, sweep_cols(m)) ||
      !encode_sweep_map(&w.rows, row_planes, row_half, sweep_cols(m), 2))
    return cudaErrorInvalidValue;
  w.result = SweepRows{row_out, n_rows, n_panel};
  w.n_stages = sweep_stages(m);
  return launch_sweep_w(w, l, st);
}

}  // namespace ibs

// Serving engine: a resident reference panel and continuous batching of
// query requests.
//
// The panel's planes stay on the device: operand planes of the tensor-core
// form (128-sample blocks), or bit planes of the POPC kernels (64-sample
// blocks), whichever the context's pair kernel is.  A host thread owns a CUDA
// stream and runs steps.  A step packs the query rows of EVERY admitted
// request densely into query blocks (a gather kernel copies each row's planes,
// and every row keeps its own output pointer) and runs them against a range
// of panel blocks.  Each panel block is therefore read once per step
// however many requests are in flight, and the items of a step are ordered
// panel-block-major so the CTAs sharing a panel block run together and hit it
// in L2.  The step length adapts to the load: with few rows in flight one step
// covers the whole panel, with many it covers about 16 waves of tiles so that
// new requests can join between steps.  A request joins at the current panel
// position and is done once it has seen every panel block; then its top-k
// kernel runs and its outputs are copied back.  Admission is FIFO, bounded by
// a row-slot limit and by a memory budget (free device memory at panel load,
// and the context's workspace limit).  Request buffers come from the
// stream-ordered memory pool, so freeing them never synchronises the device.
// At most two steps are in flight, so admission and completion are handled
// between steps while the GPU stays busy.
//
// E2M1 without a workspace limit: steps run on the sweep kernel (ibs_sweep.cu),
// over its own planes; a step of few rows (few_rows_pay) runs on the integer pipe
// over the panel's code bits (ibs_rows.cu), a second, small copy of the panel.
// Otherwise a tensor-core step with two or more query blocks runs on the two-SM
// kernel (items of two query blocks x one panel block; the faster kernel for
// panels of at least 1,024 chunks), a step of one query block on the one-SM
// kernel.  The step length is rounded so that its last wave of items is as
// full as possible.  The dense query planes are gathered again only when the
// set of admitted requests changed.  Counts bound for host memory leave the
// device step by step on a second stream (the panel columns each step wrote),
// so those copies overlap the following steps instead of trailing them.  The
// top-k of all requests that finish in a step runs as one launch.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <new>
#include <shared_mutex>
#include <thread>
#include <unordered_map>

#include "ibs_ctx.h"
#include "ibs_device.cuh"

namespace ibs {

namespace {

constexpr int kMaxQuery = 4096;     // rows per request
constexpr int kMaxK = 64;           // top-k limit of the kernel
constexpr int64_t kMaxRows = 4096;  // query rows admitted at once (slot limit)
constexpr int64_t kStepWaves = 16;  // a step aims at this many waves of (query block, panel block) tiles
constexpr int64_t kStepWavesTc = 8; // ... of the tensor-core form without the sweep kernel (a request of one query
                                    // block then takes one step over a 100,000-sample panel; two steps cost it
                                    // about 3 ms); with it: sweep_step_blocks
constexpr int64_t kMinStepDiv = 32; // ... and covers at least 1/32 of the panel
constexpr size_t kMemMargin = (size_t)1 << 30;
// Samples of this size go to the device from ibs_query, smaller ones by way of host
// memory: their copy to the device takes the caller 30 us, and a burst of them came
// in one by one, each in a step of its own.  20 requests of 1 to 16 rows against 38,314
// x 13,313: 1.6 ms with all sent to the device, 0.93 with 256 KiB (0.89 before any
// was); 1 to 512 rows (3,003 in all) against 20,000 x 100,000: 7.4 ms, 6.8 with 256
// KiB, 6.9 with 1 MiB.
constexpr size_t kDirectBytes = (size_t)256 << 10;
constexpr int64_t kTcBlock = 128;          // samples per tensor-core block
constexpr size_t kTcChunkBytes = 16384;    // one (block, chunk) of operand planes

enum class RState { Pending, Active, Finishing, Done };

struct Request {
  uint64_t id = 0;
  int64_t q = 0;
  int k = 0;
  int32_t* user_counts = nullptr;
  int32_t* user_idx = nullptr;
  double* user_dist = nullptr;
  bool counts_on_dev = false, topk_on_dev = false;
  std::vector<uint8_t> host_packed;
  DevBuf packed, planes, counts, tidx, tdist;
  size_t reserved = 0;
  bool planes_built = false;
  int32_t* map_idx = nullptr;  // pinned top-k outputs as the device sees them
  double* map_dist = nullptr;
  bool topk_direct = false;    // written there by the kernel
  bool early = false;     // took its memory with its place in the queue
  bool arriving = false;  // in the queue, its samples still on their way
  int64_t blocks_done = 0;  // panel blocks processed since admission
  cudaEvent_t done_ev = nullptr;  // recorded on the engine's copy stream after the request's last output
  ibs_status status = IBS_OK;
  RState state = RState::Pending;
};

enum class PtrKind { Device, PinnedHost, Pageable };

PtrKind ptr_kind(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return PtrKind::Pageable;
  }
  if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return PtrKind::Device;
  if (a.type == cudaMemoryTypeHost) return PtrKind::PinnedHost;
  return PtrKind::Pageable;
}

// The device's address of pinned host memory aligned for a kernel's stores of
// elements of `size` bytes, or null (a copy takes any alignment).
void* mapped(void* p, size_t size) {
  if (reinterpret_cast<uintptr_t>(p) % size != 0) return nullptr;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return a.type == cudaMemoryTypeHost ? a.devicePointer : nullptr;
}

}  // namespace

// Planes geometry in the units of the engine's pair kernel.
struct Geo {
  int64_t blocks, chunks;  // sample blocks, marker chunks
  size_t bytes;            // plane bytes
};

class ServeEngine {
 public:
  ibs_ctx* ctx;
  PlaneGeom pg;          // panel sizes (pg.n, pg.m) and, for POPC, the bit-plane geometry
  bool tc = false;       // tensor-core pair kernel (else POPC)
  int fmt = 0;           // tensor-core operand format
  int64_t blk = kSB;     // samples per block: 128 (tensor core) or 64 (POPC)
  Geo pgeo{};            // the panel's geometry
  DevBuf panel_planes, counter;
  cudaStream_t stream = nullptr;
  cudaStream_t in = nullptr;  // ibs_query's copies
  std::shared_mutex in_mu;    // shared by ibs_query while it brings a request in; shutdown waits for it
  int64_t early_rows = 0;     // rows of the unfinished early requests (mu)
  std::thread worker;
  std::mutex mu;
  std::condition_variable cv_work, cv_done;
  bool stop = false;
  std::deque<std::shared_ptr<Request>> pending;
  std::vector<std::shared_ptr<Request>> active, finishing;
  std::unordered_map<uint64_t, std::shared_ptr<Request>> all;
  std::atomic<uint64_t> next_id{1};
  ibs_serve_stats stats{};
  int64_t cursor = 0;  // first panel block of the next step
  int grid_ctas = 0;   // persistent cross-kernel CTAs (SMs x 2)
  bool sweep = false;  // the sweep kernel for every step (E2M1)
  DevBuf sweep_scratch, sweep_part;  // the steps'
  DevBuf sync_scratch, sync_part;    // the unbatched path's, one call's kernels at a time
  std::mutex sync_mu;                // from the wait for the last call's kernels to the event after this one's
  cudaEvent_t sync_ev = nullptr;     // after the last call's kernels
  DevBuf panel_words, few_words;     // sweep: the panel's code bits by sample, for steps of few rows; the rows'
  std::mutex words_mu;               // panel_words in use or given back
  bool pair = false;   // two-SM kernel for steps of two or more query blocks
  int clusters = 0;    // its clusters of two CTAs
  DevBuf sync_ctr;     // the two-SM kernel's K-lockstep counters of a step
  DevBuf topk_dev[2];  // row lists of a step's finishing requests (one top-k launch)
  TopkRow* topk_host[2] = {nullptr, nullptr};
  cudaStream_t side = nullptr;  // device -> host copies of finished columns and top-k lists
  cudaEvent_t kern_ev[2] = {nullptr, nullptr}, fin_ev[2] = {nullptr, nullptr};
  uint64_t set_version = 1, gathered_version = 0;  // the admitted set; the set the step planes hold
  size_t fixed_bytes = 0;  // panel planes + step buffers
  // double-buffered item arrays (one-SM CrossItem or two-SM PairItem)
  DevBuf items_dev[2];
  uint8_t* items_host[2] = {nullptr, nullptr};
  size_t items_cap = 0;
  cudaEvent_t step_ev[2] = {nullptr, nullptr};
  int64_t step_no = 0;
  int failing_steps = 0;  // the next steps to fail (mu; serve_fail_steps)
  DevBuf step_planes, rows_dev[2], outs_dev[2];
  std::mutex budget_mu;
  size_t pool_budget = 0;  // bytes the requests may hold together
  size_t pool_bytes = 0;   // bytes they hold now
  RowSrc* rows_host[2] = {nullptr, nullptr};
  int32_t** outs_host[2] = {nullptr, nullptr};

  explicit ServeEngine(ibs_ctx* c) : ctx(c) {}

  Geo geo(int64_t n) const {
    if (sweep) return {(n + kTcBlock - 1) / kTcBlock, sweep_cols(pg.m), sweep_planes_bytes(n, pg.m)};
    if (tc) return {(n + kTcBlock - 1) / kTcBlock, tc_chunks(pg.m, fmt), tc_planes_bytes(n, pg.m, fmt)};
    const PlaneGeom g = PlaneGeom::make(n, pg.m);
    return {g.n_blocks, g.n_chunks, g.bytes()};
  }
  size_t chunk_block_bytes() const { return tc ? (size_t)kTcChunkBytes : (size_t)kChunkBytes; }

  // Planes of n samples from a packed device matrix, on stream s.
  cudaError_t build_planes(const uint8_t* packed, int64_t n, void* planes, cudaStream_t s) const {
    if (sweep) return launch_sweep_planes(packed, n, pg.m, static_cast<uint8_t*>(planes), s);
    if (tc) return launch_tc_planes(packed, n, pg.m, static_cast<uint8_t*>(planes), fmt, s);
    BedSource src;
    src.packed = packed;
    src.row_bytes = (n + 3) / 4;
    src.n_src = n;
    return launch_planes(src, n, pg.m, PlaneGeom::make(n, pg.m), static_cast<uint32_t*>(planes), ctx->status_dev,
                         s);
  }

  cudaError_t cross(const CrossItem* items, int64_t n_items, cudaStream_t s) const {
    if (tc)
      return launch_tc_cross(static_cast<const uint8_t*>(panel_planes.p), pg.n, pgeo.chunks, items, n_items,
                             (int)std::min<int64_t>(ctx->num_sms, std::max<int64_t>(1, n_items)), fmt,
                             static_cast<int*>(counter.p), ctx->status_dev, s);
    return launch_cross(pick_mode(ctx), static_cast<const uint32_t*>(panel_planes.p), pg.n, pg.n_blocks,
                        pg.n_chunks, items, n_items, ctx->status_dev, s);
  }

  size_t mem_need(int64_t q, int k, bool counts_dev, bool topk_dev) const {
    size_t b = (size_t)pg.m * (size_t)((q + 3) / 4) + geo(q).bytes;
    if (!counts_dev) b += (size_t)q * pg.n * 16;
    if (!topk_dev) b += (size_t)q * k * 12;
    return b + 4096;
  }

  // Per-request buffers come from the device's stream-ordered memory pool
  // (cudaMallocAsync / cudaFreeAsync on the stream that uses them): no
  // device-wide synchronisation when a request's memory is returned, so the
  // step pipeline never stalls on a free.
  void free_async(Request& r, bool packed_too, cudaStream_t s) {
    for (DevBuf* b : {&r.packed, &r.planes, &r.counts, &r.tidx, &r.tdist}) {
      if (b == &r.packed && !packed_too) continue;
      if (b->p) cudaFreeAsync(b->p, s);
      b->p = nullptr;
      b->cap = 0;
    }
  }
  void release(Request& r, cudaStream_t s) {
    free_async(r, true, s);
    if (r.reserved) {
      release_bytes(ctx, r.reserved);
      std::lock_guard<std::mutex> lk(budget_mu);
      pool_bytes -= r.reserved;
    }
    r.reserved = 0;
    if (r.done_ev) cudaEventDestroy(r.done_ev);
    r.done_ev = nullptr;
  }

  // The panel's words are an extra: a request that finds no memory has them
  // given back (true if there were any; cudaFree waits for their last use).
  bool give_back_words() {
    std::lock_guard<std::mutex> lk(words_mu);
    if (!panel_words.p) return false;
    free_buf(ctx, panel_words);
    return true;
  }

  ibs_status alloc(DevBuf& b, size_t bytes, cudaStream_t s) {
    if (bytes == 0) return IBS_OK;
    cudaError_t e = cudaMallocAsync(&b.p, bytes, s);
    if (e != cudaSuccess && give_back_words()) e = cudaMallocAsync(&b.p, bytes, s);
    if (e != cudaSuccess && drop_pool_words(ctx)) e = cudaMallocAsync(&b.p, bytes, s);
    if (e != cudaSuccess) {
      cudaGetLastError();
      b.p = nullptr;
      return IBS_ENOMEM;
    }
    b.cap = bytes;
    return IBS_OK;
  }

  // Reserve a request's bytes against the serving budget (free device memory
  // at panel load minus a margin, and the context's workspace limit).
  bool reserve_request(Request& r, size_t need) {
    {
      std::lock_guard<std::mutex> lk(budget_mu);
      if (pool_bytes + need > pool_budget) return false;
      pool_bytes += need;
    }
    if (!reserve_bytes(ctx, need)) {
      std::lock_guard<std::mutex> lk(budget_mu);
      pool_bytes -= need;
      return false;
    }
    r.reserved = need;
    return true;
  }

  // The samples of a request from the caller's memory into device memory
  // (caller's thread, which holds in_mu; done on return).  Device memory is read
  // in the legacy stream's order, as by a plain copy.  The calls are allowed
  // while a thread captures a graph elsewhere.
  bool copy_in(Request& r, const uint8_t* q, size_t bytes) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    bool ok = alloc(r.packed, bytes, in) == IBS_OK;
    if (ok) {
      const cudaStream_t s = ptr_kind(q) == PtrKind::Device ? cudaStreamLegacy : in;
      ok = cudaStreamSynchronize(in) == cudaSuccess &&
           cudaMemcpyAsync(r.packed.p, q, bytes, cudaMemcpyDefault, s) == cudaSuccess &&
           cudaStreamSynchronize(s) == cudaSuccess;
      if (!ok) {
        cudaGetLastError();
        cudaFreeAsync(r.packed.p, in);
        r.packed = DevBuf{};
      }
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    return ok;
  }

  // Try to admit r (engine thread).  Returns false if it must wait; it then
  // keeps what it brought along (its memory in the budget, its samples).
  bool admit(const std::shared_ptr<Request>& r, int64_t active_rows) {
    if (active_rows + r->q > kMaxRows && active_rows > 0) return false;
    const size_t need = mem_need(r->q, r->k, r->counts_on_dev, r->topk_on_dev);
    if (!r->early && !reserve_request(*r, need)) return false;
    const size_t pk = (size_t)pg.m * (size_t)((r->q + 3) / 4);
    const bool host = r->packed.p == nullptr;  // the samples are in host_packed
    if ((host && alloc(r->packed, pk, stream)) || alloc(r->planes, geo(r->q).bytes, stream) ||
        (!r->counts_on_dev && alloc(r->counts, (size_t)r->q * pg.n * 16, stream)) ||
        (!r->topk_on_dev && r->k > 0 &&
         (alloc(r->tidx, (size_t)r->q * r->k * 4, stream) || alloc(r->tdist, (size_t)r->q * r->k * 8, stream)))) {
      if (r->early)
        free_async(*r, host, stream);
      else
        release(*r, stream);
      return false;
    }
    if (host) cudaMemcpyAsync(r->packed.p, r->host_packed.data(), pk, cudaMemcpyHostToDevice, stream);
    cudaEventCreateWithFlags(&r->done_ev, cudaEventDisableTiming);
    r->blocks_done = 0;
    r->state = RState::Active;
    return true;
  }

  // The samples of the early requests behind the first in line go back to the
  // host (nothing is on the GPU, and the first found no device memory beside
  // them); true if there were any.  lk holds mu.
  bool take_back(std::unique_lock<std::mutex>& lk) {
    std::vector<std::shared_ptr<Request>> behind;
    bool first = true;
    for (const auto& r : pending) {
      if (r->arriving) continue;
      if (!first && r->packed.p) behind.push_back(r);
      first = false;
    }
    lk.unlock();
    bool any = false;
    for (const auto& r : behind) {
      try {
        r->host_packed.resize((size_t)pg.m * (size_t)((r->q + 3) / 4));
      } catch (const std::bad_alloc&) {
        continue;
      }
      if (cudaMemcpyAsync(r->host_packed.data(), r->packed.p, r->host_packed.size(), cudaMemcpyDeviceToHost, stream) !=
              cudaSuccess ||
          cudaStreamSynchronize(stream) != cudaSuccess) {
        cudaGetLastError();
        r->host_packed.clear();
        continue;  // its samples stay where they are
      }
      free_async(*r, true, stream);
      any = true;
    }
    lk.lock();
    return any;
  }

  int32_t* counts_ptr(Request& r) { return r.counts_on_dev ? r.user_counts : static_cast<int32_t*>(r.counts.p); }

  // The request's counts columns [b0, b1) panel blocks, written by the step
  // just enqueued, to its host buffer (on the copy stream, which waits for
  // the step's kernel).
  void copy_columns(Request& r, int64_t b0, int64_t b1) {
    const int64_t c0 = b0 * blk, c1 = std::min<int64_t>(b1 * blk, pg.n);
    if (c1 <= c0) return;
    const size_t pitch = (size_t)pg.n * 16;
    cudaMemcpy2DAsync(r.user_counts + c0 * 4, pitch, static_cast<const int32_t*>(r.counts.p) + c0 * 4, pitch,
                      (size_t)(c1 - c0) * 16, (size_t)r.q, cudaMemcpyDeviceToHost, side);
  }

  // Top-k of the requests that saw their last panel block in this step (on
  // the engine stream, after the step), then their top-k lists to the host
  // and their completion events on the copy stream (after their last counts
  // columns).  After a step that failed: the events only.
  void finish(const std::vector<std::shared_ptr<Request>>& done, int slot, cudaError_t err) {
    auto ok = [&](cudaError_t e) {
      if (err == cudaSuccess) err = e;
    };
    // every row of every finishing request in one launch (at most kMaxRows
    // rows: the admitted set never holds more)
    int64_t n = 0;
    for (auto& rp : done) n += rp->k > 0 ? rp->q : 0;
    // few rows: the table goes as an argument and the lists straight to mapped
    // pinned memory, instead of three small copies
    const bool few = n <= kFewRows;
    n = 0;
    for (auto& rp : done) {
      Request& r = *rp;
      if (r.k <= 0) continue;
      r.topk_direct = few && r.map_idx && r.map_dist;
      int32_t* oi = r.topk_on_dev ? r.user_idx : r.topk_direct ? r.map_idx : static_cast<int32_t*>(r.tidx.p);
      double* od = r.topk_on_dev ? r.user_dist : r.topk_direct ? r.map_dist : static_cast<double*>(r.tdist.p);
      const int32_t* cnt = counts_ptr(r);
      for (int64_t row = 0; row < r.q && n < kMaxRows; ++row, ++n)
        topk_host[slot][n] = TopkRow{cnt + (size_t)row * pg.n * 4, oi + row * r.k, od + row * r.k, r.k, 0};
    }
    if (err == cudaSuccess && n > 0 && few) {
      ok(launch_topk_few(topk_host[slot], n, pg.n, stream));
    } else if (err == cudaSuccess && n > 0) {
      ok(cudaMemcpyAsync(topk_dev[slot].p, topk_host[slot], (size_t)n * sizeof(TopkRow), cudaMemcpyHostToDevice,
                         stream));
      ok(launch_topk_rows(static_cast<const TopkRow*>(topk_dev[slot].p), n, pg.n, stream));
    }
    if (!fin_ev[slot]) cudaEventCreateWithFlags(&fin_ev[slot], cudaEventDisableTiming);
    cudaEventRecord(fin_ev[slot], stream);
    cudaStreamWaitEvent(side, fin_ev[slot], 0);
    for (auto& rp : done) {
      Request& r = *rp;
      if (err == cudaSuccess && !r.topk_on_dev && !r.topk_direct && r.k > 0) {
        ok(cudaMemcpyAsync(r.user_idx, r.tidx.p, (size_t)r.q * r.k * 4, cudaMemcpyDeviceToHost, side));
        ok(cudaMemcpyAsync(r.user_dist, r.tdist.p, (size_t)r.q * r.k * 8, cudaMemcpyDeviceToHost, side));
      }
      cudaEventRecord(r.done_ev, side);
      r.state = RState::Finishing;
    }
    if (err == cudaSuccess) return;
    cudaGetLastError();
    for (auto& rp : done) rp->status = IBS_ECUDA;
  }

  // Rows against panel blocks [cols[0][0], cols[0][1]) and [cols[1][0], cols[1][1])
  // on the sweep kernel: the plan's lists through `host` (pinned; or pageable,
  // staged before return) into `dev`, the launches on s.  Both hold at least
  // sweep_list_bytes(plan) bytes.
  static size_t sweep_list_bytes(const SweepPlan& pl) {
    return pl.items.size() * sizeof(SweepItem) + pl.groups.size() * sizeof(SweepGroup) +
           (pl.first.size() + 8) * sizeof(int32_t);
  }
  cudaError_t run_sweep(const SweepPlan& pl, const uint8_t* row_planes, int64_t row_half, int32_t* const* row_out,
                        int64_t n_rows, uint8_t* host, uint8_t* dev, const DevBuf& scratch, const DevBuf& part,
                        DevBuf& ctr, bool library_buf, cudaStream_t s) {
    // (the kernel indexes both by the plan)
    if (sweep_scratch_bytes(pl.clusters) > scratch.cap || (size_t)pl.slots * sweep_slot_bytes() > part.cap)
      return cudaErrorInvalidValue;
    const size_t ib = pl.items.size() * sizeof(SweepItem), gb = pl.groups.size() * sizeof(SweepGroup);
    std::memcpy(host, pl.items.data(), ib);
    if (gb > 0) std::memcpy(host + ib, pl.groups.data(), gb);
    std::memcpy(host + ib + gb, pl.first.data(), pl.first.size() * sizeof(int32_t));
    cudaError_t e = cudaMemcpyAsync(dev, host, ib + gb + pl.first.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    SweepLaunch l;
    l.items = reinterpret_cast<const SweepItem*>(dev);
    l.groups = reinterpret_cast<const SweepGroup*>(dev + ib);
    l.first = reinterpret_cast<const int32_t*>(dev + ib + gb);
    l.n_groups = (int64_t)pl.groups.size();
    l.clusters = pl.clusters;
    l.scratch = static_cast<float*>(scratch.p);
    l.part = static_cast<float*>(part.p);
    l.status = ctx->status_dev;
    l.wait_ns = kWaitLimitNs;
    l.sync = sweep_sync(pl.waves, pl.wave_stages, tc_pair_sync_setting(0));
    const size_t bytes = (size_t)pl.waves * l.sync.n_seg * sizeof(int);
    if (bytes > 0) {
      if (library_buf ? ensure_buf(ctx, ctr, bytes) != IBS_OK : alloc(ctr, bytes, s) != IBS_OK) {
        l.sync = SweepSync{};
      } else {
        if ((e = cudaMemsetAsync(ctr.p, 0, bytes, s)) != cudaSuccess) return e;
        l.sync.ctr = static_cast<int*>(ctr.p);
      }
    }
    return launch_sweep_cross(row_planes, row_half, static_cast<const uint8_t*>(panel_planes.p), pg.n, pg.m, row_out,
                              n_rows, l, s);
  }

  // Parts that a plan over C clusters can need: its shares meet at C - 1 cuts,
  // each the end of one piece and the start of another, and a piece touches at
  // most three products; in rounds, at most as many by their own rule.
  size_t sweep_part_bytes() const { return (size_t)sweep_max_slots(clusters) * sweep_slot_bytes(); }

  cudaError_t ensure_items(size_t n) {
    if (n <= items_cap) return cudaSuccess;
    const size_t each = std::max(std::max(sizeof(CrossItem), sizeof(PairItem)), sizeof(SweepItem));
    items_cap = 0;
    cudaError_t err = cudaSuccess;
    for (int s = 0; s < 2; ++s) {
      if (step_ev[s]) cudaEventSynchronize(step_ev[s]);
      if (items_dev[s].p) cudaFree(items_dev[s].p);
      if (items_host[s]) cudaFreeHost(items_host[s]);
      items_dev[s].p = nullptr;
      items_host[s] = nullptr;
      if (err == cudaSuccess) err = cudaMalloc(&items_dev[s].p, n * each);
      if (err == cudaSuccess)
        err = cudaHostAlloc(reinterpret_cast<void**>(&items_host[s]), n * each, cudaHostAllocDefault);
    }
    if (err == cudaSuccess) items_cap = n;
    return err;
  }

  // K-lockstep of a two-SM launch of n_items equal items (whole waves of one
  // item per cluster take part); counters zeroed on stream s.  Off (an empty
  // PairSync) when the setting is off or the counters cannot be had.
  PairSync pair_sync(int64_t n_items, DevBuf& ctr, bool library_buf, cudaStream_t s) {
    PairSync ps;
    const int2 ss = tc_pair_sync_setting(pgeo.chunks);
    const int64_t waves = n_items / std::max(1, clusters);
    if (ss.x <= 0 || waves < 1) return ps;
    const int32_t n_seg = (int32_t)((pgeo.chunks + ss.x - 1) / ss.x);
    const size_t bytes = (size_t)waves * n_seg * sizeof(int);
    if (library_buf ? ensure_buf(ctx, ctr, bytes) != IBS_OK : alloc(ctr, bytes, s) != IBS_OK) return ps;
    if (cudaMemsetAsync(ctr.p, 0, bytes, s) != cudaSuccess) return ps;
    ps.ctr = static_cast<int*>(ctr.p);
    ps.seg = ss.x;
    ps.lag = ss.y;
    ps.n_seg = n_seg;
    ps.n_items = waves * clusters;
    return ps;
  }

  // Step length in panel blocks for `units` item rows (query blocks, or query
  // block pairs on the two-SM kernel) run by C persistent CTAs or clusters:
  // about kStepWaves(Tc) waves of items, at least 1/kMinStepDiv of the panel,
  // at most all of it; among the lengths up to one more wave, the one whose
  // last wave is fullest (the items of a step all cost the same), the
  // shortest of equals.
  int64_t step_len(int64_t units, int64_t C) const {
    units = std::max<int64_t>(1, units);
    C = std::max<int64_t>(1, C);
    int64_t lo = ((tc ? kStepWavesTc : kStepWaves) * C + units - 1) / units;
    lo = std::max<int64_t>(lo, (pgeo.blocks + kMinStepDiv - 1) / kMinStepDiv);
    lo = std::min<int64_t>(lo, pgeo.blocks);
    const int64_t hi = std::min<int64_t>(pgeo.blocks, lo + (C + units - 1) / units);
    int64_t best = lo;
    double best_fill = 0.0;
    for (int64_t L = lo; L <= hi; ++L) {
      const int64_t n = units * L;
      const double fill = (double)n / (double)(((n + C - 1) / C) * C);
      if (fill > best_fill + 1e-3) {
        best_fill = fill;
        best = L;
      }
    }
    return best;
  }

  // Step-level buffers: dense query planes for kMaxRows rows and the per-row
  // source / output tables (double-buffered host staging).
  ibs_status alloc_step_buffers() {
    if (ibs_status s = ensure_buf(ctx, step_planes, geo(kMaxRows).bytes)) return s;
    if (ibs_status s = ensure_buf(ctx, counter, 256)) return s;
    for (int s = 0; s < 2; ++s) {
      if (ibs_status e = ensure_buf(ctx, topk_dev[s], kMaxRows * sizeof(TopkRow))) return e;
      if (cudaHostAlloc(reinterpret_cast<void**>(&topk_host[s]), kMaxRows * sizeof(TopkRow), cudaHostAllocDefault) !=
          cudaSuccess)
        return fail(IBS_ENOMEM, "pinned top-k tables could not be allocated");
      if (ibs_status e = ensure_buf(ctx, rows_dev[s], kMaxRows * sizeof(RowSrc))) return e;
      if (ibs_status e = ensure_buf(ctx, outs_dev[s], kMaxRows * sizeof(int32_t*))) return e;
      if (cudaHostAlloc(reinterpret_cast<void**>(&rows_host[s]), kMaxRows * sizeof(RowSrc), cudaHostAllocDefault) !=
              cudaSuccess ||
          cudaHostAlloc(reinterpret_cast<void**>(&outs_host[s]), kMaxRows * sizeof(int32_t*), cudaHostAllocDefault) !=
              cudaSuccess)
        return fail(IBS_ENOMEM, "pinned step tables could not be allocated");
    }
    return IBS_OK;
  }

  // One step: every active request's rows, packed densely into query blocks,
  // against the current panel chunk.  When a copy or a launch of it fails, the
  // requests in it end with IBS_ECUDA; the engine goes on.
  void run_step() {
    cudaGetLastError();  // (a query of an event that is not ready leaves one: no launch reports it as its own)
    cudaError_t err = cudaSuccess;
    auto ok = [&](cudaError_t e) {
      if (err == cudaSuccess) err = e;
    };
    {
      std::lock_guard<std::mutex> lk(mu);
      if (failing_steps > 0) {
        --failing_steps;
        err = cudaErrorLaunchFailure;
      }
    }
    const int slot = (int)(step_no & 1);
    if (step_ev[slot]) cudaEventSynchronize(step_ev[slot]);  // slot's host tables are free again
    int64_t n_rows = 0;
    for (auto& r : active) n_rows += r->q;
    // Few rows: the panel's code bits instead of its operand planes
    std::unique_lock<std::mutex> words_lk(words_mu);
    const bool few = few_rows_pay(n_rows, pg.n, pg.m) && panel_words.p;
    if (!few) words_lk.unlock();
    n_rows = 0;
    for (auto& r : active)
      for (int64_t row = 0; row < r->q; ++row) {
        rows_host[slot][n_rows].planes = static_cast<const uint32_t*>(few ? r->packed.p : r->planes.p);
        rows_host[slot][n_rows].row = row;
        rows_host[slot][n_rows].n_half = few ? (r->q + 3) / 4 : (r->q + 63) / 64;
        outs_host[slot][n_rows] = counts_ptr(*r) + (size_t)row * pg.n * 4;
        ++n_rows;
      }
    const int64_t qblocks = (n_rows + blk - 1) / blk;
    // Step length: few rows in flight -> one step covers the whole panel (a
    // lone request costs one launch, as on the unbatched path); many rows ->
    // shorter steps that new requests can join between.
    const bool two_sm = pair && qblocks >= 2;
    const int64_t units = two_sm || sweep ? (qblocks + 1) / 2 : qblocks;
    int64_t left = 0;  // panel blocks that some request still has to see
    for (auto& r : active) left = std::max(left, pgeo.blocks - r->blocks_done);
    const int64_t len = few     ? left
                        : sweep ? sweep_step_blocks(pgeo.blocks, qblocks, left, clusters)
                                : step_len(units, two_sm ? clusters : grid_ctas);
    const size_t n_items = (size_t)units * (size_t)len;
    SweepPlan pl;
    const int64_t end = cursor + len;  // wraps around the panel at most once
    const int64_t cols[2][2] = {{cursor, std::min(end, pgeo.blocks)}, {0, std::max<int64_t>(0, end - pgeo.blocks)}};
    if (sweep && n_rows > 0 && !few) {
      pl = sweep_plan_cross(qblocks, cols, pg.m, clusters);
      ok(ensure_items(std::max<size_t>(sweep_list_bytes(pl) / sizeof(SweepItem) + 1, n_items)));
    } else {
      ok(ensure_items(std::max<size_t>(n_items, 1)));
    }
    size_t t = 0;
    int32_t** outs_d = static_cast<int32_t**>(outs_dev[slot].p);
    if (err != cudaSuccess) {
      // nothing to list
    } else if (few) {
      t = 1;
    } else if (sweep) {
      t = pl.items.size();
    } else if (two_sm) {
      PairItem* h = reinterpret_cast<PairItem*>(items_host[slot]);
      for (int64_t k = 0; k < len; ++k) {
        const int64_t pb = (cursor + k) % pgeo.blocks;  // wraps around the panel
        for (int64_t u = 0; u < units; ++u) {
          PairItem& it = h[t++];
          it = PairItem{};
          it.I0 = (int32_t)(2 * u);
          it.I1 = 2 * u + 1 < qblocks ? (int32_t)(2 * u + 1) : -1;
          it.J = (int32_t)pb;
          it.c0 = 0;
          it.c1 = (int32_t)pgeo.chunks;
        }
      }
    } else {
      CrossItem* h = reinterpret_cast<CrossItem*>(items_host[slot]);
      const size_t qblock_bytes = (size_t)pgeo.chunks * chunk_block_bytes();
      for (int64_t k = 0; k < len; ++k) {
        const int64_t pb = (cursor + k) % pgeo.blocks;  // wraps around the panel
        for (int64_t b = 0; b < qblocks; ++b) {
          CrossItem& it = h[t++];
          it.qplanes =
              reinterpret_cast<const uint32_t*>(static_cast<const uint8_t*>(step_planes.p) + b * qblock_bytes);
          it.row_out = outs_d + b * blk;
          it.q_rows = (int32_t)std::min<int64_t>(blk, n_rows - b * blk);
          it.pb = (int32_t)pb;
        }
      }
    }
    if (t > 0) {
      if (!few && gathered_version != set_version) {
        for (auto& r : active) {
          if (r->planes_built) continue;
          ok(build_planes(static_cast<const uint8_t*>(r->packed.p), r->q, r->planes.p, stream));
          r->planes_built = true;
        }
        // the admitted set changed: pack its rows into the step planes again
        ok(cudaMemcpyAsync(rows_dev[slot].p, rows_host[slot], n_rows * sizeof(RowSrc), cudaMemcpyHostToDevice, stream));
        if (sweep)
          ok(launch_sweep_gather_rows(static_cast<const RowSrc*>(rows_dev[slot].p), n_rows, pgeo.chunks,
                                      static_cast<uint8_t*>(step_planes.p), kMaxRows / 64, stream));
        else if (tc)
          ok(launch_tc_gather_rows(static_cast<const RowSrc*>(rows_dev[slot].p), n_rows, pgeo.chunks,
                                   static_cast<uint8_t*>(step_planes.p), stream));
        else
          ok(launch_gather_rows(static_cast<const RowSrc*>(rows_dev[slot].p), n_rows, pg.n_chunks,
                                static_cast<uint32_t*>(step_planes.p), stream));
        gathered_version = set_version;
      }
      if (!few)
        ok(cudaMemcpyAsync(outs_dev[slot].p, outs_host[slot], n_rows * sizeof(int32_t*), cudaMemcpyHostToDevice, stream));
      if (err != cudaSuccess) {
        // nothing reads what may not be there
      } else if (few) {
        const int64_t samples[2][2] = {{cols[0][0] * blk, std::min<int64_t>(cols[0][1] * blk, pg.n)},
                                       {0, std::min<int64_t>(cols[1][1] * blk, pg.n)}};
        FewTables tab;
        for (int64_t r = 0; r < n_rows; ++r) {
          tab.rows[r] = rows_host[slot][r];
          tab.out[r] = outs_host[slot][r];
        }
        ok(launch_few_rows(tab, n_rows,
                           static_cast<const uint32_t*>(panel_words.p), pg.n, pg.m, samples, few_words.p, sweep_part.p,
                           sweep_part.cap, ctx->num_sms, stream));
      } else if (sweep) {
        ok(run_sweep(pl, static_cast<const uint8_t*>(step_planes.p), kMaxRows / 64, outs_d, n_rows, items_host[slot],
                     static_cast<uint8_t*>(items_dev[slot].p), sweep_scratch, sweep_part, sync_ctr, true, stream));
      } else if (two_sm) {
        ok(cudaMemcpyAsync(items_dev[slot].p, items_host[slot], t * sizeof(PairItem), cudaMemcpyHostToDevice, stream));
        ok(launch_tc_pair_cross(static_cast<const uint8_t*>(panel_planes.p), pg.n, pgeo.chunks,
                                static_cast<const uint8_t*>(step_planes.p), geo(kMaxRows).blocks, outs_d, n_rows,
                                static_cast<const PairItem*>(items_dev[slot].p), (int64_t)t, ctx->status_dev, stream,
                                pair_sync((int64_t)t, sync_ctr, true, stream)));
      } else {
        ok(cudaMemcpyAsync(items_dev[slot].p, items_host[slot], t * sizeof(CrossItem), cudaMemcpyHostToDevice, stream));
        ok(cross(static_cast<const CrossItem*>(items_dev[slot].p), (int64_t)t, stream));
      }
      // this step's panel columns of requests whose counts go to host memory
      bool any_host = false;
      for (auto& r : active) any_host |= err == cudaSuccess && !r->counts_on_dev && r->user_counts;
      if (any_host) {
        if (!kern_ev[slot]) cudaEventCreateWithFlags(&kern_ev[slot], cudaEventDisableTiming);
        cudaEventRecord(kern_ev[slot], stream);
        cudaStreamWaitEvent(side, kern_ev[slot], 0);
        const int64_t b0 = cursor, b1 = cursor + len;  // may wrap once
        for (auto& r : active) {
          if (r->counts_on_dev || !r->user_counts) continue;
          copy_columns(*r, b0, std::min<int64_t>(b1, pgeo.blocks));
          if (b1 > pgeo.blocks) copy_columns(*r, 0, b1 - pgeo.blocks);
        }
      }
    }
    if (few) words_lk.unlock();
    cursor = (cursor + len) % pgeo.blocks;
    std::vector<std::shared_ptr<Request>> still, done;
    for (auto& r : active) {
      // A request joined at some cursor position and is done once it has seen
      // every panel block (blocks seen twice near the end are rewritten with
      // the same counts), or when its step failed.
      r->blocks_done += len;
      if (r->blocks_done >= pgeo.blocks || err != cudaSuccess) {
        done.push_back(r);
        finishing.push_back(r);
      } else {
        still.push_back(r);
      }
    }
    if (!done.empty()) {
      finish(done, slot, err);
      ++set_version;
    }
    active.swap(still);
    if (!step_ev[slot]) cudaEventCreateWithFlags(&step_ev[slot], cudaEventDisableTiming);
    cudaEventRecord(step_ev[slot], stream);
    ++step_no;
    std::lock_guard<std::mutex> lk(mu);
    stats.steps++;
  }

  void check_finishing() {
    std::vector<std::shared_ptr<Request>> still;
    bool any = false;
    for (auto& r : finishing) {
      const cudaError_t q = cudaEventQuery(r->done_ev);
      if (q != cudaErrorNotReady) {
        const int st = __atomic_load_n(ctx->status_host, __ATOMIC_SEQ_CST);
        std::lock_guard<std::mutex> lk(mu);
        if (q != cudaSuccess) r->status = IBS_ECUDA;
        if (r->status == IBS_OK && st == kDevTimeout) r->status = IBS_ETIMEOUT;
        release(*r, stream);
        if (r->early) early_rows -= r->q;
        r->state = RState::Done;
        stats.requests_done++;
        any = true;
      } else {
        still.push_back(r);
      }
    }
    finishing.swap(still);
    if (any) cv_done.notify_all();
  }

  void loop() {
    cudaSetDevice(ctx->device);
    for (;;) {
      check_finishing();
      {
        std::unique_lock<std::mutex> lk(mu);
        if (stop) break;
        int64_t rows = 0;
        for (auto& r : active) rows += r->q;
        // In the order of the queue, past the requests whose samples are still on
        // their way; callers only add at its end.
        for (size_t i = 0; i < pending.size();) {
          auto r = pending[i];
          if (r->arriving) {
            ++i;
            continue;
          }
          lk.unlock();
          const bool ok = admit(r, rows);
          lk.lock();
          if (!ok) break;
          pending.erase(pending.begin() + (std::ptrdiff_t)i);
          active.push_back(r);
          ++set_version;
          rows += r->q;
          stats.peak_rows = std::max<uint64_t>(stats.peak_rows, (uint64_t)rows);
        }
        if (active.empty()) {
          auto waiting = [&] {
            return std::any_of(pending.begin(), pending.end(), [](const auto& r) { return !r->arriving; });
          };
          if (finishing.empty()) {
            if (!waiting())
              cv_work.wait(lk, [&] { return stop || waiting(); });
            else if (!take_back(lk))  // the first in line waits for memory held elsewhere
              cv_work.wait_for(lk, std::chrono::microseconds(200));
          } else if (waiting()) {  // (for memory)
            cv_work.wait_for(lk, std::chrono::microseconds(200));
          } else {
            // the last results are a few hundred microseconds away: poll (a timed
            // wait would add its period to every lone request's latency)
            const auto t0 = std::chrono::steady_clock::now();
            do {
              lk.unlock();
              const bool done = cudaEventQuery(finishing.front()->done_ev) != cudaErrorNotReady;
              lk.lock();
              if (done || stop || waiting()) break;
            } while (std::chrono::steady_clock::now() - t0 < std::chrono::milliseconds(2));
            if (!stop && !waiting() && cudaEventQuery(finishing.front()->done_ev) == cudaErrorNotReady)
              cv_work.wait_for(lk, std::chrono::microseconds(200));
          }
          continue;
        }
      }
      run_step();
    }
  }

  void start() { worker = std::thread([this] { loop(); }); }

  void shutdown() {
    {
      std::lock_guard<std::mutex> lk(mu);
      stop = true;
    }
    cv_work.notify_all();
    if (worker.joinable()) worker.join();
    {
      // A call that is bringing its request in uses the engine's memory and the
      // context: it has returned before either goes.
      std::unique_lock<std::shared_mutex> in_lk(in_mu);
      if (in) cudaStreamDestroy(in);
      in = nullptr;
    }
    cudaStreamSynchronize(stream);
    if (side) cudaStreamSynchronize(side);
    std::lock_guard<std::mutex> lk(mu);
    for (auto& kv : all) {
      Request& r = *kv.second;
      if (r.state != RState::Done) {
        r.status = IBS_ECANCELLED;
        r.state = RState::Done;
      }
      release(r, stream);
    }
    pending.clear();
    active.clear();
    finishing.clear();
    cv_done.notify_all();
    for (int s = 0; s < 2; ++s) {
      if (items_dev[s].p) cudaFree(items_dev[s].p);
      if (items_host[s]) cudaFreeHost(items_host[s]);
      if (step_ev[s]) cudaEventDestroy(step_ev[s]);
      if (kern_ev[s]) cudaEventDestroy(kern_ev[s]);
      if (fin_ev[s]) cudaEventDestroy(fin_ev[s]);
      items_dev[s].p = nullptr;
      items_host[s] = nullptr;
      step_ev[s] = nullptr;
      kern_ev[s] = nullptr;
      fin_ev[s] = nullptr;
    }
    if (panel_planes.p) free_buf(ctx, panel_planes);
    free_buf(ctx, step_planes);
    free_buf(ctx, counter);
    free_buf(ctx, sync_ctr);
    for (DevBuf* b : {&sweep_scratch, &sweep_part, &sync_scratch, &sync_part, &panel_words, &few_words}) free_buf(ctx, *b);
    for (int s = 0; s < 2; ++s) {
      free_buf(ctx, topk_dev[s]);
      if (topk_host[s]) cudaFreeHost(topk_host[s]);
      topk_host[s] = nullptr;
      free_buf(ctx, rows_dev[s]);
      free_buf(ctx, outs_dev[s]);
      if (rows_host[s]) cudaFreeHost(rows_host[s]);
      if (outs_host[s]) cudaFreeHost(outs_host[s]);
      rows_host[s] = nullptr;
      outs_host[s] = nullptr;
    }
    if (stream) cudaStreamDestroy(stream);
    if (side) cudaStreamDestroy(side);
    {
      std::lock_guard<std::mutex> sync_lk(sync_mu);
      if (sync_ev) cudaEventDestroy(sync_ev);
      sync_ev = nullptr;
    }
    stream = nullptr;
    side = nullptr;
  }
};

std::shared_ptr<ServeEngine> engine_of(ibs_ctx* ctx) {
  std::lock_guard<std::mutex> lk(ctx->mu);
  return ctx->serve;
}

bool serve_give_back_words(ibs_ctx* ctx) {
  const auto e = engine_of(ctx);
  return e && e->give_back_words();
}

void serve_stop(ibs_ctx* ctx) {
  std::shared_ptr<ServeEngine> e;
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    e.swap(ctx->serve);
  }
  // Waiters hold their own reference, so the engine outlives them.
  if (e) e->shutdown();
}

ibs_status serve_panel_load(ibs_ctx* ctx, const uint8_t* panel, int64_t n_panel, int64_t m) {
  if (!panel) return fail(IBS_EINVAL, "panel_packed is NULL");
  if (n_panel < 1 || n_panel > 2147483647LL || m < 1 || m > 2147483647LL)
    return fail(IBS_EINVAL, "panel size out of range");
  DeviceGuard g(ctx->device);
  serve_stop(ctx);
  auto eng = std::make_shared<ServeEngine>(ctx);
  eng->pg = PlaneGeom::make(n_panel, m);
  eng->fmt = ctx_tc_format(ctx);
  // The tensor-core form covers a panel's whole marker range in one
  // accumulation, exact up to 2^21 markers; longer panels are served by the
  // integer-pipe kernels.
  eng->tc = ctx_use_tc(ctx) && tc_chunks(m, eng->fmt) <= tc_max_chunks(eng->fmt);
  eng->blk = eng->tc ? kTcBlock : kSB;
  // The sweep kernel where it can run, unless the caller bounds the library's
  // memory (its workspace would leave less of the bound to the requests); its
  // planes have a layout of their own, so this is settled before the panel's
  // are built.
  auto no_sweep = [&] {
    for (DevBuf* b : {&eng->sweep_scratch, &eng->sweep_part, &eng->sync_scratch, &eng->sync_part}) free_buf(ctx, *b);
    eng->sweep = false;
    eng->clusters = 0;
    eng->pgeo = eng->geo(n_panel);
  };
  if (ctx->sweep_on && eng->tc && eng->fmt == kTcFp4 && ctx->ws_limit == 0 && tc_pair_mode() >= 0 && sweep_usable(std::max<int64_t>(n_panel, kMaxRows), m)) {
    eng->clusters = sweep_clusters();
    eng->sweep = true;
    for (DevBuf* b : {&eng->sweep_scratch, &eng->sync_scratch})
      eng->sweep = eng->sweep && ensure_buf(ctx, *b, sweep_scratch_bytes(eng->clusters)) == IBS_OK;
    for (DevBuf* b : {&eng->sweep_part, &eng->sync_part})
      eng->sweep = eng->sweep && ensure_buf(ctx, *b, eng->sweep_part_bytes()) == IBS_OK;
    if (!eng->sweep) no_sweep();
    clear_error();
  }
  eng->pgeo = eng->geo(n_panel);
  if (cudaStreamCreateWithFlags(&eng->stream, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    no_sweep();
    return fail(IBS_ECUDA, "engine stream could not be created");
  }
  if (cudaStreamCreateWithFlags(&eng->side, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    cudaStreamDestroy(eng->stream);
    no_sweep();
    return fail(IBS_ECUDA, "copy stream could not be created");
  }
  ibs_status ps = ensure_buf(ctx, eng->panel_planes, eng->pgeo.bytes);
  if (ps == IBS_ENOMEM && eng->sweep) {
    no_sweep();
    ps = ensure_buf(ctx, eng->panel_planes, eng->pgeo.bytes);
  }
  if (ps) {
    cudaStreamDestroy(eng->stream);
    cudaStreamDestroy(eng->side);
    no_sweep();
    return ps;
  }
  clear_error();
  const size_t bytes = (size_t)m * (size_t)((n_panel + 3) / 4);
  const uint8_t* src_dev = panel;
  void* tmp = nullptr;
  if (ptr_kind(panel) != PtrKind::Device) {
    cudaError_t e = cudaMalloc(&tmp, bytes);
    if (e != cudaSuccess && drop_pool_words(ctx)) e = cudaMalloc(&tmp, bytes);
    if (e != cudaSuccess) {
      free_buf(ctx, eng->panel_planes);
      no_sweep();
      cudaStreamDestroy(eng->stream);
      cudaStreamDestroy(eng->side);
      cudaGetLastError();
      return fail(IBS_ENOMEM, "panel staging cudaMalloc(%zu) failed", bytes);
    }
    IBS_CUDA_TRY(cudaMemcpyAsync(tmp, panel, bytes, cudaMemcpyHostToDevice, eng->stream));
    src_dev = static_cast<const uint8_t*>(tmp);
  }
  IBS_CUDA_TRY(eng->build_planes(src_dev, n_panel, eng->panel_planes.p, eng->stream));
  if (eng->sweep) {
    // The panel's words, where they take at most an eighth of the free memory
    // and a step's parts have room for kFewRows rows.
    const size_t wb = (size_t)((m + 31) / 32) * (size_t)n_panel * 8;
    size_t free_b = 0, total_b = 0;
    if ((size_t)kFewRows * n_panel * 12 <= eng->sweep_part.cap && cudaMemGetInfo(&free_b, &total_b) == cudaSuccess &&
        wb <= free_b / 8 && ensure_buf(ctx, eng->few_words, few_rows_bytes((m + 31) / 32)) == IBS_OK &&
        ensure_buf(ctx, eng->panel_words, wb) == IBS_OK) {
      SweepPool sp;
      sp.packed = src_dev;
      sp.row_bytes = (n_panel + 3) / 4;
      sp.n = n_panel;
      sp.m = m;
      sp.cols = (m + 31) / 32;
      sp.words = static_cast<uint32_t*>(eng->panel_words.p);
      IBS_CUDA_TRY(launch_sweep_words(sp, ctx->num_sms, eng->stream));
    }
    cudaGetLastError();
    clear_error();
  }
  IBS_CUDA_TRY(cudaStreamSynchronize(eng->stream));
  if (tmp) cudaFree(tmp);
  if (ibs_status st = eng->alloc_step_buffers()) {
    eng->shutdown();
    return st;
  }
  eng->grid_ctas = eng->tc ? ctx->num_sms : ctx->num_sms * pair_kernel_ctas_per_sm(pick_mode(ctx));
  eng->pair = eng->tc && !eng->sweep && tc_pair_cross_usable(n_panel, eng->pgeo.chunks, eng->fmt);
  if (!eng->sweep) eng->clusters = eng->pair ? tc_pair_clusters(eng->pgeo.chunks) : 0;
  if (eng->clusters < 1) eng->pair = false;
  if (eng->sweep) {
    // lockstep counters for the most waves of a step (all 4,096 rows, every
    // panel block), so that a step never grows them while earlier steps run
    const int64_t cols[2][2] = {{0, eng->pgeo.blocks}, {0, 0}};
    const SweepPlan pl = sweep_plan_cross(kMaxRows / kTcBlock, cols, m, eng->clusters);
    const SweepSync sy = sweep_sync(pl.waves + 1, 4 * sweep_stages(m), tc_pair_sync_setting(0));
    const size_t bytes = (size_t)(pl.waves + 1) * sy.n_seg * sizeof(int);
    if (bytes > 0)
      if (ibs_status st = ensure_buf(ctx, eng->sync_ctr, bytes)) {
        eng->shutdown();
        return st;
      }
  }
  if (eng->pair) {
    // lockstep counters for the largest step (all 4,096 rows, every panel
    // block), so that a step never grows them while earlier steps run
    const int2 ss = tc_pair_sync_setting(eng->pgeo.chunks);
    const int64_t max_items = (eng->geo(kMaxRows).blocks + 1) / 2 * eng->pgeo.blocks;
    if (ss.x > 0) {
      const size_t bytes =
          (size_t)(max_items / eng->clusters + 1) * (size_t)((eng->pgeo.chunks + ss.x - 1) / ss.x) * sizeof(int);
      if (ibs_status st = ensure_buf(ctx, eng->sync_ctr, bytes)) {
        eng->shutdown();
        return st;
      }
    }
  }
  // Requests draw on the device's default stream-ordered pool; keep freed
  // blocks cached in it so steady-state serving does not go back to the driver.
  cudaMemPool_t mp;
  if (cudaDeviceGetDefaultMemPool(&mp, ctx->device) == cudaSuccess) {
    uint64_t keep = UINT64_MAX;
    cudaMemPoolSetAttribute(mp, cudaMemPoolAttrReleaseThreshold, &keep);
  }
  {
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    // the sweep kernel's workspace comes out of the margin
    const size_t held = eng->sweep ? std::min(kMemMargin / 2, 2 * (eng->sweep_scratch.cap + eng->sweep_part.cap)) : 0;
    free_b += eng->panel_words.cap;  // given back when a request needs the room
    eng->pool_budget = free_b > kMemMargin - held ? free_b - (kMemMargin - held) : 0;
  }
  eng->fixed_bytes = eng->panel_planes.cap + eng->step_planes.cap + eng->counter.cap + 2 * (eng->sweep_scratch.cap + eng->sweep_part.cap) +
                     2 * (eng->rows_dev[0].cap + eng->outs_dev[0].cap);
  if (cudaStreamCreateWithFlags(&eng->in, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    eng->in = nullptr;  // requests are kept on the host
  }
  eng->start();
  std::lock_guard<std::mutex> lk(ctx->mu);
  ctx->serve = std::move(eng);
  return IBS_OK;
}

namespace {

ibs_status validate_query(const std::shared_ptr<ServeEngine>& eng, const uint8_t* q, int64_t nq, int k, int32_t* oc,
                          int32_t* oi, double* od, bool& counts_dev, bool& topk_dev) {
  if (!eng) return fail(IBS_ESTATE, "no panel loaded (call ibs_panel_load first)");
  if (!q) return fail(IBS_EINVAL, "query_packed is NULL");
  if (nq < 1 || nq > kMaxQuery) return fail(IBS_EINVAL, "n_query %lld out of range [1, %d]", (long long)nq, kMaxQuery);
  if (k < 0 || k > kMaxK) return fail(IBS_EINVAL, "k=%d out of range [0, %d]", k, kMaxK);
  if (k > 0 && (!oi || !od)) return fail(IBS_EINVAL, "k > 0 needs out_topk_idx and out_topk_dist");
  if (oc && reinterpret_cast<uintptr_t>(oc) % 16) return fail(IBS_EINVAL, "out_counts must be 16-byte aligned");
  counts_dev = oc ? ptr_kind(oc) == PtrKind::Device : false;
  if (oc && !counts_dev && ptr_kind(oc) != PtrKind::PinnedHost)
    return fail(IBS_EINVAL, "out_counts must be device memory or pinned host memory");
  topk_dev = false;
  if (k > 0) {
    const PtrKind a = ptr_kind(oi), b = ptr_kind(od);
    if (a != b) return fail(IBS_EINVAL, "out_topk_idx and out_topk_dist must be the same kind of memory");
    if (a == PtrKind::Pageable) return fail(IBS_EINVAL, "top-k outputs must be device memory or pinned host memory");
    topk_dev = a == PtrKind::Device;
  }
  return IBS_OK;
}

std::vector<uint8_t> copy_query(const uint8_t* q, size_t bytes) {
  std::vector<uint8_t> v(bytes);
  if (ptr_kind(q) == PtrKind::Device) cudaMemcpy(v.data(), q, bytes, cudaMemcpyDeviceToHost);
  else std::memcpy(v.data(), q, bytes);
  return v;
}

}  // namespace

ibs_status serve_query(ibs_ctx* ctx, const uint8_t* q, int64_t nq, int k, int32_t* oc, int32_t* oi, double* od,
                       uint64_t* id) {
  if (!id) return fail(IBS_EINVAL, "req_id is NULL");
  DeviceGuard g(ctx->device);
  bool counts_dev = false, topk_dev = false;
  auto eng = engine_of(ctx);
  if (ibs_status s = validate_query(eng, q, nq, k, oc, oi, od, counts_dev, topk_dev)) return s;
  ServeEngine& e = *eng;
  std::shared_lock<std::shared_mutex> in_lk(e.in_mu);  // until return: neither engine nor context goes away
  {
    std::lock_guard<std::mutex> lk(e.mu);
    if (e.stop) return fail(IBS_ECANCELLED, "engine is shutting down");
  }
  const size_t need = e.mem_need(nq, k, counts_dev, topk_dev);
  // The engine's own buffers (panel planes, step tables) are always held, so a
  // request is refused at once when it could not fit even beside them alone.
  size_t avail;
  {
    std::lock_guard<std::mutex> lk(e.budget_mu);
    avail = e.pool_budget;
  }
  if (ctx->ws_limit) avail = std::min(avail, ctx->ws_limit > e.fixed_bytes ? ctx->ws_limit - e.fixed_bytes : 0);
  if (need > avail) {
    std::lock_guard<std::mutex> lk(e.mu);
    e.stats.rejected++;
    return fail(IBS_EBUSY, "request needs %zu bytes, more than the %zu bytes the serving budget leaves", need, avail);
  }
  auto r = std::make_shared<Request>();
  r->q = nq;
  r->k = k;
  r->user_counts = oc;
  r->user_idx = oi;
  r->user_dist = od;
  r->counts_on_dev = counts_dev;
  r->topk_on_dev = topk_dev;
  if (k > 0 && !topk_dev) {
    r->map_idx = static_cast<int32_t*>(mapped(oi, sizeof(int32_t)));
    r->map_dist = static_cast<double*>(mapped(od, sizeof(double)));
  }
  // A request that the engine can admit at once is early: it takes its memory and
  // its place together, so no request holds memory that one ahead of it in the
  // queue waits for, and its samples go straight to the device when they are many
  // (kDirectBytes).  One behind others that wait for memory, or past the rows of
  // a step, is kept on the host.
  const size_t bytes = (size_t)e.pg.m * (size_t)((nq + 3) / 4);
  r->id = e.next_id.fetch_add(1);
  if (ctx->ws_limit == 0) {
    std::lock_guard<std::mutex> lk(e.mu);
    bool early = !e.stop && e.early_rows + nq <= kMaxRows;
    for (const auto& p : e.pending) early = early && p->early;
    if (early && e.reserve_request(*r, need)) {
      r->early = r->arriving = true;
      e.early_rows += nq;
      e.all[r->id] = r;
      e.pending.push_back(r);
    }
  }
  const bool direct = r->early && e.in && bytes >= kDirectBytes;
  if (!direct || !e.copy_in(*r, q, bytes)) r->host_packed = copy_query(q, bytes);
  {
    std::lock_guard<std::mutex> lk(e.mu);
    if (e.stop) return fail(IBS_ECANCELLED, "engine is shutting down");
    if (r->early) {
      r->arriving = false;
    } else {
      e.all[r->id] = r;
      e.pending.push_back(r);
    }
  }
  e.cv_work.notify_all();
  *id = r->id;
  return IBS_OK;
}

ibs_status serve_fail_steps(ibs_ctx* ctx, int steps) {
  auto eng = engine_of(ctx);
  if (!eng) return fail(IBS_ESTATE, "no panel loaded");
  std::lock_guard<std::mutex> lk(eng->mu);
  eng->failing_steps = steps;
  return IBS_OK;
}

ibs_status serve_set_budget(ibs_ctx* ctx, size_t bytes) {
  auto eng = engine_of(ctx);
  if (!eng) return fail(IBS_ESTATE, "no panel loaded");
  std::lock_guard<std::mutex> lk(eng->budget_mu);
  eng->pool_budget = bytes;
  return IBS_OK;
}

ibs_status serve_wait(ibs_ctx* ctx, uint64_t id, int64_t timeout_ms) {
  auto eng = engine_of(ctx);
  if (!eng) return fail(IBS_ESTATE, "no panel loaded");
  ServeEngine& e = *eng;
  std::unique_lock<std::mutex> lk(e.mu);
  auto it = e.all.find(id);
  if (it == e.all.end()) return fail(IBS_EINVAL, "unknown request id %llu", (unsigned long long)id);
  auto r = it->second;
  auto done = [&] { return r->state == RState::Done; };
  if (timeout_ms < 0) {
    e.cv_done.wait(lk, done);
  } else if (!e.cv_done.wait_for(lk, std::chrono::milliseconds(timeout_ms), done)) {
    return fail(IBS_ETIMEOUT, "request %llu not done after %lld ms", (unsigned long long)id, (long long)timeout_ms);
  }
  e.all.erase(id);
  if (r->status != IBS_OK) return fail(r->status, "request %llu failed with status %d", (unsigned long long)id, r->status);
  return IBS_OK;
}

ibs_status serve_poll(ibs_ctx* ctx, uint64_t id) {
  auto eng = engine_of(ctx);
  if (!eng) return fail(IBS_ESTATE, "no panel loaded");
  ServeEngine& e = *eng;
  std::lock_guard<std::mutex> lk(e.mu);
  auto it = e.all.find(id);
  if (it == e.all.end()) return fail(IBS_EINVAL, "unknown request id");
  return it->second->state == RState::Done ? IBS_OK : IBS_EBUSY;
}

ibs_status serve_stats(ibs_ctx* ctx, ibs_serve_stats* out) {
  auto eng = engine_of(ctx);
  if (!eng) return fail(IBS_ESTATE, "no panel loaded");
  std::lock_guard<std::mutex> lk(eng->mu);
  *out = eng->stats;
  return IBS_OK;
}

// One request, one launch sequence, synchronous: the unbatched baseline.
ibs_status serve_query_sync(ibs_ctx* ctx, const uint8_t* q, int64_t nq, int k, int32_t* oc, int32_t* oi, double* od) {
  DeviceGuard g(ctx->device);
  bool counts_dev = false, topk_dev = false;
  auto eng = engine_of(ctx);
  if (ibs_status s = validate_query(eng, q, nq, k, oc, oi, od, counts_dev, topk_dev)) return s;
  ServeEngine& e = *eng;
  const PlaneGeom pg = e.pg;
  const Geo qg = e.geo(nq);
  const size_t pk = (size_t)pg.m * (size_t)((nq + 3) / 4);
  Request r;
  r.q = nq;
  r.k = k;
  ibs_status st = IBS_OK;
  cudaStream_t s;
  IBS_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  const size_t need = e.mem_need(nq, k, counts_dev, topk_dev);
  if (!e.reserve_request(r, need)) {
    cudaStreamDestroy(s);
    return fail(IBS_ENOMEM, "the serving memory budget is exhausted");
  }
  DevBuf counter;
  if (e.alloc(r.packed, pk, s) || e.alloc(r.planes, qg.bytes, s) || e.alloc(counter, 256, s) ||
      (!counts_dev && e.alloc(r.counts, (size_t)nq * pg.n * 16, s)) ||
      (!topk_dev && k > 0 && (e.alloc(r.tidx, (size_t)nq * k * 4, s) || e.alloc(r.tdist, (size_t)nq * k * 8, s)))) {
    if (counter.p) cudaFreeAsync(counter.p, s);
    e.release(r, s);
    cudaStreamSynchronize(s);
    cudaStreamDestroy(s);
    return fail(IBS_ENOMEM, "device allocation failed");
  }
  int32_t* cnt = counts_dev ? oc : static_cast<int32_t*>(r.counts.p);
  std::vector<int32_t*> outs((size_t)nq);
  for (int64_t row = 0; row < nq; ++row) outs[row] = cnt + (size_t)row * pg.n * 4;
  DevBuf outs_d;
  cudaError_t ce = cudaMallocAsync(&outs_d.p, outs.size() * sizeof(int32_t*), s);
  // the engine's kernel rule: two or more query blocks on the two-SM kernel
  const bool two_sm = e.pair && qg.blocks >= 2;
  SweepPlan pl;
  std::vector<uint8_t> sweep_host;
  if (e.sweep) {
    const int64_t cols[2][2] = {{0, e.pgeo.blocks}, {0, 0}};
    pl = sweep_plan_cross(qg.blocks, cols, pg.m, e.clusters);
    sweep_host.resize(ServeEngine::sweep_list_bytes(pl));
  }
  std::vector<CrossItem> items;
  std::vector<PairItem> pitems;
  const size_t qblock_bytes = (size_t)qg.chunks * e.chunk_block_bytes();
  for (int64_t pb = 0; !e.sweep && pb < e.pgeo.blocks; ++pb) {
    if (two_sm) {
      for (int64_t u = 0; 2 * u < qg.blocks; ++u) {
        PairItem it{};
        it.I0 = (int32_t)(2 * u);
        it.I1 = 2 * u + 1 < qg.blocks ? (int32_t)(2 * u + 1) : -1;
        it.J = (int32_t)pb;
        it.c1 = (int32_t)qg.chunks;
        pitems.push_back(it);
      }
      continue;
    }
    for (int64_t qb = 0; qb < qg.blocks; ++qb) {
      CrossItem it;
      it.qplanes = reinterpret_cast<const uint32_t*>(static_cast<const uint8_t*>(r.planes.p) + qb * qblock_bytes);
      it.row_out = static_cast<int32_t**>(outs_d.p) + qb * e.blk;
      it.q_rows = (int32_t)std::min<int64_t>(e.blk, nq - qb * e.blk);
      it.pb = (int32_t)pb;
      items.push_back(it);
    }
  }
  const size_t item_bytes = e.sweep ? sweep_host.size() : two_sm ? pitems.size() * sizeof(PairItem) : items.size() * sizeof(CrossItem);
  const void* item_src = two_sm ? static_cast<const void*>(pitems.data()) : static_cast<const void*>(items.data());
  DevBuf items_dev, sync_d;
  if (ce == cudaSuccess) ce = cudaMallocAsync(&items_dev.p, item_bytes, s);
  if (ce == cudaSuccess)
    ce = cudaMemcpyAsync(outs_d.p, outs.data(), outs.size() * sizeof(int32_t*), cudaMemcpyHostToDevice, s);
  if (ce == cudaSuccess) {
    if (ptr_kind(q) == PtrKind::Device) ce = cudaMemcpyAsync(r.packed.p, q, pk, cudaMemcpyDeviceToDevice, s);
    else ce = cudaMemcpyAsync(r.packed.p, q, pk, cudaMemcpyHostToDevice, s);
  }
  if (ce == cudaSuccess && !e.sweep)
    ce = cudaMemcpyAsync(items_dev.p, item_src, item_bytes, cudaMemcpyHostToDevice, s);
  if (ce == cudaSuccess) ce = e.build_planes(static_cast<const uint8_t*>(r.packed.p), nq, r.planes.p, s);
  if (ce == cudaSuccess) {
    if (e.sweep) {
      // The scratch and the parts pass from call to call in the streams' order, so
      // that the copies and the operands of one call overlap the kernels of another.
      std::lock_guard<std::mutex> lk(e.sync_mu);
      if (!e.sync_ev)
        ce = cudaEventCreateWithFlags(&e.sync_ev, cudaEventDisableTiming);
      else
        ce = cudaStreamWaitEvent(s, e.sync_ev, 0);
      if (ce == cudaSuccess)
        ce = e.run_sweep(pl, static_cast<const uint8_t*>(r.planes.p), (nq + 63) / 64,
                         static_cast<int32_t* const*>(outs_d.p), nq, sweep_host.data(),
                         static_cast<uint8_t*>(items_dev.p), e.sync_scratch, e.sync_part, sync_d, false, s);
      if (e.sync_ev) {
        const cudaError_t re = cudaEventRecord(e.sync_ev, s);
        if (ce == cudaSuccess) ce = re;
      }
    } else if (two_sm)
      ce = launch_tc_pair_cross(static_cast<const uint8_t*>(e.panel_planes.p), pg.n, e.pgeo.chunks,
                                static_cast<const uint8_t*>(r.planes.p), qg.blocks,
                                static_cast<int32_t* const*>(outs_d.p), nq,
                                static_cast<const PairItem*>(items_dev.p), (int64_t)pitems.size(), ctx->status_dev, s,
                                e.pair_sync((int64_t)pitems.size(), sync_d, false, s));
    else if (e.tc)
      ce = launch_tc_cross(static_cast<const uint8_t*>(e.panel_planes.p), pg.n, e.pgeo.chunks,
                           static_cast<const CrossItem*>(items_dev.p), (int64_t)items.size(),
                           (int)std::min<int64_t>(ctx->num_sms, (int64_t)items.size()), e.fmt,
                           static_cast<int*>(counter.p), ctx->status_dev, s);
    else
      ce = e.cross(static_cast<const CrossItem*>(items_dev.p), (int64_t)items.size(), s);
  }
  if (ce == cudaSuccess && k > 0)
    ce = launch_topk(cnt, nq, pg.n, k, topk_dev ? oi : static_cast<int32_t*>(r.tidx.p),
                     topk_dev ? od : static_cast<double*>(r.tdist.p), s);
  if (ce == cudaSuccess && oc && !counts_dev)
    ce = cudaMemcpyAsync(oc, r.counts.p, (size_t)nq * pg.n * 16, cudaMemcpyDeviceToHost, s);
  if (ce == cudaSuccess && k > 0 && !topk_dev) {
    ce = cudaMemcpyAsync(oi, r.tidx.p, (size_t)nq * k * 4, cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(od, r.tdist.p, (size_t)nq * k * 8, cudaMemcpyDeviceToHost, s);
  }
  if (items_dev.p) cudaFreeAsync(items_dev.p, s);
  if (sync_d.p) cudaFreeAsync(sync_d.p, s);
  if (outs_d.p) cudaFreeAsync(outs_d.p, s);
  if (counter.p) cudaFreeAsync(counter.p, s);
  e.release(r, s);
  cudaError_t se = cudaStreamSynchronize(s);
  if (ce == cudaSuccess) ce = se;
  cudaStreamDestroy(s);
  if (ce != cudaSuccess) st = fail(IBS_ECUDA, "query_sync failed: %s", cudaGetErrorString(ce));
  else if (__atomic_load_n(ctx->status_host, __ATOMIC_SEQ_CST) == kDevTimeout)
    st = fail(IBS_ETIMEOUT, "a bounded device wait timed out");
  return st;
}

}  // namespace ibs

// Attention kernel for batches without dense tiles (decode, tiny verify windows): HBM-bound.
//
// Two CTAs of 160 threads per SM: while one is between tasks (first tiles on their way, merge of
// the warps, output), the other one keeps the SM's loads in flight.  Roles of a CTA:
//   warps 0..3  consumers: 32 keys of every 128-key tile each (stream.cuh)
//   warp  4     producer: takes the next task (the first by block index, the following ones from the
//               head of the queue), copies its Q rows and its description into shared memory while
//               the previous task is still being worked on, and keeps a ring of K and V tiles filled
//               by TMA, its lanes issuing the boxes of a tile's pages side by side
// What bounds it: the bytes of K and V.  96 KiB of tiles per CTA, 192 KiB per SM, are in flight
// (fp8: 80 and 160).  Every wait is bounded and reports a timeout in the status word.
// Measured (device time of one call) against the meta-kernel, whose single CTA per SM drains between
// tasks: 13 requests of 300 - 2500 keys, 32/8 heads 34.9 -> 23.8 us; 24 requests up to 3000 keys, 64/8
// heads 47.5 -> 38.6 us; 64 requests up to 8192 keys, 28/4 heads 101.3 -> 100.0 us, over an fp8 cache 88.5 ->
// 56.6 us.  (With the first task read and its first tiles asked for before the dependency wait 90.6, 0.97 of the copy
// bandwidth by the bytes a batch cannot do without, and 52.6.)
#include <cuda.h>
#include <cuda_runtime.h>

#include "ptx.cuh"
#include "stream.cuh"
#include "xy_kernels.h"

namespace xy {
namespace {

using namespace ptx;

constexpr int kWarpsS = 4;
constexpr int kThreadsS = (kWarpsS + 1) * 32;
// Descriptions of tasks: the one being worked on and up to three that the look-ahead has reached.
constexpr int kTaskSlots = 4;
// Key tiles of the first task that are asked for while the launch before is still running.
constexpr int kPrefetchTiles = 2;

template <bool kFp8>
struct StreamCfg {
  static constexpr int kStageBytes = kFp8 ? 16384 : 32768;
  static constexpr int kStages = kFp8 ? 5 : 3;
  static constexpr int kRing = kStages * kStageBytes;
  static constexpr int kXch = kStreamXchFloats<kWarpsS> * 4;
  static constexpr int kQ = 16 * 256;
  static constexpr int kMl = kWarpsS * 16 * 8;
  static constexpr int kScales = kFp8 ? kScaleSlots * 64 : 0;
  static constexpr int kSmem = kRing + kXch + kQ + kMl + kScales + kTaskSlots * static_cast<int>(sizeof(TaskDesc)) + 16 * kStages + 32;
};

// Two CTAs have to fit the 228 KiB of an SM, each in units of 128 bytes with the 1 KiB that the system takes.
template <bool kFp8>
constexpr bool kTwoPerSm = 2 * ((StreamCfg<kFp8>::kSmem + 127) / 128 * 128 + 1024) <= 228 * 1024;
static_assert(kTwoPerSm<false> && kTwoPerSm<true>, "the grid counts on two CTAs per SM");

template <bool kFp8>
__global__ void __launch_bounds__(kThreadsS, 2)
stream_attention_kernel(const __grid_constant__ RunArgs a, const __grid_constant__ CUtensorMap k_map,
                        const __grid_constant__ CUtensorMap v_map) {
  using Cfg = StreamCfg<kFp8>;
  constexpr int kStages = Cfg::kStages;
  extern __shared__ __align__(1024) uint8_t smem[];
  float* xch = reinterpret_cast<float*>(smem + Cfg::kRing);
  uint8_t* q_gen = smem + Cfg::kRing + Cfg::kXch;
  float* ml = reinterpret_cast<float*>(q_gen + Cfg::kQ);
  float* scale_ring = ml + Cfg::kMl / 4;
  TaskDesc* desc = reinterpret_cast<TaskDesc*>(q_gen + Cfg::kQ + Cfg::kMl + Cfg::kScales);
  uint64_t* bars = reinterpret_cast<uint64_t*>(desc + kTaskSlots);
  int* s_last = reinterpret_cast<int*>(bars + 2 * kStages + 2);
  int* s_failed = s_last + 1;  // a thread has reported a timeout
  int* s_dead = s_last + 2;    // the consumers leave together
  const uint32_t ring = smem_u32(smem), q_smem = smem_u32(q_gen);
  const uint32_t full = smem_u32(bars), empty = full + 8 * kStages, task_full = empty + 8 * kStages, task_free = task_full + 8;

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full + 8 * s, 1);
      mbar_init(empty + 8 * s, kWarpsS);
    }
    mbar_init(task_full, 33);  // lane 0 once the description is written, every lane once its Q chunks have landed
    mbar_init(task_free, kWarpsS);
    *s_failed = 0;
    *s_dead = 0;
    fence_mbar_init();
  }
  if (warp == kWarpsS && lane == 0) {
    prefetch_tensormap(&k_map);
    prefetch_tensormap(&v_map);
  }
  __syncthreads();
  // The producer reads the description of the first task while the launch before is still running: the
  // plan's tables come over by a copy, which this launch is ordered behind in full.
  TaskDesc d{};
  if (warp == kWarpsS) {
    d = a.first[blockIdx.x];
    // Its first key tiles are brought into L2 meanwhile, when HBM would idle: beside the append kernel and
    // between the launches.  The block table may still be written by a kernel before: this is a hint, made from
    // whatever the table holds, with page ids outside the pool left out; the copies below read the table again
    // behind the wait.  For it to come early enough the description is one read, not a chain of three (queue,
    // task, request).  Two steps of eight layers, 13 requests of 300 - 2500 keys with appends: 349 us -> 340 with
    // the hint alone, 313 with both (one tile 312, three 318); 64 requests up to 8192 keys 98 -> 95.5, over an fp8
    // cache 55.9 -> 54.8 (one tile 55.4, three 54.7).  An append kernel that lets this one in before its own wait: 323.
    const int lane_page = kFp8 ? lane : lane >> 1, ppt = kKeyTile >> a.page_shift;
    if (!a.side_by_side && lane_page < ppt) {
      const int npages = (d.rq.kv_len + d.rq.q_len + a.page_size - 1) >> a.page_shift;
      const int32_t* bt = a.block_table + static_cast<int64_t>(d.rq.bt_row) * a.bt_stride;
      int page[kPrefetchTiles];
#pragma unroll
      for (int i = 0; i < kPrefetchTiles; ++i) page[i] = ld_l2(bt + min((d.t.kt_lo + i) * ppt + lane_page, npages - 1));
#pragma unroll
      for (int i = 0; i < kPrefetchTiles; ++i) {
        if (d.t.kt_lo + i < d.t.kt_hi && page[i] >= 0 && page[i] < a.num_pages) {
          tma_prefetch_4d(&k_map, kFp8 ? 0 : (lane & 1) * 64, 0, d.t.kv_head, page[i]);
          tma_prefetch_4d(&v_map, kFp8 ? 0 : (lane & 1) * 64, 0, d.t.kv_head, page[i]);
        }
      }
    }
    __syncwarp();
  }
  // (Beside the dense launch: its CTAs have let this one in only after their own wait.)  What a kernel before may have
  // written is read by ordinary loads from here on; __ldg, which may be moved across the wait, reads the plan's
  // tables alone.
  if (!a.side_by_side) grid_dependency_wait();
  unsigned long long t_start = 0;
  if (threadIdx.x == 0) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_start));
  const int G = a.num_q_heads / a.num_kv_heads;

  if (warp == kWarpsS) {
    // ================================== producer ==========================================
    // `dead` is the same in all lanes, as is everything that decides the warp's way; a lane whose wait for a stage has
    // run out goes on without copies until the vote behind the tile.
    bool dead = false, failed = false;
    if ((ring & 1023u) != 0) {  // the TMA swizzle needs it; dynamic shared memory starts there
      report_timeout(a, s_failed);
      dead = true;
    }
    const int ppt = kKeyTile >> a.page_shift;  // pages per tile
    // bf16: two 64-element boxes per page, lane 2 p + half; fp8: one box per page, lane p
    const int lane_page = kFp8 ? lane : lane >> 1;
    const bool has_box = lane_page < ppt;
    const uint32_t box_bytes = static_cast<uint32_t>(a.page_size) * 128u;
    const uint32_t box_off = kFp8 ? lane_page * box_bytes : (lane & 1) * 16384u + lane_page * box_bytes;
    const uint64_t policy = make_l2_policy_evict_first();
    struct Tile {
      int kv_head, kt, page;
      float ks, vs;
      bool first, valid;
    };
    // A cursor over the CTA's (task, key tile) sequence: a tile's block-table entry is requested
    // three tiles before its copy is issued, which reaches into the next tasks.
    int kt = 0, n_grab = 0;
    const int32_t* bt = a.block_table;
    int npages = 1;
    bool open = false, out = false;
    auto next_tile = [&]() {
      Tile x{0, 0, 0, 1.f, 1.f, false, false};
      if (!open || kt >= d.t.kt_hi) {
        open = false;
        if (out) return x;
        if (n_grab > 0) {  // (the grid has no more CTAs than there are tasks)
          const int grid = static_cast<int>(gridDim.x);
          int k = a.num_tasks;
          if (lane == 0 && a.num_tasks > grid)
            k = grid + static_cast<int>(atomicInc(reinterpret_cast<unsigned*>(a.queue_head), a.queue_wrap));
          k = __shfl_sync(0xffffffffu, k, 0);
          if (k >= a.num_tasks) {
            out = true;
            return x;
          }
          const int ti = __ldg(a.queue + k);
          d.t = a.tasks[ti];
          d.rq = a.reqs[d.t.req];
          d.rq.pad1 = (a.task_unit != nullptr && d.t.part >= 0) ? __ldg(a.task_unit + ti) : -1;
          if (d.rq.pad1 >= 0) {
            d.nsplit = a.units[d.rq.pad1].nsplit;
            d.part0 = a.units[d.rq.pad1].part0;
          }
        }
        ++n_grab;
        if (lane == 0) desc[(n_grab - 1) % kTaskSlots] = d;
        kt = d.t.kt_lo;
        npages = (d.rq.kv_len + d.rq.q_len + a.page_size - 1) >> a.page_shift;
        bt = a.block_table + static_cast<int64_t>(d.rq.bt_row) * a.bt_stride;
        open = true;
        x.first = true;
      }
      x.valid = true;
      x.kv_head = d.t.kv_head;
      x.kt = kt;
      if (has_box) x.page = bt[min(kt * ppt + lane_page, npages - 1)];  // past the end: the last page again
      ++kt;
      return x;
    };
    auto request_scales = [&](Tile& x) {
      if constexpr (kFp8) {
        if (x.valid && has_box) {
          const int64_t si = static_cast<int64_t>(x.page) * a.num_kv_heads + x.kv_head;
          x.ks = a.k_scale[si];
          x.vs = a.v_scale[si];
        }
      }
    };
    uint32_t n_tasks = 0;
    // Hands a task (or, with last, the end) to the consumers: description and Q rows.  The previous
    // task's are in its consumers' registers by then (task_free).
    auto publish = [&](bool last) {
      if (n_tasks > 0 && !mbar_wait_warp(task_free, (n_tasks - 1) & 1u, a.status)) {
        report_timeout(a, s_failed);
        dead = true;
        return;
      }
      if (!last) {
        __syncwarp();
        const TaskDesc& nd = desc[n_tasks % kTaskSlots];
        const int rows = nd.t.ntok * G;
        const uint16_t* q0 = a.q + static_cast<int64_t>(nd.rq.q_start + nd.t.tok0) * a.q_token_stride +
                             static_cast<int64_t>(nd.t.kv_head) * G * kHeadDim + (lane & 15) * 8;
        const int rows8 = rows <= 8 ? 8 : 16;  // rows the consumers read; those past the task are zeros
        for (int x = lane >> 4; x < rows8; x += 2) {
          const bool ok = x < rows;
          const uint16_t* src = ok ? q0 + static_cast<int64_t>(x / G) * a.q_token_stride + (x % G) * kHeadDim : q0;
          cp_async_16(q_smem + x * 256u + (((lane & 15u) ^ (x & 7u)) << 4), src, ok);
        }
      } else if (lane == 0) {
        desc[n_tasks % kTaskSlots].t.req = -1;
      }
      ++n_tasks;
      cp_async_mbar_arrive(task_full);
      if (lane == 0) mbar_arrive(task_full);
    };
    RingPos pos{0, 0};
    int n_fill = 0;
    uint32_t k_fills = 0, used = 0, fill_par = 0;
    uint32_t left_out = 0;  // stage whose copy the test hook has left out: nobody hands it back any more
    auto fill = [&](const CUtensorMap* map, const Tile& x, bool is_k) {
      const uint32_t bit = 1u << pos.stage, bar = full + 8 * pos.stage;
      if (used & bit) {
        // wait for the readers of this stage's previous fill
        if (!failed && !mbar_wait_block(empty + 8 * pos.stage, (fill_par >> pos.stage) & 1u, a.status)) {
          report_timeout(a, s_failed);
          failed = true;
        }
        fill_par ^= bit;
      }
      used |= bit;
      if (n_fill++ == a.debug_skip_fill) {  // failure-path test hook: this copy is left out
        left_out = bit;
        pos.advance<kStages>();
        return;
      }
      if constexpr (kFp8) {
        if (is_k) {
          float* slot = scale_ring + (k_fills % kScaleSlots) * 16;
          ++k_fills;
          if (has_box) {
            slot[lane_page] = x.ks;
            slot[8 + lane_page] = x.vs;
          }
          __syncwarp();
        }
      }
      if (lane == 0 && !failed) mbar_arrive_expect_tx(bar, Cfg::kStageBytes);
      __syncwarp();
      if (has_box && !failed)
        tma_load_4d_hint(ring + pos.stage * Cfg::kStageBytes + box_off, map, bar, kFp8 ? 0 : (lane & 1) * 64, 0, x.kv_head,
                         x.page, policy);
      pos.advance<kStages>();
    };
    Tile q0 = next_tile(), q1 = next_tile(), q2 = next_tile();
    request_scales(q0);
    request_scales(q1);
    while (q0.valid && !dead) {
      const Tile cur = q0;
      if (cur.first) publish(false);
      q0 = q1;
      q1 = q2;
      q2 = next_tile();
      request_scales(q1);
      if (!dead) {
        fill(&k_map, cur, true);
        fill(&v_map, cur, false);
        dead = __any_sync(0xffffffffu, failed);
      }
    }
    if (!dead) publish(true);
    // No copy of this CTA may still be in flight when it exits (immediate on the normal path).
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int s = 0; s < kStages; ++s)
      if (used & ~left_out & (1u << s)) mbar_wait_block(full + 8 * s, (fill_par >> s) & 1u, a.status);
  } else {
    // ================================== consumers =========================================
    const float scale_log2 = a.sm_scale * 1.4426950408889634f;
    const StreamRing sr{ring, Cfg::kStageBytes, full, empty};
    auto q_addr = [&](uint32_t row, uint32_t ch) { return q_smem + row * 256u + ((ch ^ (row & 7u)) << 4); };
    RingPos pos{0, 0};
    bool dead = false;
    uint32_t tile_seq = 0;
    for (uint32_t n = 0;; ++n) {
      if (!dead && !mbar_wait_block(task_full, n & 1u, a.status)) {
        report_timeout(a, s_failed);
        dead = true;
      }
      // All warps leave together (a warp whose wait ran out must not keep away from the barriers of
      // a task the others have started); the barrier also keeps the exchange areas of two tasks apart.
      if (dead) *s_dead = 1;
      named_bar_sync(1, kWarpsS * 32);
      if (*reinterpret_cast<volatile int*>(s_dead) != 0) break;
      TaskView tv;
      tv.t = desc[n % kTaskSlots].t;
      tv.rq = desc[n % kTaskSlots].rq;
      if (tv.t.req < 0) break;
      const int unit = tv.rq.pad1;
      const UnitRef ref{desc[n % kTaskSlots].nsplit, desc[n % kTaskSlots].part0};
      auto unit_ref = [&]() { return ref; };
      tv.G = G;
      tv.rows = tv.t.ntok * G;
      auto take_q = [&](auto& w) {
        w.init();
        w.load_q(q_addr, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(task_free);  // description and Q rows are in registers
      };
      if (tv.rows <= 8) {
        StreamWarp<kWarpsS, 1, kFp8> w;
        take_q(w);
        stream_task<kWarpsS, 1, kFp8, kStages>(a, tv, w, sr, xch, ml, pos, dead, scale_log2, scale_ring, tile_seq, unit, unit_ref, warp, 1,
                                               s_last, s_failed);
      } else {
        StreamWarp<kWarpsS, 2, kFp8> w;
        take_q(w);
        stream_task<kWarpsS, 2, kFp8, kStages>(a, tv, w, sr, xch, ml, pos, dead, scale_log2, scale_ring, tile_seq, unit, unit_ref, warp, 1,
                                               s_last, s_failed);
      }
    }
  }
  // Beside the dense launch: that one is waited for here, so that whoever follows this launch follows both.
  unsigned long long t_end = 0;
  if (a.side_by_side) {
    if (threadIdx.x == 0) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_end));
    grid_dependency_wait();
  }
  // The next launch's CTAs come in as these leave.  (Letting them in from the start filled the SMs
  // unevenly: a CTA took whichever slot was free first, 55.3 -> 60.4 us for 64 requests on an fp8 cache.)
  grid_launch_dependents();
  __syncthreads();
  if (threadIdx.x == 0 && blockIdx.x < static_cast<unsigned>(a.num_workers)) {
    unsigned long long now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    unsigned long long* w = a.worker_times + 4 * blockIdx.x;
    const bool add = blockIdx.x < static_cast<unsigned>(a.dense_ctas);  // the dense launch's is there
    if (add) atomicMin(w, t_start); else w[0] = t_start;
    w[1] = now;
    if (!add) w[2] = 0ull;
    w[3] = (a.side_by_side ? t_end : now) - t_start;
  }
  end_of_run(a, s_last, s_failed);
}

}  // namespace

// Up to ctas_per_worker CTAs per worker, never more than tasks.
cudaError_t launch_stream(const RunArgs& a, int64_t num_pages, MetaLaunchCache* cache, cudaStream_t s) {
  const bool fp8 = a.kv_fp8 != 0;
  const int smem = fp8 ? StreamCfg<true>::kSmem : StreamCfg<false>::kSmem;
  auto kernel = fp8 ? stream_attention_kernel<true> : stream_attention_kernel<false>;
  if (!cache->attr_set[4 + fp8]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    cache->attr_set[4 + fp8] = true;
  }
  const cudaError_t e = pool_maps(a, num_pages, cache);
  if (e != cudaSuccess) return e;
  const int slots = a.ctas_per_worker * a.num_workers;
  const int grid = a.num_tasks < slots ? a.num_tasks : slots;
  cache->ctas = grid;
  RunArgs args = a;
  args.num_pages = num_pages;
  args.queue_wrap = static_cast<uint32_t>(a.num_tasks - 1);  // one grab less per CTA for its first task, one more in vain
  return launch_after(kernel, dim3(grid), kThreadsS, smem, s, args, *reinterpret_cast<const CUtensorMap*>(cache->maps[0]),
                      *reinterpret_cast<const CUtensorMap*>(cache->maps[1]));
}

}  // namespace xy

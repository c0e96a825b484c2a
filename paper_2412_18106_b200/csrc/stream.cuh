// Streaming attention (at most 16 packed query rows against a long run of keys: decode, tiny
// verify windows), shared by the meta-kernel and by the kernel for batches without dense tiles.
//
// Each of kWarps consumer warps owns 128 / kWarps keys of every 128-key tile and works on the
// transposed problem with mma.sync.m16n8k16:
//   S^T[keys x rows] = K Q^T      A = 16 keys of K (ldmatrix), B = 8 rows of Q (registers)
//   O^T[d x rows]   += V^T P^T    A = 16 columns of V (ldmatrix.trans), B = P^T (movmatrix)
// Keys, not query rows, fill the 16-row side of the instruction: a decode step has 4 - 8 rows
// (the q heads of one kv head), so with the rows there half of every MMA, of the score registers
// and of the accumulator was padding.  The softmax reference of a row moves only when some score
// exceeds it by 2^8 (one vote per tile); no maximum is reduced otherwise.  An fp8 cache is widened
// to f16 in registers, fragment by fragment, instead of in shared memory.
// Measured inside the meta-kernel against the form with query rows on the 16-row side: 2048-token
// chunk beside 48 decode requests 467 -> 438 us, 64 decode requests 105 -> 101.5 us, over an fp8
// cache 122 -> 86 us, 128 requests on shared prefixes 112 -> 102 us.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "ptx.cuh"
#include "xy_kernels.h"

namespace xy {
namespace {

using namespace ptx;

constexpr float kRescaleThresholdWarp = 8.0f;  // log2 units
constexpr float kLn2 = 0.6931471805599453f;

struct TaskView {
  xy_attn_task t;
  ReqInfo rq;
  int G, rows;
};

// Visibility of key column `col` for new token i (Sections 4.1.2, 4.2.2, 5.2).
__device__ __forceinline__ bool visible(const RunArgs& a, const ReqInfo& rq, int i, int col) {
  if (col > rq.kv_len + i) return false;  // causal frontier; also excludes everything >= L
  if (col < rq.kv_len || rq.mask_kind == XY_MASK_CAUSAL) return true;
  const int jp = col - rq.kv_len;
  const uint64_t w = ld_u64(a.tree_mask + rq.tree_off + static_cast<int64_t>(i) * rq.tree_words + (jp >> 6));
  return (w >> (jp & 63)) & 1ull;
}

// Word 0 of the status block is this run's (zero when it starts, polled by every wait); the sticky word
// is what xy_attn_device_status reads and clears.
__device__ __forceinline__ void report_timeout(const RunArgs& a, int* s_failed = nullptr) {
  if (s_failed != nullptr) *const_cast<volatile int*>(s_failed) = 1;
  atomicExch(a.status, XY_ERR_DEVICE_TIMEOUT);
  atomicExch(a.status + kStatusSticky, XY_ERR_DEVICE_TIMEOUT);
}

// Called by all threads of a CTA that is through with its tasks, behind a barrier; s_failed is set when
// a thread of the CTA has reported a timeout (null: the status word says whether any CTA has).  Leaves
// the status block as the next run expects it (so that no memset has to stand between two runs) and
// clears the time stamps of workers that had no CTA.
//
// A run without a failure has nothing to wait for: the queue head and the count of finished CTAs have
// wrapped to zero by themselves, and the task that completed a unit has put its counter back.  (Finding
// the last CTA instead, to let it clean up, takes a fence and an atomic whose result is waited for: 1.3 -
// 1.7 us on each launch, 10.8 -> 9.5 us for 13 requests of 500 keys.)  After a failure one of the CTAs
// that know of it waits (with a limit) until all others have counted themselves, and cleans up.  If it gives
// up (the others may wait for an SM that another stream's kernels hold), the next one that knows tries; if
// none succeeds the block stays as it is, the sticky word says that a run has failed, and reading that
// (xy_attn_device_status) clears the whole block.
__device__ __forceinline__ void end_of_run(const RunArgs& a, int* s_flag, const int* s_failed) {
  if (blockIdx.x == 0 && a.side_by_side != 1)
    for (int w = max(static_cast<int>(gridDim.x), a.dense_ctas) * 4 + threadIdx.x; w < a.num_workers * 4; w += blockDim.x) a.worker_times[w] = 0ull;
  unsigned* exits = reinterpret_cast<unsigned*>(a.exits);
  const unsigned others = gridDim.x - 1;
  if (a.side_by_side) {
    // Two launches share the status word: the last CTA of the second, which ends behind the first, cleans up.
    if (threadIdx.x == 0) {
      __threadfence();
      *s_flag = atomicInc(exits, others) == others ? 1 : 0;
    }
    __syncthreads();
    if (*s_flag == 0) return;
    __threadfence();
    const bool failed = *const_cast<volatile int32_t*>(a.status) != 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      *a.queue_head = 0;
      if (a.side_by_side == 2) a.status[0] = 0;
    }
    if (failed && a.side_by_side == 2)
      for (int i = threadIdx.x; i < a.num_units; i += blockDim.x) a.unit_count[i] = 0;
    return;
  }
  if (threadIdx.x >= 32) return;
  int failed;
  if (s_failed != nullptr) {
    failed = *const_cast<volatile const int*>(s_failed);
  } else {
    // One lane's reading for the whole warp: another CTA may report a failure between two lanes' loads, and
    // the lanes have to take the same way.
    failed = threadIdx.x == 0 ? *const_cast<volatile const int32_t*>(a.status) : 0;
    failed = __shfl_sync(0xffffffffu, failed, 0);
  }
  if (failed == 0) {
    if (threadIdx.x == 0) atomicInc(exits, others);
    return;
  }
  int clean = 0;
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicExch(a.status + kStatusCleaner, 1) == 0) {
      const int limit = *const_cast<volatile const int32_t*>(a.status + kStatusWaitLimit);
      for (int i = 1; i < limit && !clean; ++i) {  // (a limit of one poll, from a test: none)
        clean = *const_cast<volatile unsigned*>(exits) == others ? 1 : 0;
        if (!clean) __nanosleep(256);
      }
      if (!clean) atomicExch(a.status + kStatusCleaner, 0);
    }
    __threadfence();
  }
  if (__shfl_sync(0xffffffffu, clean, 0)) {
    for (int i = threadIdx.x; i < a.num_units; i += 32) a.unit_count[i] = 0;
    if (threadIdx.x == 0) *a.queue_head = a.status[0] = a.status[kStatusCleaner] = 0;
    __threadfence();
    __syncwarp();
  }
  if (threadIdx.x == 0) atomicInc(exits, others);
}

// A ring of shared-memory stages as its readers see it.
struct RingPos {
  int stage;
  uint32_t phase;
  template <int kStages>
  __device__ __forceinline__ void advance() {
    if (++stage == kStages) {
      stage = 0;
      phase ^= 1u;
    }
  }
};

// The part of a merge unit that its tasks do not hold themselves.
struct UnitRef {
  int nsplit, part0;
};

// Merge of a split unit (the cross-task Update stage of Section 4.2.1) by the task of the unit that
// finished last: rows <= 16, one warp per row.  Lane c holds LSE_c of splits c, c + 32, ...; the
// weights are broadcast, and the partial rows are read eight at a time straight from L2.
template <int kWarps>
__device__ __forceinline__ void merge_unit_in_kernel(const RunArgs& a, const UnitRef& u, const TaskView& tv, int warp, int lane) {
  const int rows = tv.rows, ns = u.nsplit;
  for (int x = warp; x < rows; x += kWarps) {
    const float* lse_c = a.lse_part + u.part0 + x;  // split c: + c * rows
    const float4* o_c = reinterpret_cast<const float4*>(a.o_part) + (static_cast<int64_t>(u.part0) + x) * (kHeadDim / 4) + lane;
    float mx = -INFINITY;
    float first = -INFINITY;  // LSE of split `lane`
    for (int c = lane; c < ns; c += 32) {
      const float v = __ldcg(lse_c + static_cast<int64_t>(c) * rows);
      if (c == lane) first = v;
      mx = fmaxf(mx, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float z = first != -INFINITY ? __expf(first - mx) : 0.f;
    for (int c = lane + 32; c < ns; c += 32) {
      const float v = __ldcg(lse_c + static_cast<int64_t>(c) * rows);
      if (v != -INFINITY) z += __expf(v - mx);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const float lse = mx + logf(z);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < ns; c0 += 8) {
      if (c0 > 0 && (c0 & 31) == 0)
        first = c0 + lane < ns ? __ldcg(lse_c + static_cast<int64_t>(c0 + lane) * rows) : -INFINITY;
      float w[8];
      float4 v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int c = c0 + e;
        const float lc = __shfl_sync(0xffffffffu, first, c & 31);
        w[e] = c < ns && lc != -INFINITY ? __expf(lc - lse) : 0.f;
        // an empty split (weight 0) is not read
        v[e] = w[e] != 0.f ? __ldcg(o_c + static_cast<int64_t>(c) * rows * (kHeadDim / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        acc.x += w[e] * v[e].x;
        acc.y += w[e] * v[e].y;
        acc.z += w[e] * v[e].z;
        acc.w += w[e] * v[e].w;
      }
    }
    const int64_t token = tv.rq.q_start + tv.t.tok0 + x / tv.G;
    const int head = tv.t.kv_head * tv.G + x % tv.G;
    uint2 packed;
    packed.x = pack_bf16(acc.x, acc.y);
    packed.y = pack_bf16(acc.z, acc.w);
    *reinterpret_cast<uint2*>(a.o + token * a.o_token_stride + head * kHeadDim + lane * 4) = packed;
    if (lane == 0) a.lse[token * a.num_q_heads + head] = lse;
  }
}

// The stage layout of a bf16 tile: element (key, d) at (d / 64) * 16 KiB + key * 128 B +
// (((d % 64) / 8) ^ (key % 8)) * 16 B; of an fp8 tile: key * 128 B + ((d / 16) ^ (key % 8)) * 16 B.
template <bool kFp8>
__device__ __forceinline__ uint32_t tile_chunk(uint32_t key, uint32_t chunk16) {
  if constexpr (kFp8) return key * 128u + ((chunk16 ^ (key & 7u)) << 4);
  return (chunk16 >> 3) * 16384u + key * 128u + (((chunk16 & 7u) ^ (key & 7u)) << 4);
}

// (not volatile: the compiler may interleave the MMAs with the loads and the softmax)
template <bool kF16>
__device__ __forceinline__ void mma_free(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if constexpr (kF16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Transpose of the 8 x 8 matrix of 16-bit elements whose row i, columns 2j, 2j+1 thread 4i + j holds.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// State of one consumer warp for one task with at most 8 * NR rows.
template <int kWarps, int NR, bool kFp8>
struct StreamWarp {
  static constexpr int U = 8 / kWarps;  // 16-key groups of a tile this warp owns
  float o[8][NR][4];         // O^T: columns d of m-tile x rows 8 nr + 2 (lane % 4), + 1
  float m[NR][2], l[NR][2];  // softmax reference (the same in the whole warp) and this thread's part of the sum
  float qf[NR][2];           // fp8: power of two that undoes the row's Q scaling
  uint32_t qb[8][NR][2];     // Q^T fragments

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int mt = 0; mt < 8; ++mt)
#pragma unroll
      for (int nr = 0; nr < NR; ++nr)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[mt][nr][e] = 0.f;
#pragma unroll
    for (int nr = 0; nr < NR; ++nr)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        m[nr][e] = -INFINITY;
        l[nr][e] = 0.f;
        qf[nr][e] = 1.f;
      }
  }

  // Q rows from shared memory; addr(row, chunk) is the address of 16-byte chunk `chunk` of a row.
  // fp8: the contraction index k of a k-step c stands for d = 16 c + 4 (lane % 4) + {0, 1} (k < 8) and
  // + {2, 3} (k >= 8), the order in which ldmatrix hands out the bytes of K; the rows become f16 with
  // a power-of-two factor that brings the row's largest element below 4 (bf16's exponents do not fit).
  template <class Addr>
  __device__ __forceinline__ void load_q(Addr addr, int lane) {
    if constexpr (!kFp8) {
#pragma unroll
      for (int nr = 0; nr < NR; ++nr)
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2)
          ldmatrix_x4(addr(8 * nr + (lane & 7), 2 * ks + (lane >> 3)), qb[ks][nr][0], qb[ks][nr][1], qb[ks + 1][nr][0],
                      qb[ks + 1][nr][1]);
    } else {
      const int g = lane >> 2, t = lane & 3;
#pragma unroll
      for (int nr = 0; nr < NR; ++nr) {
        uint32_t emax = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                       : "=r"(qb[c][nr][0]), "=r"(qb[c][nr][1])
                       : "r"(addr(8 * nr + g, 2 * c + (t >> 1)) + (t & 1) * 8u));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t w = qb[c][nr][e];
            emax = max(emax, max(w & 0x7F80u, (w >> 16) & 0x7F80u));
          }
        }
        emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 1));
        emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 2));
        uint32_t e = emax >> 7;                     // biased exponent of the row's largest element
        e = e == 0 ? 127u : min(max(e, 2u), 253u);  // an all-zero row keeps factor 1
        const float down = __uint_as_float((254u - e) << 23), up = __uint_as_float(e << 23);
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const uint32_t w = qb[c][nr][k];
            qb[c][nr][k] = pack_f16(__uint_as_float(w << 16) * down, __uint_as_float(w & 0xFFFF0000u) * down);
          }
        // the factor of row g -> the threads that hold rows 2 (lane % 4), + 1 as columns of S^T
        qf[nr][0] = __shfl_sync(0xffffffffu, up, 8 * t);
        qf[nr][1] = __shfl_sync(0xffffffffu, up, 8 * t + 4);
      }
    }
  }

  // Fragments of 16 keys (rows key0 ..) of a K or V tile.
  struct Frags {
    uint32_t r[kFp8 ? 4 : 8][4];
  };
  __device__ __forceinline__ void load_k(uint32_t tile, int key0, int lane, Frags& f) {
    const uint32_t key = key0 + (lane & 7) + ((lane >> 3) & 1) * 8;
#pragma unroll
    for (int i = 0; i < (kFp8 ? 4 : 8); ++i)
      ldmatrix_x4(tile + tile_chunk<kFp8>(key, 2 * i + (lane >> 4)), f.r[i][0], f.r[i][1], f.r[i][2], f.r[i][3]);
  }
  __device__ __forceinline__ void load_v(uint32_t tile, int key0, int lane, Frags& f) {
    // bf16: registers 0 .. 3 = keys 0-7 / d 0-7, keys 0-7 / d 8-15, keys 8-15 / d 0-7, keys 8-15 / d 8-15
    // fp8:  keys 0-7, keys 8-15 of a 16-byte chunk, then of the next one (a 16-bit element is two d's)
    const uint32_t lo = (lane >> 3) & 1, hi = lane >> 4;
    const uint32_t key = key0 + (lane & 7) + (kFp8 ? lo : hi) * 8;
#pragma unroll
    for (int i = 0; i < (kFp8 ? 4 : 8); ++i)
      ldmatrix_x4_trans(tile + tile_chunk<kFp8>(key, 2 * i + (kFp8 ? hi : lo)), f.r[i][0], f.r[i][1], f.r[i][2], f.r[i][3]);
  }
  __device__ __forceinline__ static void widen(uint32_t w, uint32_t& lo, uint32_t& hi) {
    lo = e4m3x2_to_f16x2(static_cast<uint16_t>(w & 0xFFFFu));
    hi = e4m3x2_to_f16x2(static_cast<uint16_t>(w >> 16));
  }
  __device__ __forceinline__ void qk(const Frags& f, float (&s)[NR][4]) {
    float t[NR][4];
#pragma unroll
    for (int nr = 0; nr < NR; ++nr)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[nr][e] = t[nr][e] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 8; ks += 2) {
      uint32_t a0[4], a1[4];
      if constexpr (kFp8) {
        const uint32_t(&r)[4] = f.r[kFp8 ? ks / 2 : 0];
        widen(r[0], a0[0], a0[2]);
        widen(r[1], a0[1], a0[3]);
        widen(r[2], a1[0], a1[2]);
        widen(r[3], a1[1], a1[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          a0[e] = f.r[kFp8 ? 0 : ks][e];
          a1[e] = f.r[kFp8 ? 0 : ks + 1][e];
        }
      }
#pragma unroll
      for (int nr = 0; nr < NR; ++nr) {  // even and odd k-steps: two chains of four
        mma_free<kFp8>(s[nr], a0, qb[ks][nr][0], qb[ks][nr][1]);
        mma_free<kFp8>(t[nr], a1, qb[ks + 1][nr][0], qb[ks + 1][nr][1]);
      }
    }
#pragma unroll
    for (int nr = 0; nr < NR; ++nr)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[nr][e] += t[nr][e];
  }
  __device__ __forceinline__ void pv(const Frags& f, const uint32_t (&pb)[NR][2]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t a0[4], a1[4];  // m-tiles 2 i and 2 i + 1
      if constexpr (kFp8) {
        // bytes (key, d) (key, d + 1) (key + 1, d) (key + 1, d + 1) -> pairs of keys; rows 0-7 of the
        // m-tile are the even d's of its 16, rows 8-15 the odd ones
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          widen(__byte_perm(f.r[kFp8 ? i : 0][h], 0u, 0x3120), a0[2 * h], a0[2 * h + 1]);
          widen(__byte_perm(f.r[kFp8 ? i : 0][2 + h], 0u, 0x3120), a1[2 * h], a1[2 * h + 1]);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          a0[e] = f.r[kFp8 ? 0 : 2 * i][e];
          a1[e] = f.r[kFp8 ? 0 : 2 * i + 1][e];
        }
      }
#pragma unroll
      for (int nr = 0; nr < NR; ++nr) {
        mma_free<kFp8>(o[2 * i][nr], a0, pb[nr][0], pb[nr][1]);
        mma_free<kFp8>(o[2 * i + 1][nr], a1, pb[nr][0], pb[nr][1]);
      }
    }
  }

  // Scores (in place, times f and the K scale of the keys' page) -> P^T fragments; tok[nr][e]: token of
  // the thread's rows (mask only).
  template <bool kMask>
  __device__ __forceinline__ void softmax(const RunArgs& a, const ReqInfo& rq, float (&s)[U][NR][4], const float (&f)[NR][2],
                                          const float (&k_scale)[U], const float (&v_scale)[U], int col0,
                                          const int (&tok)[NR][2], int lane, uint32_t (&pb)[U][NR][2]) {
    bool grow = false;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int nr = 0; nr < NR; ++nr)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float v = s[u][nr][e] * (kFp8 ? f[nr][e & 1] * k_scale[u] : f[nr][e & 1]);
          if (kMask && !visible(a, rq, tok[nr][e & 1], col0 + u * 16 + (lane >> 2) + (e >> 1) * 8)) v = -INFINITY;
          s[u][nr][e] = v;
          grow |= v > m[nr][e & 1] + kRescaleThresholdWarp;  // no reference yet (-inf): any finite score
        }
    if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
      for (int nr = 0; nr < NR; ++nr)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float mx = m[nr][e];
#pragma unroll
          for (int u = 0; u < U; ++u) mx = fmaxf(mx, fmaxf(s[u][nr][e], s[u][nr][e + 2]));
#pragma unroll
          for (int w = 4; w < 32; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
          const float al = mx == -INFINITY ? 1.f : ex2(m[nr][e] - mx);
          m[nr][e] = mx;
          l[nr][e] *= al;
#pragma unroll
          for (int mt = 0; mt < 8; ++mt) {
            o[mt][nr][e] *= al;
            o[mt][nr][e + 2] *= al;
          }
        }
    }
#pragma unroll
    for (int nr = 0; nr < NR; ++nr) {
      const float ref0 = m[nr][0] == -INFINITY ? 0.f : m[nr][0], ref1 = m[nr][1] == -INFINITY ? 0.f : m[nr][1];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float p0 = ex2(s[u][nr][0] - ref0), p1 = ex2(s[u][nr][1] - ref1);
        const float p2 = ex2(s[u][nr][2] - ref0), p3 = ex2(s[u][nr][3] - ref1);
        l[nr][0] += p0 + p2;
        l[nr][1] += p1 + p3;
        if constexpr (kFp8) {  // the V scale of the keys' page rides on P (l keeps the unscaled sum)
          pb[u][nr][0] = movmatrix_trans(pack_f16(p0 * v_scale[u], p1 * v_scale[u]));
          pb[u][nr][1] = movmatrix_trans(pack_f16(p2 * v_scale[u], p3 * v_scale[u]));
        } else {
          pb[u][nr][0] = movmatrix_trans(pack_bf16(p0, p1));
          pb[u][nr][1] = movmatrix_trans(pack_bf16(p2, p3));
        }
      }
    }
  }
};

// The ring a task's tiles arrive in: K and V tiles alternate.
struct StreamRing {
  uint32_t base, stage_bytes;  // tile of stage s at base + s * stage_bytes
  uint32_t full, empty;        // barriers of stage s at + 8 s; a stage's readers arrive once per warp
};

constexpr int kScaleSlots = 8;  // fp8: ring of per-tile page scales, [slot][16]: K scales [0..7], V scales [8..15]

// floats of exchange memory the merge of a task's warps needs
template <int kWarps>
constexpr int kStreamXchFloats = kWarps * (kWarps - 1) * (8 / kWarps) * 128;

// One streaming task, run by kWarps consumer warps whose Q fragments are loaded (w).  Keeps the
// warps' online-softmax states apart and merges them through shared memory at the end (the in-CTA
// Update stage of Section 4.2.1): warp w finishes m-tiles [w * 8 / kWarps, + 8 / kWarps), so every
// thread exchanges with the same lane of the other warps (conflict-free, one barrier per 8 rows).
// The caller puts a barrier of the warps between two tasks: the exchange area is read to the end.
template <int kWarps, int NR, bool kFp8, int kStages, typename UnitOf>
__device__ __forceinline__ void stream_task(const RunArgs& a, const TaskView& tv, StreamWarp<kWarps, NR, kFp8>& w,
                                            const StreamRing& ring, float* xch, float* ml, RingPos& pos, bool& dead,
                                            float scale_log2, const float* scale_ring, uint32_t& tile_seq, int unit,
                                            UnitOf&& unit_ref, int warp, int bar_id, int* s_last, int* s_failed) {
  constexpr int U = 8 / kWarps, kMt = 8 / kWarps;
  const int lane = threadIdx.x & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  const int h = tv.rq.kv_len;
  const bool tree = tv.rq.mask_kind == XY_MASK_TREE;
  const int koff = warp * (16 * U);
  int tok[NR][2];
#pragma unroll
  for (int nr = 0; nr < NR; ++nr)
#pragma unroll
    for (int e = 0; e < 2; ++e) tok[nr][e] = tv.t.tok0 + min(8 * nr + t2 + e, tv.rows - 1) / tv.G;
  const int i_max = tv.t.tok0 + tv.t.ntok - 1;
  float f_row[NR][2];
#pragma unroll
  for (int nr = 0; nr < NR; ++nr)
#pragma unroll
    for (int e = 0; e < 2; ++e) f_row[nr][e] = kFp8 ? scale_log2 * w.qf[nr][e] : scale_log2;
  auto wait_full = [&]() {
    if (!dead && !mbar_wait_block(ring.full + 8u * pos.stage, pos.phase, a.status)) {
      report_timeout(a, s_failed);
      dead = true;
    }
  };
  // (a warp that has given up hands no stage back: its copy may be on the way still, and a stage is not armed twice)
  auto release = [&]() {
    __syncwarp();
    if (lane == 0 && !dead) mbar_arrive(ring.empty + 8u * pos.stage);
    pos.advance<kStages>();
  };
  // Tiles that every row of the task sees in full need neither the mask nor the test whether the
  // warp's keys are visible at all; the last tiles (causal frontier, speculative corner) take the
  // general step.
  auto step = [&](int kt, auto tail_tag) {
    constexpr bool kTail = decltype(tail_tag)::value;
    const int col0 = kt * kKeyTile + koff;
    const bool work = kTail ? (col0 <= h + i_max) : true;
    float s[U][NR][4];
    typename StreamWarp<kWarps, NR, kFp8>::Frags f[U];
    wait_full();
    float k_scale[U], v_scale[U];
    if constexpr (kFp8) {  // 16 keys lie in one page (of at least 16 tokens)
      const float* sc = scale_ring + (tile_seq % kScaleSlots) * 16;
      ++tile_seq;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        k_scale[u] = sc[(koff + 16 * u) >> a.page_shift];
        v_scale[u] = sc[8 + ((koff + 16 * u) >> a.page_shift)];
      }
    }
    if (work) {
      const uint32_t tile = ring.base + pos.stage * ring.stage_bytes;
      // all groups' fragments in flight together where the registers allow it (up to 8 rows)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        w.load_k(tile, koff + u * 16, lane, f[u]);
        if (NR > 1) w.qk(f[u], s[u]);
      }
      if (NR == 1) {
#pragma unroll
        for (int u = 0; u < U; ++u) w.qk(f[u], s[u]);
      }
    }
    release();
    wait_full();
    if (work) {
      const uint32_t tile = ring.base + pos.stage * ring.stage_bytes;
      if (NR == 1) {  // in flight during the softmax
#pragma unroll
        for (int u = 0; u < U; ++u) w.load_v(tile, koff + u * 16, lane, f[u]);
      }
      uint32_t pb[U][NR][2];
      if constexpr (kTail) {
        const bool need_mask = tree ? (col0 + 16 * U > h) : (col0 + 16 * U > h + tv.t.tok0 + 1);
        if (need_mask) w.template softmax<true>(a, tv.rq, s, f_row, k_scale, v_scale, col0, tok, lane, pb);
        else w.template softmax<false>(a, tv.rq, s, f_row, k_scale, v_scale, col0, tok, lane, pb);
      } else {
        w.template softmax<false>(a, tv.rq, s, f_row, k_scale, v_scale, col0, tok, lane, pb);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (NR > 1) w.load_v(tile, koff + u * 16, lane, f[u]);
        w.pv(f[u], pb[u]);
      }
    }
    release();
  };
  const int full_cols = tree ? h : h + tv.t.tok0 + 1;  // columns below this are visible to every row
  const int kt_mid = max(tv.t.kt_lo, min(tv.t.kt_hi, full_cols / kKeyTile));
  int kt = tv.t.kt_lo;
  for (; kt < kt_mid; ++kt) step(kt, std::false_type{});
  for (; kt < tv.t.kt_hi; ++kt) step(kt, std::true_type{});

  // ---- merge the warps' partials
#pragma unroll
  for (int nr = 0; nr < NR; ++nr)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float v = w.l[nr][e];
#pragma unroll
      for (int x = 4; x < 32; x <<= 1) v += __shfl_xor_sync(0xffffffffu, v, x);
      if (g == 0) *(reinterpret_cast<float2*>(ml) + warp * 16 + 8 * nr + t2 + e) = make_float2(w.m[nr][e], v);
    }
  float4* x4 = reinterpret_cast<float4*>(xch);
  auto slot = [&](int dst, int src, int k) {  // m-tile k of dst's share, from warp src
    return x4 + ((dst * (kWarps - 1) + (src < dst ? src : src - 1)) * kMt + k) * 32 + lane;
  };
#pragma unroll
  for (int nr = 0; nr < NR; ++nr) {
    if (nr > 0) {
      if (8 * nr >= tv.rows) break;
      named_bar_sync(bar_id, kWarps * 32);  // the exchange area is read before it is written again
    }
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
      const int dst = mt / kMt;
      if (dst != warp) *slot(dst, warp, mt % kMt) = make_float4(w.o[mt][nr][0], w.o[mt][nr][1], w.o[mt][nr][2], w.o[mt][nr][3]);
    }
    named_bar_sync(bar_id, kWarps * 32);
    float M[2] = {-INFINITY, -INFINITY}, L[2] = {0.f, 0.f};
    float4 wm[kWarps];  // m, l of the thread's two rows in every warp
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) {
      wm[ww] = *reinterpret_cast<const float4*>(ml + (ww * 16 + 8 * nr + t2) * 2);
      M[0] = fmaxf(M[0], wm[ww].x);
      M[1] = fmaxf(M[1], wm[ww].z);
    }
    float acc[kMt][4];
#pragma unroll
    for (int k = 0; k < kMt; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[k][e] = 0.f;
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) {
      const float f0 = wm[ww].x == -INFINITY ? 0.f : ex2(wm[ww].x - M[0]);
      const float f1 = wm[ww].z == -INFINITY ? 0.f : ex2(wm[ww].z - M[1]);
      L[0] += f0 * wm[ww].y;
      L[1] += f1 * wm[ww].w;
#pragma unroll
      for (int k = 0; k < kMt; ++k) {
        float4 v;
        if (ww == warp) {
          v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int d = 0; d < kWarps; ++d)  // o[] is indexed by constants only: it lives in registers
            if (d == warp)
              v = make_float4(w.o[d * kMt + k][nr][0], w.o[d * kMt + k][nr][1], w.o[d * kMt + k][nr][2], w.o[d * kMt + k][nr][3]);
        } else {
          v = *slot(warp, ww, k);
        }
        acc[k][0] += f0 * v.x;
        acc[k][1] += f1 * v.y;
        acc[k][2] += f0 * v.z;
        acc[k][3] += f1 * v.w;
      }
    }
    const float inv0 = L[0] > 0.f ? 1.f / L[0] : 0.f, inv1 = L[1] > 0.f ? 1.f / L[1] : 0.f;
    const int r0 = 8 * nr + t2, r1 = r0 + 1;
    auto row_out = [&](int x) {  // packed row -> its bf16 output row
      return a.o + static_cast<int64_t>(tv.rq.q_start + tv.t.tok0 + x / tv.G) * a.o_token_stride +
             (tv.t.kv_head * tv.G + x % tv.G) * kHeadDim;
    };
#pragma unroll
    for (int k = 0; k < kMt; ++k) {
      const int d0 = (warp * kMt + k) * 16;
      const float c0 = acc[k][0] * inv0, c1 = acc[k][1] * inv1, c2 = acc[k][2] * inv0, c3 = acc[k][3] * inv1;
      // bf16 cache: c0, c1 = column d0 + g of rows r0, r1; c2, c3 = column d0 + 8 + g.
      // fp8 cache:  c0, c1 = column d0 + 2 g; c2, c3 = column d0 + 2 g + 1.
      if (tv.t.part < 0) {
        if constexpr (kFp8) {
          if (r0 < tv.rows) *reinterpret_cast<uint32_t*>(row_out(r0) + d0 + 2 * g) = pack_bf16(c0, c2);
          if (r1 < tv.rows) *reinterpret_cast<uint32_t*>(row_out(r1) + d0 + 2 * g) = pack_bf16(c1, c3);
        } else {
          const uint32_t lo = movmatrix_trans(pack_bf16(c0, c1)), hi = movmatrix_trans(pack_bf16(c2, c3));
          if (8 * nr + g < tv.rows) {
            uint16_t* dst = row_out(8 * nr + g) + d0 + t2;
            *reinterpret_cast<uint32_t*>(dst) = lo;
            *reinterpret_cast<uint32_t*>(dst + 8) = hi;
          }
        }
      } else {
        float* dst = a.o_part + static_cast<int64_t>(tv.t.part + r0) * kHeadDim + d0;
        if constexpr (kFp8) {
          if (r0 < tv.rows) *reinterpret_cast<float2*>(dst + 2 * g) = make_float2(c0, c2);
          if (r1 < tv.rows) *reinterpret_cast<float2*>(dst + kHeadDim + 2 * g) = make_float2(c1, c3);
        } else {
          if (r0 < tv.rows) {
            dst[g] = c0;
            dst[g + 8] = c2;
          }
          if (r1 < tv.rows) {
            dst[kHeadDim + g] = c1;
            dst[kHeadDim + g + 8] = c3;
          }
        }
      }
    }
    if (warp == 0 && g == 0) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int x = r0 + e;
        if (x < tv.rows) {
          const float lse = L[e] > 0.f ? (M[e] + log2f(L[e])) * kLn2 : -INFINITY;
          if (tv.t.part < 0)
            a.lse[static_cast<int64_t>(tv.rq.q_start + tv.t.tok0 + x / tv.G) * a.num_q_heads + tv.t.kv_head * tv.G + x % tv.G] = lse;
          else
            a.lse_part[tv.t.part + x] = lse;
        }
      }
    }
  }
  if (unit >= 0) {
    // This task is one KV split of a unit that is merged here: publish the partial, count the
    // finished splits, and let the task that completes the unit merge it.  (Writers: stores, fence,
    // barrier, one atomic; the last one: atomic, fence, loads that bypass L1.)
    __threadfence();
    named_bar_sync(bar_id, kWarps * 32);
    if (warp == 0 && lane == 0) {
      const int ns = unit_ref().nsplit;
      const bool last = atomicAdd(a.unit_count + unit, 1) == ns - 1;
      if (last) a.unit_count[unit] = 0;
      *s_last = last ? 1 : 0;
    }
    named_bar_sync(bar_id, kWarps * 32);
    if (*s_last) {
      __threadfence();
      merge_unit_in_kernel<kWarps>(a, unit_ref(), tv, warp, lane);
    }
  }
}

}  // namespace
}  // namespace xy

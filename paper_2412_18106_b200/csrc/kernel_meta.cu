// Hybrid-batch attention meta-kernel (Meta-Attention, Sections 4.1-4.2), sm_100a.
//
// One persistent CTA per worker (SM) of 384 threads runs meta-tasks until none are left: its own
// Task-Table list (Section 3.3.1) or, for balanced plans, the head of one global queue.  Roles:
//   warps 0..7  consumers: softmax (and, on the warp-level paths, the MMAs), O / LSE output
//   warps 8, 10 producers: take the next task, look page ids up in the block table and stage 128-key
//               K and V tiles (V: warp 10 with tensor memory; a TMA box per page and 64-element half) into a
//               ring of four shared-memory stages; they run ahead across task boundaries
//   warp  9     tcgen05 issuer for both 128-row sub-tiles of a dense task
// Shared-memory tiles use the 128-byte TMA swizzle: element (row, d) of a tile lives at
//   (d / 64) * 16 KiB + row * 128 B + (((d % 64) / 8) ^ (row % 8)) * 16 B + (d % 8) * 2 B,
// which both ldmatrix and the tcgen05 shared-memory descriptors read without bank conflicts.
//
// Two task kinds share the ring:
//   dense     (rows > 16: prefill, verify): two 128-row sub-tiles of packed Q rows; S = Q K^T
//             and O += P V run on tcgen05 with S, P and O in tensor memory, and each consumer
//             warpgroup does the online softmax of one sub-tile (thread = row).  In the variant
//             without tensor memory (kUmma = false) a dense task is one 128-row tile on
//             mma.sync, each consumer warp owning 16 rows.
//   streaming (rows <= 16: decode, tiny verify; stream.cuh): each consumer warp owns 16 keys of every tile
//             against all rows on mma.sync; the warps' partial (m, l, O) are merged in shared
//             memory at the end of the task.  HBM-bound.
// Online softmax runs in the log2 domain in fp32; P is rounded to bf16 before P V; masked scores
// are selected to -inf, never added.  Every wait is bounded and reports a timeout in the status
// word instead of spinning forever.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "ptx.cuh"
#include "stream.cuh"
#include "xy_kernels.h"

namespace xy {

namespace {

using namespace ptx;

constexpr int kConsumerWarps = 8;
constexpr int kConsumerThreads = kConsumerWarps * 32;
constexpr int kThreads = kConsumerThreads + 128;  // + one warpgroup: K producer, MMA issuer, V producer, 1 idle
constexpr int kRegsConsumer = 216;  // setmaxnreg budgets: 256 x 216 + 128 x 72 = 168 x 384, the launch allocation
constexpr int kRegsOther = 72;
constexpr int kStages = 4;  // K tiles in 0 and 2, V tiles in 1 and 3
constexpr int kTileBytes = 32768;  // 2 halves x 128 rows x 128 B
constexpr int kHalfBytes = 16384;
constexpr float kLog2e = 1.4426950408889634f;

struct __align__(8) SmemBarriers {
  uint64_t full[kStages];
  uint64_t empty[kStages];      // released by the eight consumer warps (warp-level MMA paths)
  uint64_t empty_umma[kStages];  // released by a tcgen05.commit of the issuer (tensor-memory path)
};

constexpr int kSmemQ = 2 * kTileBytes;
constexpr int kSmemRing = kStages * kTileBytes;
constexpr int kSmemMl = kConsumerWarps * 16 * 2 * 4;
constexpr int kSmemFp8 = 1024;  // fp8 KV path: per-row Q factors [128] and a ring of per-tile page scales [8][16]
constexpr int kSmemTotal = 1024 /*align slack*/ + kSmemQ + kSmemRing + kSmemMl + sizeof(SmemBarriers) + 128 + 256 + kSmemFp8;

__device__ __forceinline__ uint32_t swz(uint32_t row, uint32_t chunk16 /*0..15*/) {
  return (chunk16 >> 3) * kHalfBytes + row * 128u + (((chunk16 & 7u) ^ (row & 7u)) << 4);
}

struct MetaParams {
  RunArgs a;
};

// One consumer warp of a dense task without tensor memory: 16 packed rows (x0 .. x0+15) against
// NT*8 keys.  Keeps m (log2 domain), l (thread-partial) and O in registers; the Q fragments are
// re-read from shared memory at every k-step to leave registers for the 128-key score tile.
// F16: operands are f16 (the fp8 KV-cache path: K / V widened exactly from e4m3, Q converted with a
// power-of-two factor per row) and the scores carry per-row and per-page factors (FpScale).
struct FpScale {
  float q_lo, q_hi;        // 2^e of the two rows this thread holds: undoes the row's Q pre-scaling
  const float* tile;       // shared memory: [0..7] K scale, [8..15] V scale of the tile's pages
  int page_shift;
};

template <bool F16>
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if constexpr (F16) mma_f16_16816(c, a, b0, b1); else mma_bf16_16816(c, a, b0, b1);
}

template <int NT, bool F16 = false>
struct WarpTile {
  float o[16][4];
  float m_lo, m_hi, l_lo, l_hi;
  uint32_t q_addr, q_row7, q_hi;  // this lane's ldmatrix row address for k-step 0, row % 8, chunk parity

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int n = 0; n < 16; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
    m_lo = m_hi = -INFINITY;
    l_lo = l_hi = 0.f;
  }

  __device__ __forceinline__ void load_q(uint32_t q_smem, int x0, int lane) {
    const int mi = lane >> 3;
    const uint32_t row = x0 + (lane & 7) + (mi & 1) * 8;
    q_addr = q_smem + row * 128u;
    q_row7 = row & 7u;
    q_hi = mi >> 1;
  }

  // S = Q K^T for this warp's keys; returns scores (raw dot products) in s.
  __device__ __forceinline__ void qk(uint32_t k_smem, int koff, int lane, float (&s)[NT][4]) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[n][e] = 0.f;
    const int mi = lane >> 3;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      uint32_t qa[4];
      const uint32_t ch = ks * 2 + q_hi;
      ldmatrix_x4(q_addr + (ch >> 3) * kHalfBytes + (((ch & 7u) ^ q_row7) << 4), qa[0], qa[1], qa[2], qa[3]);
#pragma unroll
      for (int np = 0; np < NT / 2; ++np) {
        const uint32_t key = koff + np * 16 + (lane & 7) + (mi >> 1) * 8;
        uint32_t b0, b1, b2, b3;
        ldmatrix_x4(k_smem + swz(key, ks * 2 + (mi & 1)), b0, b1, b2, b3);
        mma16816<F16>(s[2 * np], qa, b0, b1);
        mma16816<F16>(s[2 * np + 1], qa, b2, b3);
      }
    }
  }

  // Mask + online softmax (Update rescale) on s; leaves P (bf16 A fragments) in p.
  // koff: key offset of s[0] inside the 128-key tile (selects the page whose scales apply)
  __device__ __forceinline__ void softmax(const RunArgs& a, const ReqInfo& rq, float (&s)[NT][4],
                                          uint32_t (&p)[NT / 2][4], int col0, int i_lo, int i_hi,
                                          bool need_mask, float scale_log2, int lane, const FpScale* fs = nullptr,
                                          int koff = 0) {
    float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      float f_lo = scale_log2, f_hi = scale_log2;
      if constexpr (F16) {
        const float ks = fs->tile[(koff + n * 8) >> fs->page_shift];
        f_lo = scale_log2 * fs->q_lo * ks;
        f_hi = scale_log2 * fs->q_hi * ks;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float v = s[n][e] * ((e < 2) ? f_lo : f_hi);
        if (need_mask) {
          const int col = col0 + n * 8 + 2 * (lane & 3) + (e & 1);
          if (!visible(a, rq, (e < 2) ? i_lo : i_hi, col)) v = -INFINITY;
        }
        s[n][e] = v;
        if (e < 2) mx_lo = fmaxf(mx_lo, v); else mx_hi = fmaxf(mx_hi, v);
      }
    }
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
    const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
    // Lazy Update: the reference moves (and O, l are rescaled) only when some row of the warp
    // would otherwise exceed it by more than 2^kRescaleThresholdWarp, or has no reference yet.
    const bool grow = (mn_lo - m_lo > kRescaleThresholdWarp) || (mn_hi - m_hi > kRescaleThresholdWarp) ||
                      (m_lo == -INFINITY && mn_lo != -INFINITY) || (m_hi == -INFINITY && mn_hi != -INFINITY);
    if (__any_sync(0xffffffffu, grow)) {
      const float u_lo = (mn_lo == -INFINITY) ? 0.f : mn_lo, u_hi = (mn_hi == -INFINITY) ? 0.f : mn_hi;
      const float al_lo = ex2(m_lo - u_lo), al_hi = ex2(m_hi - u_hi);
      m_lo = mn_lo;
      m_hi = mn_hi;
      l_lo *= al_lo;
      l_hi *= al_hi;
#pragma unroll
      for (int n = 0; n < 16; ++n) {
        o[n][0] *= al_lo;
        o[n][1] *= al_lo;
        o[n][2] *= al_hi;
        o[n][3] *= al_hi;
      }
    }
    const float use_lo = (m_lo == -INFINITY) ? 0.f : m_lo;
    const float use_hi = (m_hi == -INFINITY) ? 0.f : m_hi;
    float sum_lo = 0.f, sum_hi = 0.f;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const float p0 = ex2(s[n][0] - use_lo), p1 = ex2(s[n][1] - use_lo);
      const float p2 = ex2(s[n][2] - use_hi), p3 = ex2(s[n][3] - use_hi);
      sum_lo += p0 + p1;
      sum_hi += p2 + p3;
      // A fragment of k-step n/2: a0,a1 from the even n-tile, a2,a3 from the odd one
      if constexpr (F16) {
        // the V scale of the key's page rides on P (l keeps the unscaled sum)
        const float vs = fs->tile[8 + ((koff + n * 8) >> fs->page_shift)];
        p[n >> 1][(n & 1) * 2 + 0] = pack_f16(p0 * vs, p1 * vs);
        p[n >> 1][(n & 1) * 2 + 1] = pack_f16(p2 * vs, p3 * vs);
      } else {
        p[n >> 1][(n & 1) * 2 + 0] = pack_bf16(p0, p1);
        p[n >> 1][(n & 1) * 2 + 1] = pack_bf16(p2, p3);
      }
    }
    l_lo += sum_lo;
    l_hi += sum_hi;
  }

  // O += P V for this warp's keys.
  __device__ __forceinline__ void pv(uint32_t v_smem, int koff, int lane, const uint32_t (&p)[NT / 2][4]) {
    const int mi = lane >> 3;
#pragma unroll
    for (int kk = 0; kk < NT / 2; ++kk) {
      const uint32_t key = koff + kk * 16 + (lane & 7) + (mi & 1) * 8;
#pragma unroll
      for (int dp = 0; dp < 8; ++dp) {
        uint32_t b0, b1, b2, b3;
        ldmatrix_x4_trans(v_smem + swz(key, dp * 2 + (mi >> 1)), b0, b1, b2, b3);
        mma16816<F16>(o[2 * dp], p[kk], b0, b1);
        mma16816<F16>(o[2 * dp + 1], p[kk], b2, b3);
      }
    }
  }

  __device__ __forceinline__ void reduce_l() {
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
  }
};

// ------------------------------------------------------------------------------------------
// fp8 KV-cache path (a variant beside the paper's bf16 cache; Section 4.1.1's paged layout with
// e4m3 bytes and one fp32 scale per page and kv head).  A 128-key tile arrives as 16 KiB of
// bytes in the upper half of its 32 KiB stage (row = key, 128 B, 16-byte chunks XOR-swizzled by
// row like every other tile); the warp that is going to read 16 of its rows first widens them in
// place to the f16 tile layout (exact: every e4m3 value is an f16 value).  Two lanes share a row;
// the upper-half destination of a row is the very line its bytes came from, hence the warp-wide
// barrier between the loads and the stores.
__device__ __forceinline__ void widen_rows16(uint32_t stage, int row0, int lane) {
  const uint32_t row = row0 + (lane >> 1), half = lane & 1u, r7 = row & 7u;
  const uint32_t src = stage + kHalfBytes + row * 128u;
  uint4 in[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) in[q] = lds128(src + (((half * 4u + q) ^ r7) << 4));
  // the partner lane's source chunks lie in the line this lane is about to overwrite (and vice versa)
  asm volatile("" ::"r"(in[0].x), "r"(in[1].x), "r"(in[2].x), "r"(in[3].x), "r"(in[0].w), "r"(in[1].w), "r"(in[2].w),
               "r"(in[3].w));
  __syncwarp();
  const uint32_t dst = stage + half * kHalfBytes + row * 128u;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t w[4] = {in[q].x, in[q].y, in[q].z, in[q].w};
    uint32_t h[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      h[2 * k] = e4m3x2_to_f16x2(static_cast<uint16_t>(w[k] & 0xFFFFu));
      h[2 * k + 1] = e4m3x2_to_f16x2(static_cast<uint16_t>(w[k] >> 16));
    }
    sts128(dst + ((static_cast<uint32_t>(2 * q) ^ r7) << 4), make_uint4(h[0], h[1], h[2], h[3]));
    sts128(dst + ((static_cast<uint32_t>(2 * q + 1) ^ r7) << 4), make_uint4(h[4], h[5], h[6], h[7]));
  }
  __syncwarp();
}

// Q rows of the tile in shared memory, bf16 -> f16 in place, each row multiplied by a power of two
// that brings its largest element below 4 (exact in f16 for every element within 2^-14 of the
// row's largest; bf16's exponent range does not fit f16 otherwise).  qmult[row] receives the
// inverse factor, which the softmax folds into the score scale.  kLanesPerRow lanes share a row.
template <int kLanesPerRow>
__device__ __forceinline__ void q_rows_to_f16(uint32_t q_smem, int row0, float* qmult, int lane) {
  constexpr int kChunks = 16 / kLanesPerRow;  // 16-byte chunks (8 elements) per lane
  const uint32_t row = row0 + lane / kLanesPerRow, c0 = (lane % kLanesPerRow) * kChunks;
  uint4 v[kChunks];
  uint32_t emax = 0;
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    v[c] = lds128(q_smem + swz(row, c0 + c));
    const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) emax = max(emax, max(w[k] & 0x7F80u, (w[k] >> 16) & 0x7F80u));
  }
#pragma unroll
  for (int o = 1; o < kLanesPerRow; o <<= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  uint32_t e = emax >> 7;                       // biased exponent of the row's largest element
  e = e == 0 ? 127u : min(max(e, 2u), 253u);    // an all-zero row keeps factor 1
  const float down = __uint_as_float((254u - e) << 23), up = __uint_as_float(e << 23);
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      w[k] = pack_f16(__uint_as_float(w[k] << 16) * down, __uint_as_float(w[k] & 0xFFFF0000u) * down);
    sts128(q_smem + swz(row, c0 + c), make_uint4(w[0], w[1], w[2], w[3]));
  }
  if (lane % kLanesPerRow == 0) qmult[row] = up;
}

// Destination of packed row x: final O / LSE or the fp32 partial.
__device__ __forceinline__ void write_row_pair(const RunArgs& a, const TaskView& tv, int x, int col,
                                               float v0, float v1) {
  if (tv.t.part < 0) {
    const int i = tv.t.tok0 + x / tv.G, head = tv.t.kv_head * tv.G + x % tv.G;
    uint32_t* dst = reinterpret_cast<uint32_t*>(
        a.o + static_cast<int64_t>(tv.rq.q_start + i) * a.o_token_stride + head * kHeadDim + col);
    *dst = pack_bf16(v0, v1);
  } else {
    float2* dst = reinterpret_cast<float2*>(a.o_part + static_cast<int64_t>(tv.t.part + x) * kHeadDim + col);
    *dst = make_float2(v0, v1);
  }
}
__device__ __forceinline__ void write_lse(const RunArgs& a, const TaskView& tv, int x, float lse) {
  if (tv.t.part < 0) {
    const int i = tv.t.tok0 + x / tv.G, head = tv.t.kv_head * tv.G + x % tv.G;
    a.lse[static_cast<int64_t>(tv.rq.q_start + i) * a.num_q_heads + head] = lse;
  } else {
    a.lse_part[tv.t.part + x] = lse;
  }
}

// Debug trace of worker 0: one record per call, (tag << 48) | SM cycle counter.  Compiled in
// only with -DXY_ENABLE_TRACE (the stamps cost issue slots on the critical path).
struct Tracer {
#ifdef XY_ENABLE_TRACE
  unsigned long long* p;
  int n, len;
  // two warps may share a role: each has its half of the records then
  __device__ __forceinline__ void init(const RunArgs& a, int role, bool on, int half = -1) {
    len = half < 0 ? kTraceLen : kTraceLen / 2;
    p = (a.trace != nullptr && blockIdx.x == 0 && on) ? a.trace + role * kTraceLen + max(half, 0) * len : nullptr;
    n = 0;
  }
  __device__ __forceinline__ void operator()(unsigned tag) {
    if (p != nullptr && n < len) p[n++] = (static_cast<unsigned long long>(tag) << 48) | (clock64() & 0xFFFFFFFFFFFFull);
  }
#else
  __device__ __forceinline__ void init(const RunArgs&, int, bool, int = -1) {}
  __device__ __forceinline__ void operator()(unsigned) {}
#endif
};

// ------------------------------------------------------------------------------------------
// tcgen05 dense path.  TMEM columns: S_A [0,128) S_B [128,256) O_A [256,384) O_B [384,512);
// P (bf16, two keys per 32-bit column) overwrites the first 64 columns of its S block.
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemS = 0, kTmemO = 256;
constexpr float kRescaleThreshold = 8.0f;  // log2 units: rescale O only when the row max grows by > 2^8

// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = 128.
constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kIdescQK = kIdescBase;              // A, B K-major
constexpr uint32_t kIdescPV = kIdescBase | (1u << 16);  // B (V) MN-major

// Task indices travel from the producer (which takes them from the global queue) to the other
// roles of the CTA through a small ring in shared memory.
constexpr int kTaskRing = 8;
struct __align__(8) TaskRing {
  uint64_t full[kTaskRing];   // producer -> readers: the slot holds a task index (or -1: no more)
  uint64_t empty[kTaskRing];  // readers -> producer: every reader has taken the slot's index
  int32_t ti[kTaskRing];
};

struct DenseShape {
  int n[2];  // KV tiles sub-tile A / B visits in this task
  int n_all;
};
__device__ __forceinline__ DenseShape dense_shape(const xy_attn_task& t, const ReqInfo& rq, int G) {
  DenseShape d;
  const int rows = t.ntok * G;
#pragma unroll
  for (int X = 0; X < 2; ++X) {
    if (X * 128 >= rows) {
      d.n[X] = 0;
      continue;
    }
    const int last_tok = t.tok0 + (min(rows, (X + 1) * 128) - 1) / G;
    const int frontier = (rq.kv_len + last_tok + 1 + kKeyTile - 1) / kKeyTile;
    d.n[X] = max(0, min(t.kt_hi, frontier) - t.kt_lo);
  }
  d.n_all = t.kt_hi - t.kt_lo;
  return d;
}

struct __align__(8) UmmaBarriers {
  uint64_t q_full[2];  // consumers -> MMA: packed Q sub-tile is in shared memory
  uint64_t s_full[2];  // MMA -> consumers: S = Q K^T of the next KV tile is in TMEM
  uint64_t p_full[2][2];  // consumers -> MMA: [sub-tile][half] 64 keys of P are in TMEM (O rescaled if need be)
  uint64_t o_done[2];  // MMA -> consumers: the task's last P V has completed
  uint64_t drained;  // every MMA the issuer has issued has completed (waited for once, before exit)
  uint32_t tmem_base;
};

static_assert(kStatusWaitLimit == kStatusWaitLimitWord, "one word, two names");
static_assert(sizeof(UmmaBarriers) <= 128, "the shared-memory layout reserves 128 bytes for UmmaBarriers");

template <bool kUmma, bool kFp8>
__global__ void __launch_bounds__(kThreads, 1)
meta_attention_kernel(const __grid_constant__ MetaParams P, const __grid_constant__ CUtensorMap k_map,
                      const __grid_constant__ CUtensorMap v_map) {
  extern __shared__ uint8_t smem_raw[];
  const RunArgs& a = P.a;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t q_smem = base;
  const uint32_t ring = base + kSmemQ;
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  float* ml = reinterpret_cast<float*>(gen_base + kSmemQ + kSmemRing);
  SmemBarriers* bars = reinterpret_cast<SmemBarriers*>(gen_base + kSmemQ + kSmemRing + kSmemMl);
  UmmaBarriers* ub = reinterpret_cast<UmmaBarriers*>(gen_base + kSmemQ + kSmemRing + kSmemMl + sizeof(SmemBarriers));
  TaskRing* tq = reinterpret_cast<TaskRing*>(gen_base + kSmemQ + kSmemRing + kSmemMl + sizeof(SmemBarriers) + 128);
  float* xch = reinterpret_cast<float*>(gen_base + kTileBytes);  // streaming merge area, aliases sub-tile B's Q
  constexpr bool kTwoProducers = kUmma;
  static_assert(!(kUmma && kFp8), "the fp8 KV path runs on the warp-level MMA paths");
  float* qmult = reinterpret_cast<float*>(gen_base + kSmemQ + kSmemRing + kSmemMl + sizeof(SmemBarriers) + 128 + 256);
  float* scale_ring = qmult + 128;  // [kScaleSlots][16]: K scales [0..7], V scales [8..15] of a tile's pages

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 1);
      mbar_init(smem_u32(&bars->empty[s]), kConsumerWarps);
      mbar_init(smem_u32(&bars->empty_umma[s]), 1);
    }
    for (int i = 0; i < kTaskRing; ++i) {
      mbar_init(smem_u32(&tq->full[i]), 1);
      mbar_init(smem_u32(&tq->empty[i]), kConsumerWarps + (kUmma ? 1 : 0) + (kTwoProducers ? 1 : 0));
    }
    for (int X = 0; X < 2; ++X) {
      mbar_init(smem_u32(&ub->q_full[X]), 4);
      mbar_init(smem_u32(&ub->s_full[X]), 1);
      mbar_init(smem_u32(&ub->p_full[X][0]), 4);
      mbar_init(smem_u32(&ub->p_full[X][1]), 4);
      mbar_init(smem_u32(&ub->o_done[X]), 1);
    }
    mbar_init(smem_u32(&ub->drained), 1);
    fence_mbar_init();
  }
  if (kUmma && warp == kConsumerWarps + 1) {
    tmem_alloc(smem_u32(&ub->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  if (warp == kConsumerWarps && lane == 0) {
    prefetch_tensormap(&k_map);
    prefetch_tensormap(&v_map);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // (What a kernel before may have written, block table, scales, masks, Q, is read by ordinary loads behind this wait.
  // __ldg is for the plan's tables alone: it asks for data that nobody writes while this kernel lives, and may be
  // moved across the wait.)
  grid_dependency_wait();
  if (a.side_by_side) grid_launch_dependents();  // every launch before this one is complete: the second may run
  if (threadIdx.x == 0) {
    unsigned long long now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    a.worker_times[4 * blockIdx.x] = now;
  }
  const uint32_t tmem = kUmma ? __shfl_sync(0xffffffffu, ub->tmem_base, 0) : 0u;

  const bool dynamic = a.dynamic != 0;
  const int t_begin = dynamic ? 0 : a.worker_off[blockIdx.x], t_end = dynamic ? 0 : a.worker_off[blockIdx.x + 1];
  // Every role but warp 8 reads its task sequence here: the worker's own Task-Table list (static dealing) or
  // the indices that warp 8 publishes (dynamic dealing).  Warp-uniform.  All readers follow the sequence to its -1,
  // after a failure too: the consumers meet at barriers inside a task, and one that left alone would keep the
  // others waiting there.  So only warp 8 ends a sequence early (grab below), and a reader's wait for it does
  // not give up with the others.
  int seq_static = t_begin;
  uint32_t n_read = 0;
  bool feed_dead = false;
  auto next_task = [&]() -> int {  // called by all 32 lanes
    if (!dynamic) return seq_static < t_end ? seq_static++ : -1;
    const uint32_t slot = n_read % kTaskRing;
    if (!feed_dead && !mbar_wait_handoff(smem_u32(&tq->full[slot]), (n_read / kTaskRing) & 1u)) {
      report_timeout(a);
      feed_dead = true;
    }
    const int ti = feed_dead ? -1 : tq->ti[slot];
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&tq->empty[slot]));
    ++n_read;
    return ti;
  };
  const int G = a.num_q_heads / a.num_kv_heads;
  const float scale_log2 = a.sm_scale * kLog2e;

  if (warp >= kConsumerWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == kConsumerWarps || (kTwoProducers && warp == kConsumerWarps + 2)) {
      static_assert(kStages == 4, "two stages per producer");
      // ================================ producers ======================================
      // With tensor memory warp 8 stages the K tiles (even stages of the ring) and warp 10 the V tiles (odd
      // stages), without it warp 8 both; warp 8 also takes the tasks and hands them to everyone.  Each lane
      // issues the box of one page and half, side by side.  (One lane that did all of it, K and V, box after box,
      // needed 1600 - 2400 cycles per fill of an empty ring, about what a streaming tile takes its SM, and its
      // per-stage state cost the consumers of the variant with tensor memory 90 bytes of spills, now none; the other
      // two spill about 400 bytes either way.  One lane / two warps: 2048-token chunk beside 48 decode requests 435 ->
      // 401 us, serving mix of 96 requests 5023 -> 4746, 4 prompts of 4096 tokens 1126 -> 1077, 32 verify trees 878 ->
      // 854, two planned steps of a tiny batch 36.9 -> 34.0; a chunk of 512 tokens on 2048 beside 40 decode
      // requests of 1000 - 8000 on pages of 16 tokens 229 -> 115, of 32 tokens 157 -> 109.  The variants without tensor
      // memory are bound by their consumers' instructions, and there the second warp is no gain for all: that mix on
      // the bf16 variant, one lane / one warp / two, 273 / 258 / 255 us, on pages of 16 tokens 376 / 302 / 294, over an
      // fp8 cache 345 / 291 / 283; but with requests of 200 - 2000 121 / 120 / 127 and 147 / 133 / 156.  One warp does
      // both there, which nowhere measured is slower than one lane.)
      const int op = warp == kConsumerWarps ? 0 : 1;
      bool dead = false;  // the same in all lanes, as is everything that decides the warp's way
      // Of this producer's stages: who read the stage last (bit set: the tcgen05 path), the parity
      // to wait for on each of its two empty barriers, and of its `full` phase that the latest fill completes;
      // a stage that was never filled needs no wait.
      uint32_t used = 0, last_umma = 0, ph_cons = 0, ph_umma = 0, fill_par = 0;
      uint32_t left_out = 0;  // stage whose copy the test hook has left out: nobody hands it back any more
      Tracer tr;
      tr.init(a, 3, lane == 0, kTwoProducers ? op : -1);
      const int ppt = kKeyTile >> a.page_shift;  // pages per 128-key tile
      const int lane_page = kFp8 ? lane : lane >> 1;
      const bool has_box = lane_page < ppt;
      const uint32_t page_bytes = static_cast<uint32_t>(a.page_size) * 128u;
      // bf16: two 64-element boxes per page; e4m3 bytes: one box per page (128 B per key) into the upper half of the stage
      const uint32_t box_off = (kFp8 ? kHalfBytes : (lane & 1) * kHalfBytes) + lane_page * page_bytes;
      const int box_x = kFp8 ? 0 : (lane & 1) * 64;
      const uint64_t pol_stream = make_l2_policy_evict_first(), pol_keep = make_l2_policy_evict_last();
      // A cursor over the worker's (task, key tile) sequence.  The block-table entries of a tile are
      // requested three tiles before the tile is issued, so their global-memory latency (and the
      // task / request loads at a task boundary) never sits between a stage's release and its
      // TMA: that latency would otherwise add to every refill of the ring.
      struct Tile {
        int kv_head, page;  // page: of this lane's box
        float ks, vs;       // fp8: that page's K and V scale
        bool by_umma, valid;
      };
      int f_ti = t_begin, f_kt = 0, f_hi = 0, f_head = 0, f_npages = 1;
      uint32_t n_pub = 0;
      bool f_done = false;
      // Next task of this worker: its own list, or the head of the global queue (published by warp 8 to the
      // other roles through the ring; -1 is published once, when the queue is exhausted).
      auto grab = [&]() -> int {
        if (op == 1) return next_task();
        if (!dynamic) return f_ti < t_end ? f_ti++ : -1;
        int ti = -1;
        if (lane == 0 && !dead) {
          const int k = static_cast<int>(atomicInc(reinterpret_cast<unsigned*>(a.queue_head), a.queue_wrap));
          if (k < a.num_tasks) ti = __ldg(a.queue + k);
        }
        ti = __shfl_sync(0xffffffffu, ti, 0);
        const uint32_t slot = n_pub % kTaskRing;
        // (the readers come this far whatever fails: they do not stop before the -1)
        if (n_pub >= kTaskRing && !mbar_wait_handoff(smem_u32(&tq->empty[slot]), ((n_pub / kTaskRing) - 1u) & 1u)) {
          report_timeout(a);
          dead = true;
        }
        __syncwarp();
        if (lane == 0) {
          tq->ti[slot] = ti;
          mbar_arrive(smem_u32(&tq->full[slot]));
        }
        ++n_pub;
        return ti;
      };
      const int32_t* f_bt = a.block_table;
      bool f_umma = false, f_open = false;
      auto next_tile = [&]() {
        Tile x{0, 0, 1.f, 1.f, false, false};
        while (!f_open || f_kt >= f_hi) {
          if (f_done) return x;
          const int ti = grab();
          if (ti < 0) {
            f_done = true;
            return x;
          }
          const xy_attn_task t = a.tasks[ti];
          const ReqInfo rq = a.reqs[t.req];
          f_kt = t.kt_lo;
          f_hi = t.kt_hi;
          f_head = t.kv_head;
          f_npages = (rq.kv_len + rq.q_len + a.page_size - 1) >> a.page_shift;
          f_bt = a.block_table + static_cast<int64_t>(rq.bt_row) * a.bt_stride;
          f_umma = kUmma && t.kind == 0;
          f_open = true;
        }
        x.valid = true;
        x.kv_head = f_head;
        x.by_umma = f_umma;
        if (has_box) x.page = f_bt[min(f_kt * ppt + lane_page, f_npages - 1)];  // past the end: the last page again
        ++f_kt;
        return x;
      };
      // fp8: the page's scales are requested one step after its block-table entry (which they depend
      // on) and used one step later still.
      auto request_scales = [&](Tile& x) {
        if constexpr (kFp8) {
          if (op == 0 && x.valid && has_box) {
            const int64_t si = static_cast<int64_t>(x.page) * a.num_kv_heads + x.kv_head;
            x.ks = a.k_scale[si];
            x.vs = a.v_scale[si];
          }
        }
      };
      // Fill this producer's next stage once its previous reader has released it.
      int n = 0;  // tiles staged so far
      auto fill = [&](const Tile& x, int op) {
        const uint32_t stage = 2 * (n % (kStages / 2)) + op, bit = 1u << stage;
        const uint32_t full = smem_u32(&bars->full[stage]);
        if (used & bit) {
          bool ok;
          if (last_umma & bit) {
            ok = mbar_wait_warp(smem_u32(&bars->empty_umma[stage]), (ph_umma >> stage) & 1u, a.status);
            ph_umma ^= bit;
          } else {
            ok = mbar_wait_warp(smem_u32(&bars->empty[stage]), (ph_cons >> stage) & 1u, a.status);
            ph_cons ^= bit;
          }
          if (!ok) {
            report_timeout(a);
            dead = true;
            return;
          }
          fill_par ^= bit;
        }
        used |= bit;
        last_umma = x.by_umma ? (last_umma | bit) : (last_umma & ~bit);
        // Failure-path test hook (xy_attn_debug_inject): this worker leaves out one copy, so that the stage's `full`
        // barrier does not complete and the readers' bounded waits run out.
        if (2 * n + op == a.debug_skip_fill) {
          left_out = bit;
          return;
        }
        tr(1 + op);
        if constexpr (kFp8) {
          // the K fill also leaves the K and V scales of the tile's pages in the tile's scale slot,
          // before the arrive that the readers' wait synchronises with
          if (op == 0) {
            float* slot = scale_ring + (n % kScaleSlots) * 16;
            if (has_box) {
              slot[lane_page] = x.ks;
              slot[8 + lane_page] = x.vs;
            }
            __syncwarp();
          }
        }
        if (lane == 0) mbar_arrive_expect_tx(full, kFp8 ? kHalfBytes : kTileBytes);
        __syncwarp();
        // K/V of streaming tasks is read once: mark it evict-first in L2 so that it does not
        // push out the K/V that the q tiles of a prefill share through L2 (kept evict-last).
        if (has_box)
          tma_load_4d_hint(ring + stage * kTileBytes + box_off, op == 0 ? &k_map : &v_map, full, box_x, 0, x.kv_head, x.page,
                           x.by_umma ? pol_keep : pol_stream);
      };
      Tile q0 = next_tile(), q1 = next_tile(), q2 = next_tile();
      request_scales(q0);
      request_scales(q1);
      while (q0.valid) {  // (after a failure without copies: the sequence of tasks is ended, or read to its end)
        const Tile cur = q0;
        q0 = q1;
        q1 = q2;
        q2 = next_tile();
        request_scales(q1);
        if (!dead) fill(cur, op);
        if (!kTwoProducers && !dead) fill(cur, 1);
        ++n;
      }
      // No bulk copy of this CTA may still be in flight when it exits: the latest fill of every
      // stage has landed once its `full` phase completes (immediate on the normal path, where the
      // readers have long consumed it; a bounded wait after a failure).
      for (int s = 0; s < kStages; ++s)
        if (used & ~left_out & (1u << s)) mbar_wait_block(smem_u32(&bars->full[s]), (fill_par >> s) & 1u, a.status);
    } else if (kUmma && warp == kConsumerWarps + 1) {
      // ================================ tcgen05 MMA issuer ==============================
      // One warp issues for both 128-row sub-tiles.  Each sub-tile is a chain
      //   S_X(0);  for j: [P_X(j) ready] O_X += P_X(j) V(j);  S_X(j+1) = Q_X K(j+1)^T
      // and the two chains alternate (A, B, A, B, ... skipping a sub-tile that has nothing left),
      // so that one sub-tile's softmax overlaps the other's MMAs.  MMAs execute in order, which is
      // what lets P overwrite S in place.  The whole warp walks the loop and waits, so that every
      // operand is warp-uniform; one elected lane issues.  (Two issuing lanes, one per sub-tile, that
      // took turns through a polled shared-memory word: 3.65 k cycles per pair of 128 x 128 tiles,
      // this form 3.27 k; 4 prompts of 4096 tokens 1172 -> 1136 us, tree verification 916 -> 879 us
      // at the power cap.  Waits that end with a vote and leave the loop on a failure, instead of a flag that each
      // group of MMAs asks: serving mix of 96 requests 4766 -> 4678 us, 4 prompts 1078 -> 1071; the same flag at
      // the hand-overs too: tiny batch 33.2 -> 33.9; a predicate that changes on a failure: trees 860 -> 913.)
      const bool elected = elect_one();
      uint32_t pos = 0;  // ring position: stage = pos % kStages, parity = (pos / kStages) & 1
      uint32_t ph_q = 0, ph_p = 0;  // bit X: parity of sub-tile X's next wait
      Tracer tr;
      tr.init(a, 2, elected);
      // Once a wait has run out nothing more is issued or handed on (a stage's copy may be on the way still, and
      // its producer must not arm it twice): the tasks that are left are only read.
      auto wait = [&](uint32_t bar, uint32_t parity) {
        const bool ok = mbar_wait_warp(bar, parity, a.status);
        tc_fence_after();
        return ok;
      };
      auto wait_full = [&](uint32_t p) { return wait(smem_u32(&bars->full[p % kStages]), (p / kStages) & 1u); };
      // Descriptor halves.  High word (same for every operand here): 8-row groups 1024 B apart,
      // sm_100 descriptor version, 128-byte swizzle.  Low word: start address >> 4 in bits 0-13,
      // leading byte offset >> 4 in bits 16-29 (16 B for the K-major Q / K tiles; 16 KiB, the
      // distance to the second 64-element half, for the MN-major V tile).
      constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
      constexpr uint64_t kDescHi64 = static_cast<uint64_t>(kDescHi) << 32;
      const uint32_t ring_lo = (ring >> 4) & 0x3FFFu, q_lo = (q_smem >> 4) & 0x3FFFu;
      auto commit = [&](uint64_t* bar) {
        if (elected) umma_commit(smem_u32(bar));
      };
      // S_X = Q_X K^T: 8 k-steps of 16 elements, 32 B apart, the second half 16 KiB away
      auto issue_qk = [&](int X, uint32_t p) {
        const uint32_t k0 = (ring_lo + (p % kStages) * (kTileBytes >> 4)) | (1u << 16);
        const uint32_t q0 = (q_lo + X * (kTileBytes >> 4)) | (1u << 16);
        if (elected) {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            const uint32_t off = (ks >> 2) * (kHalfBytes >> 4) + (ks & 3) * 2;
            umma_ss64(tmem + kTmemS + X * 128, kDescHi64 | (q0 + off), kDescHi64 | (k0 + off), kIdescQK, ks > 0 ? 1u : 0u);
          }
        }
        commit(&ub->s_full[X]);
      };
      // O_X (+)= P_X V with P in TMEM, in two halves of 64 keys: the first half is issued while
      // the softmax warps are still exponentiating the second.  V (MN-major): 8 k-steps of 16
      // keys, 2 KiB apart.
      auto issue_pv = [&](int X, uint32_t p, int half, bool accumulate) {
        const uint32_t v0 = (ring_lo + (p % kStages) * (kTileBytes >> 4)) | ((kHalfBytes >> 4) << 16);
        if (elected) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int ks = half * 4 + k;
            umma_ts64(tmem + kTmemO + X * 128, tmem + kTmemS + X * 128 + ks * 8, kDescHi64 | (v0 + ks * 128), kIdescPV,
                      (accumulate || ks > 0) ? 1u : 0u);
          }
        }
      };
      int ti = next_task();
      for (; ti >= 0; ti = next_task()) {
        const xy_attn_task t = a.tasks[ti];
        const uint32_t n_all = t.kt_hi - t.kt_lo;
        const uint32_t pos0 = pos;
        pos += 2 * n_all;
        if (t.kind == 1) continue;  // streaming tasks never touch the tensor-memory path
        const ReqInfo rq = a.reqs[t.req];
        const DenseShape ds = dense_shape(t, rq, G);
        const int n_max = max(ds.n[0], ds.n[1]);
        if (n_max == 0) continue;
#pragma unroll
        for (int X = 0; X < 2; ++X) {
          if (ds.n[X] == 0) continue;
          // q_full first: streaming tasks are skipped without a look at the ring, so this warp may be
          // several fills of a stage ahead, where the parity of `full` says nothing.  Q is there once
          // the consumers are through with every earlier task, that is, with every earlier fill.
          if (!wait(smem_u32(&ub->q_full[X]), (ph_q >> X) & 1u)) goto given_up;
          ph_q ^= 1u << X;
          if (!wait_full(pos0)) goto given_up;
          issue_qk(X, pos0);
        }
        commit(&bars->empty_umma[pos0 % kStages]);
        for (int j = 0; j < n_max; ++j) {
          const uint32_t pv = pos0 + 2 * j + 1, pk = pv + 1;
          if (!wait_full(pv)) goto given_up;
#pragma unroll
          for (int X = 0; X < 2; ++X) {
            if (j >= ds.n[X]) continue;
            const bool more = j + 1 < ds.n[X];
            if (!wait(smem_u32(&ub->p_full[X][0]), (ph_p >> X) & 1u)) goto given_up;
            tr(12);
            issue_pv(X, pv, 0, j > 0);
            if (more && !wait_full(pk)) goto given_up;
            if (!wait(smem_u32(&ub->p_full[X][1]), (ph_p >> X) & 1u)) goto given_up;  // second half of P
            ph_p ^= 1u << X;
            issue_pv(X, pv, 1, true);
            if (!more) commit(&ub->o_done[X]);
            // the stage goes back to the producer behind its last reader
            if (X == 1 || j >= ds.n[1]) commit(&bars->empty_umma[pv % kStages]);
            if (more) {
              issue_qk(X, pk);
              if (X == 1 || j + 1 >= ds.n[1]) commit(&bars->empty_umma[pk % kStages]);
            }
            tr(16);
          }
        }
      }
    given_up:
      if (ti >= 0) report_timeout(a);
      while (ti >= 0) ti = next_task();
      // Tensor memory is freed after the final barrier: no MMA of this thread may still be in
      // flight then.  On the normal path they completed long ago (immediate); after a failure
      // this is a bounded wait.
      commit(&ub->drained);
      mbar_wait_block(smem_u32(&ub->drained), 0u, a.status);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsConsumer));
    // ================================ consumers ========================================
    RingPos pipe{0, 0};
    bool dead = false;
    uint32_t ph_s = 0, ph_o = 0;  // this warpgroup's s_full / o_done parities
    uint32_t tile_seq = 0;        // key tiles consumed so far (fp8: selects the scale slot)
    Tracer tr;
    tr.init(a, warp >> 2, (threadIdx.x & 127) == 0);
    const int X = warp >> 2;       // sub-tile this warpgroup owns on the tcgen05 path
    // Time this worker spends in dense / streaming tasks, kept by thread 0 in shared memory.
    __shared__ unsigned long long acct_ns[2], acct_prev;
    __shared__ int acct_kind;
    if (threadIdx.x == 0) {
      acct_ns[0] = acct_ns[1] = 0ull;
      acct_kind = -1;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(acct_prev));
    }
    auto account = [&](int kind_now) {  // called by thread 0 at every task boundary
      unsigned long long now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (acct_kind >= 0) acct_ns[acct_kind] += now - acct_prev;
      acct_prev = now;
      acct_kind = kind_now;
    };
    for (int ti = next_task(); ti >= 0; ti = next_task()) {
      TaskView tv;
      tv.t = a.tasks[ti];
      tv.rq = a.reqs[tv.t.req];
      tv.G = G;
      tv.rows = tv.t.ntok * G;
      const int h = tv.rq.kv_len;
      const bool tree = tv.rq.mask_kind == XY_MASK_TREE;
      const bool stream = tv.t.kind == 1;
      if (threadIdx.x == 0) account(stream ? 1 : 0);
      tr(30);

      if (kUmma && !stream) {
        // ---------------- dense on tcgen05: this thread owns packed row x of sub-tile X ----
        const DenseShape ds = dense_shape(tv.t, tv.rq, G);
        {  // the ring moves on without us: 2 n_all positions
          const uint32_t np = static_cast<uint32_t>(pipe.stage) + 2u * static_cast<uint32_t>(ds.n_all);
          pipe.stage = static_cast<int>(np % kStages);
          pipe.phase ^= (np / kStages) & 1u;
        }
        const int r = (warp & 3) * 32 + lane;
        const int x = X * 128 + r;
        const bool exists = X * 128 < tv.rows;
        const bool valid = x < tv.rows;
        if (!exists) continue;
        // A warp whose 32 rows all lie past the tile's last row has nothing to compute: it only
        // keeps step with the hand-offs (its rows of Q are zero, so are its rows of S, P and O).
        const bool warp_active = X * 128 + (warp & 3) * 32 < tv.rows;
        const int nX = ds.n[X];
        const int i_row = tv.t.tok0 + min(x, tv.rows - 1) / G;
        if (nX == 0) {  // a KV split that lies wholly above this sub-tile's causal frontier
          if (valid) {
            for (int c = 0; c < kHeadDim; c += 2) write_row_pair(a, tv, x, c, 0.f, 0.f);
            write_lse(a, tv, x, -INFINITY);
          }
          continue;
        }
        // packed Q sub-tile -> shared memory, then hand it to the async proxy
        {
          // Thread t copies 16-byte chunk (t & 15) of rows (t >> 4) + 8 it; the (token, head) of
          // a row advances by 8 packed rows per step, so one division per task suffices.
          tr(31);
          const int t128 = threadIdx.x & 127;
          const int ch = t128 & 15;
          const int x0 = X * 128 + (t128 >> 4);
          int i_q = x0 / G, h_q = x0 - i_q * G;
          const int di = 8 / G, dh = 8 - di * G;
          const uint16_t* qbase = a.q + static_cast<int64_t>(tv.rq.q_start + tv.t.tok0) * a.q_token_stride +
                                  static_cast<int64_t>(tv.t.kv_head) * G * kHeadDim + ch * 8;
#pragma unroll 4
          for (int it = 0; it < 16; ++it) {
            const int rr = (t128 >> 4) + 8 * it;
            const bool ok = X * 128 + rr < tv.rows;
            const uint16_t* src = ok ? qbase + static_cast<int64_t>(i_q) * a.q_token_stride + h_q * kHeadDim : qbase;
            cp_async_16(q_smem + X * kTileBytes + swz(rr, ch), src, ok);
            i_q += di;
            h_q += dh;
            if (h_q >= G) {
              h_q -= G;
              ++i_q;
            }
          }
          tr(32);
          cp_async_commit_wait_all();
          fence_proxy_async_smem();
          __syncwarp();
          tr(29);
          if (lane == 0) mbar_arrive(smem_u32(&ub->q_full[X]));
        }
        const uint32_t lane_base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t t_s = lane_base + kTmemS + X * 128, t_o = lane_base + kTmemO + X * 128;
        const int i_min = tv.t.tok0 + (X * 128) / G;
        float m_ref = -INFINITY, l = 0.f;
        for (int j = 0; j < nX; ++j) {
          const int col0 = (tv.t.kt_lo + j) * kKeyTile;
          tr(20);
          if (!dead && !mbar_wait_block(smem_u32(&ub->s_full[X]), ph_s, a.status)) {
            report_timeout(a);
            dead = true;
          }
          ph_s ^= 1u;
          if (!warp_active) {
            __syncwarp();
            if (lane == 0) {
              mbar_arrive(smem_u32(&ub->p_full[X][0]));
              mbar_arrive(smem_u32(&ub->p_full[X][1]));
            }
            continue;
          }
          tc_fence_after();
          uint32_t sr[128];
          tmem_ld_32x32b_x32(t_s, &sr[0]);
          tmem_ld_32x32b_x32(t_s + 32, &sr[32]);
          tmem_ld_32x32b_x32(t_s + 64, &sr[64]);
          tmem_ld_32x32b_x32(t_s + 96, &sr[96]);
          tr(21);
          tmem_wait_ld();
          tr(22);
          const bool need_mask = tree ? (col0 + kKeyTile > h) : (col0 + kKeyTile > h + i_min + 1);
          if (need_mask) {
            // 128-bit visibility mask of this row for columns col0 .. col0 + 127, built with word
            // operations and applied with one test + select per element (no per-element branches).
            const int nvis = min(max(h + i_row - col0 + 1, 0), kKeyTile);  // causal frontier
            uint64_t v_lo = nvis >= 64 ? ~0ull : ((1ull << nvis) - 1ull);
            uint64_t v_hi = nvis >= 128 ? ~0ull : (nvis <= 64 ? 0ull : ((1ull << (nvis - 64)) - 1ull));
            if (tree) {
              // corner bit of column col is bit (col - h) of the row's ancestor-or-self words;
              // columns below h (the cached prefix) are visible to every row.
              const int jp0 = col0 - h;
              const int wbase = max(jp0, 0) >> 6;
              const uint64_t* mrow = a.tree_mask + tv.rq.tree_off + static_cast<int64_t>(i_row) * tv.rq.tree_words;
              uint64_t w0 = 0ull, w1 = 0ull, w2 = 0ull;
              if (wbase < tv.rq.tree_words) w0 = ld_u64(mrow + wbase);
              if (wbase + 1 < tv.rq.tree_words) w1 = ld_u64(mrow + wbase + 1);
              if (wbase + 2 < tv.rq.tree_words) w2 = ld_u64(mrow + wbase + 2);
              uint64_t t_lo, t_hi;
              if (jp0 >= 0) {
                const int sh = jp0 & 63;
                t_lo = sh ? ((w0 >> sh) | (w1 << (64 - sh))) : w0;
                t_hi = sh ? ((w1 >> sh) | (w2 << (64 - sh))) : w1;
              } else {
                const int pre = -jp0;  // 1 .. 127 prefix columns lead the tile
                if (pre < 64) {
                  t_lo = ((1ull << pre) - 1ull) | (w0 << pre);
                  t_hi = (w0 >> (64 - pre)) | (w1 << pre);
                } else {
                  const int p2 = pre - 64;
                  t_lo = ~0ull;
                  t_hi = p2 ? (((1ull << p2) - 1ull) | (w0 << p2)) : w0;
                }
              }
              v_lo &= t_lo;
              v_hi &= t_hi;
            }
            const uint32_t vm[4] = {static_cast<uint32_t>(v_lo), static_cast<uint32_t>(v_lo >> 32),
                                    static_cast<uint32_t>(v_hi), static_cast<uint32_t>(v_hi >> 32)};
#pragma unroll
            for (int k = 0; k < 128; ++k)
              sr[k] = (vm[k >> 5] & (1u << (k & 31))) ? sr[k] : 0xff800000u;  // -inf, selected (never added)
          }
          float mx;
          {  // eight independent chains of three-input max, then a short tree
            float m8[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) m8[q] = fmaxf(__uint_as_float(sr[q]), __uint_as_float(sr[q + 8]));
#pragma unroll
            for (int k = 16; k < 128; k += 16) {
#pragma unroll
              for (int q = 0; q < 8; ++q)
                m8[q] = max3(m8[q], __uint_as_float(sr[k + q]), __uint_as_float(sr[k + q + 8]));
            }
            mx = max3(max3(m8[0], m8[1], m8[2]), max3(m8[3], m8[4], m8[5]), fmaxf(m8[6], m8[7]));
          }
          tr(23);
          const float m_cand = fmaxf(m_ref, mx * scale_log2);
          bool need = false;
          if (j == 0 || m_ref == -INFINITY) {
            m_ref = m_cand;  // nothing accumulated yet for this row: adopt the max, no rescale
          } else {
            need = m_cand - m_ref > kRescaleThreshold;
          }
          if (__any_sync(0xffffffffu, need)) {
            // Update stage: O *= 2^(m_old - m_new).  The previous P V has completed, because
            // this tile's S was issued behind it on the in-order tensor pipe.
            const float alpha = (m_cand == -INFINITY) ? 1.f : ex2(m_ref - m_cand);
            l *= alpha;
            m_ref = m_cand;
#pragma unroll 1
            for (int c = 0; c < 8; ++c) {  // rare path: small chunks, the 128 scores stay live
              uint32_t orow[16];
              tmem_ld_32x32b_x16(t_o + c * 16, orow);
              tmem_wait_ld();
#pragma unroll
              for (int k = 0; k < 16; ++k) orow[k] = __float_as_uint(__uint_as_float(orow[k]) * alpha);
              tmem_st_32x32b_x16(t_o + c * 16, orow);
            }
          }
          tr(24);
          const float neg_off = (m_ref == -INFINITY) ? 0.f : -m_ref;
          // P = 2^(s * scale - m), two keys packed per 32-bit column, written over sr in place.
          // The scale-and-subtract and the row sum run as packed f32x2 instructions.
          const uint64_t scale2 = pack_f32x2(scale_log2, scale_log2), off2 = pack_f32x2(neg_off, neg_off);
          uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
          for (int half = 0; half < 2; ++half) {
#pragma unroll
            for (int k = half * 32; k < half * 32 + 32; ++k) {
              float x0, x1;
              unpack_f32x2(
                  fma_f32x2(pack_f32x2(__uint_as_float(sr[2 * k]), __uint_as_float(sr[2 * k + 1])), scale2, off2), x0,
                  x1);
              const float p0 = ex2(x0), p1 = ex2(x1);
              sum2[k & 3] = add_f32x2(sum2[k & 3], pack_f32x2(p0, p1));
              sr[k] = pack_bf16(p0, p1);
            }
            // hand this half of P (64 keys, 32 columns) to the MMA issuer
            tmem_st_32x32b_x32(t_s + half * 32, &sr[half * 32]);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ub->p_full[X][half]));
            if (half == 0) tr(25);
          }
          {
            float a0, a1;
            unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), a0, a1);
            l += a0 + a1;
          }
          tr(26);
        }
        // ---- epilogue: O / l -> global
        if (!dead && !mbar_wait_block(smem_u32(&ub->o_done[X]), ph_o, a.status)) {
          report_timeout(a);
          dead = true;
        }
        ph_o ^= 1u;
        tc_fence_after();
        tr(27);
        const float inv = l > 0.f ? 1.f / l : 0.f;
        if (tv.t.part < 0) {
          // Final output.  A thread holds one row, so direct stores would touch 32 rows per warp
          // instruction.  The bf16 rows go through this sub-tile's Q area of shared memory instead
          // (its MMAs have completed; 16-byte chunks XOR-swizzled by row so that neither side has
          // bank conflicts) and leave as row-contiguous 256-byte stores, two rows per instruction.
          uint8_t* stage = gen_base + X * kTileBytes;
          if (warp_active) {
            uint32_t orow[128];  // the whole row with one wait: four loads in flight together
            tmem_ld_32x32b_x32(t_o, &orow[0]);
            tmem_ld_32x32b_x32(t_o + 32, &orow[32]);
            tmem_ld_32x32b_x32(t_o + 64, &orow[64]);
            tmem_ld_32x32b_x32(t_o + 96, &orow[96]);
            tmem_wait_ld();
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              uint4 v;
              v.x = pack_bf16(__uint_as_float(orow[q * 8 + 0]) * inv, __uint_as_float(orow[q * 8 + 1]) * inv);
              v.y = pack_bf16(__uint_as_float(orow[q * 8 + 2]) * inv, __uint_as_float(orow[q * 8 + 3]) * inv);
              v.z = pack_bf16(__uint_as_float(orow[q * 8 + 4]) * inv, __uint_as_float(orow[q * 8 + 5]) * inv);
              v.w = pack_bf16(__uint_as_float(orow[q * 8 + 6]) * inv, __uint_as_float(orow[q * 8 + 7]) * inv);
              *reinterpret_cast<uint4*>(stage + r * 256 + ((q ^ (r & 15)) << 4)) = v;
            }
          }
          __syncwarp();
          if (warp_active) {  // a warp stores only rows it staged itself
            const int ch = lane & 15;
            int rr = (warp & 3) * 32 + (lane >> 4);  // row of the sub-tile this lane stores first
            const int xs = X * 128 + rr;
            int i_o = xs / G, h_o = xs - i_o * G;
            const int di = 2 / G, dh = 2 - di * G;
            uint16_t* obase = a.o + static_cast<int64_t>(tv.rq.q_start + tv.t.tok0) * a.o_token_stride +
                              static_cast<int64_t>(tv.t.kv_head) * G * kHeadDim + ch * 8;
#pragma unroll 4
            for (int it = 0; it < 16; ++it) {
              if (X * 128 + rr < tv.rows) {
                const uint4 v = *reinterpret_cast<const uint4*>(stage + rr * 256 + ((ch ^ (rr & 15)) << 4));
                *reinterpret_cast<uint4*>(obase + static_cast<int64_t>(i_o) * a.o_token_stride + h_o * kHeadDim) = v;
              }
              rr += 2;
              i_o += di;
              h_o += dh;
              if (h_o >= G) {
                h_o -= G;
                ++i_o;
              }
            }
          }
          named_bar_sync(2 + X, 128);  // staging reads done before the next task's Q lands here
        } else if (warp_active) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t orow[32];
            tmem_ld_32x32b_x32(t_o + c * 32, orow);
            tmem_wait_ld();
            if (valid) {
              float4* dst = reinterpret_cast<float4*>(a.o_part + static_cast<int64_t>(tv.t.part + x) * kHeadDim + c * 32);
#pragma unroll
              for (int q = 0; q < 8; ++q)
                dst[q] = make_float4(__uint_as_float(orow[q * 4 + 0]) * inv, __uint_as_float(orow[q * 4 + 1]) * inv,
                                     __uint_as_float(orow[q * 4 + 2]) * inv, __uint_as_float(orow[q * 4 + 3]) * inv);
            }
          }
        }
        if (valid) write_lse(a, tv, x, l > 0.f ? (m_ref + log2f(l)) * kLn2 : -INFINITY);
        tc_fence_before();  // order this task's TMEM reads before the next task's MMAs
        tr(28);
        continue;
      }

      // ---- packed Q tile -> shared memory (rows past the tile are zero-filled)
      // A warpgroup that had no sub-tile in the previous dense task arrives here while the other
      // one may still be computing on its Q tile, which this load overwrites: meet first.
      if (kUmma) named_bar_sync(1, kConsumerThreads);
      {
        const int rows_pad = stream ? 16 : 128;
        for (int c = threadIdx.x; c < rows_pad * 16; c += kConsumerThreads) {
          const int x = c >> 4, ch = c & 15;
          const bool ok = x < tv.rows;
          const int xx = ok ? x : 0;
          const int i = tv.t.tok0 + xx / G, head = tv.t.kv_head * G + xx % G;
          const uint16_t* src =
              a.q + static_cast<int64_t>(tv.rq.q_start + i) * a.q_token_stride + head * kHeadDim + ch * 8;
          cp_async_16(q_smem + swz(x, ch), src, ok);
        }
        cp_async_commit_wait_all();
        named_bar_sync(1, kConsumerThreads);
        if constexpr (kFp8) {
          // dense: the Q rows become f16 with a power-of-two factor per row, each warp its own 16 rows
          if (!stream) {
            q_rows_to_f16<2>(q_smem, warp * 16, qmult, lane);
            named_bar_sync(1, kConsumerThreads);
          }
        }
      }

      if (!kUmma && !stream) {  // (with kUmma every dense task took the tcgen05 path above)
        // ---------------- dense: this warp owns rows x0 .. x0+15 -------------------------
        const int x0 = warp * 16;
        const bool active = x0 < tv.rows;
        WarpTile<16, kFp8> w;
        w.init();
        if (active) w.load_q(q_smem, x0, lane);
        FpScale fs{1.f, 1.f, scale_ring, a.page_shift};
        if constexpr (kFp8) {
          fs.q_lo = qmult[x0 + (lane >> 2)];
          fs.q_hi = qmult[x0 + (lane >> 2) + 8];
        }
        const int r_lo = min(x0 + (lane >> 2), tv.rows - 1), r_hi = min(x0 + (lane >> 2) + 8, tv.rows - 1);
        const int i_lo = tv.t.tok0 + r_lo / G, i_hi = tv.t.tok0 + r_hi / G;
        const int i_min = tv.t.tok0 + min(x0, tv.rows - 1) / G;
        const int i_max = tv.t.tok0 + min(x0 + 15, tv.rows - 1) / G;
        for (int kt = tv.t.kt_lo; kt < tv.t.kt_hi; ++kt) {
          const int col0 = kt * kKeyTile;
          const bool work = active && col0 <= h + i_max;  // mask-aware skip (Section 4.2.2)
          float s[16][4];
          uint32_t p[8][4];
          if (!dead && !mbar_wait_block(smem_u32(&bars->full[pipe.stage]), pipe.phase, a.status)) {
            report_timeout(a);
            dead = true;
          }
          if constexpr (kFp8) {
            // every warp widens 16 keys of the tile, all warps read all of it
            fs.tile = scale_ring + (tile_seq % kScaleSlots) * 16;
            ++tile_seq;
            widen_rows16(ring + pipe.stage * kTileBytes, warp * 16, lane);
            named_bar_sync(1, kConsumerThreads);
          }
          if (work) w.qk(ring + pipe.stage * kTileBytes, 0, lane, s);
          if constexpr (kFp8) fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && !dead) mbar_arrive(smem_u32(&bars->empty[pipe.stage]));
          pipe.advance<kStages>();
          if (work) {
            const bool need_mask = tree ? (col0 + kKeyTile > h) : (col0 + kKeyTile > h + i_min + 1);
            w.softmax(a, tv.rq, s, p, col0, i_lo, i_hi, need_mask, scale_log2, lane, &fs, 0);
          }
          if (!dead && !mbar_wait_block(smem_u32(&bars->full[pipe.stage]), pipe.phase, a.status)) {
            report_timeout(a);
            dead = true;
          }
          if constexpr (kFp8) {
            widen_rows16(ring + pipe.stage * kTileBytes, warp * 16, lane);
            named_bar_sync(1, kConsumerThreads);
          }
          if (work) w.pv(ring + pipe.stage * kTileBytes, 0, lane, p);
          if constexpr (kFp8) fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && !dead) mbar_arrive(smem_u32(&bars->empty[pipe.stage]));
          pipe.advance<kStages>();
        }
        if (active) {
          w.reduce_l();
          const float inv_lo = w.l_lo > 0.f ? 1.f / w.l_lo : 0.f;
          const float inv_hi = w.l_hi > 0.f ? 1.f / w.l_hi : 0.f;
          const int xl = x0 + (lane >> 2), xh = xl + 8;
#pragma unroll
          for (int n = 0; n < 16; ++n) {
            const int col = n * 8 + 2 * (lane & 3);
            if (xl < tv.rows) write_row_pair(a, tv, xl, col, w.o[n][0] * inv_lo, w.o[n][1] * inv_lo);
            if (xh < tv.rows) write_row_pair(a, tv, xh, col, w.o[n][2] * inv_hi, w.o[n][3] * inv_hi);
          }
          if ((lane & 3) == 0) {
            if (xl < tv.rows)
              write_lse(a, tv, xl, w.l_lo > 0.f ? (w.m_lo + log2f(w.l_lo)) * kLn2 : -INFINITY);
            if (xh < tv.rows)
              write_lse(a, tv, xh, w.l_hi > 0.f ? (w.m_hi + log2f(w.l_hi)) * kLn2 : -INFINITY);
          }
        }
        named_bar_sync(1, kConsumerThreads);  // Q tile may be overwritten by the next task
      } else {
        // ---------------- streaming (see stream.cuh) ----
        __shared__ int s_last;
        const int unit = (a.task_unit != nullptr && tv.t.part >= 0) ? a.task_unit[ti] : -1;
        const StreamRing sr{ring + (kFp8 ? kHalfBytes : 0), kTileBytes, smem_u32(&bars->full[0]), smem_u32(&bars->empty[0])};
        auto q_addr = [&](uint32_t row, uint32_t ch) { return q_smem + swz(row, ch); };
        auto unit_ref = [&]() { return UnitRef{a.units[unit].nsplit, a.units[unit].part0}; };
        if (tv.rows <= 8) {
          StreamWarp<kConsumerWarps, 1, kFp8> w;
          w.init();
          w.load_q(q_addr, lane);
          stream_task<kConsumerWarps, 1, kFp8, kStages>(a, tv, w, sr, xch, ml, pipe, dead, scale_log2, scale_ring, tile_seq,
                                                        unit, unit_ref, warp, 1, &s_last, nullptr);
        } else {
          StreamWarp<kConsumerWarps, 2, kFp8> w;
          w.init();
          w.load_q(q_addr, lane);
          stream_task<kConsumerWarps, 2, kFp8, kStages>(a, tv, w, sr, xch, ml, pipe, dead, scale_log2, scale_ring, tile_seq,
                                                        unit, unit_ref, warp, 1, &s_last, nullptr);
        }
        named_bar_sync(1, kConsumerThreads);
      }
    }
    if (threadIdx.x == 0) {
      account(-1);
      a.worker_times[4 * blockIdx.x + 2] = acct_ns[0];
      a.worker_times[4 * blockIdx.x + 3] = acct_ns[1];
    }
  }
  grid_launch_dependents();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    a.worker_times[4 * blockIdx.x + 1] = now;
  }
  if (kUmma && warp == kConsumerWarps + 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  __shared__ int s_flag;
  end_of_run(a, &s_flag, nullptr);
}

#include "kernel_pair.inc"

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// 4-D map over a paged pool [pages, Hkv, B, D]: box = one page of one head, 64 elements wide.
// box_tokens: tokens per box (0: a whole page)
bool encode_pool_map(CUtensorMap* m, const void* pool, int64_t num_pages, int num_kv_heads, int page_size,
                     int64_t page_stride, int64_t head_stride, int64_t token_stride, bool fp8, int box_tokens = 0) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return false;
  // bf16: two boxes of 64 elements per row; e4m3 bytes: one box of 128 - 128 B per row either way
  const cuuint64_t esz = fp8 ? 1 : 2;
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(kHeadDim), static_cast<cuuint64_t>(page_size),
                        static_cast<cuuint64_t>(num_kv_heads), static_cast<cuuint64_t>(num_pages)};
  cuuint64_t strides[3] = {static_cast<cuuint64_t>(token_stride) * esz, static_cast<cuuint64_t>(head_stride) * esz,
                           static_cast<cuuint64_t>(page_stride) * esz};
  cuuint32_t box[4] = {fp8 ? 128u : 64u, static_cast<cuuint32_t>(box_tokens > 0 ? box_tokens : page_size), 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(m, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pool), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace

// The tensor maps of the pools, encoded when the pools differ from those of the last call.
cudaError_t pool_maps(const RunArgs& a, int64_t num_pages, MetaLaunchCache* cache) {
  static_assert(sizeof(CUtensorMap) == 128, "MetaLaunchCache holds a tensor map in 128 bytes");
  const bool fp8 = a.kv_fp8 != 0;
  CUtensorMap* k_map = reinterpret_cast<CUtensorMap*>(cache->maps[0]);
  CUtensorMap* v_map = reinterpret_cast<CUtensorMap*>(cache->maps[1]);
  const bool same = cache->valid && cache->k_pool == a.k_pool && cache->v_pool == a.v_pool &&
                    cache->num_pages == num_pages && cache->page_stride == a.page_stride &&
                    cache->head_stride == a.head_stride && cache->token_stride == a.token_stride &&
                    cache->num_kv_heads == a.num_kv_heads && cache->page_size == a.page_size && cache->fp8 == fp8;
  if (!same) {
    cache->valid = false;
    if (!encode_pool_map(k_map, a.k_pool, num_pages, a.num_kv_heads, a.page_size, a.page_stride, a.head_stride,
                         a.token_stride, fp8) ||
        !encode_pool_map(v_map, a.v_pool, num_pages, a.num_kv_heads, a.page_size, a.page_stride, a.head_stride,
                         a.token_stride, fp8))
      return cudaErrorInvalidValue;
    cache->k_pool = a.k_pool;
    cache->v_pool = a.v_pool;
    cache->num_pages = num_pages;
    cache->page_stride = a.page_stride;
    cache->head_stride = a.head_stride;
    cache->token_stride = a.token_stride;
    cache->num_kv_heads = a.num_kv_heads;
    cache->page_size = a.page_size;
    cache->fp8 = fp8;
    cache->valid = true;
  }
  return cudaSuccess;
}

cudaError_t launch_meta(const RunArgs& a, int64_t num_pages, bool umma, MetaLaunchCache* cache, cudaStream_t s) {
  const bool fp8 = a.kv_fp8 != 0;
  if (fp8) umma = false;
  auto kernel = fp8 ? meta_attention_kernel<false, true>
                    : (umma ? meta_attention_kernel<true, false> : meta_attention_kernel<false, false>);
  const int which = fp8 ? 2 : (umma ? 1 : 0);
  if (!cache->attr_set[which]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTotal);
    if (e != cudaSuccess) return e;
    cache->attr_set[which] = true;
  }
  const cudaError_t e = pool_maps(a, num_pages, cache);
  if (e != cudaSuccess) return e;
  MetaParams P{a};
  const int grid = a.dynamic && a.num_tasks < a.num_workers ? a.num_tasks : a.num_workers;
  cache->ctas = grid;
  P.a.queue_wrap = static_cast<uint32_t>(a.num_tasks + grid - 1);  // every CTA grabs in vain once
  return launch_after(kernel, dim3(grid), kThreads, kSmemTotal, s, P, *reinterpret_cast<const CUtensorMap*>(cache->maps[0]),
                      *reinterpret_cast<const CUtensorMap*>(cache->maps[1]));
}

// Dense tasks on CTA pairs: `a.queue` / `a.num_tasks` / `a.queue_head` describe the dense part of the
// plan's queue.  num_workers CTAs (even) = num_workers / 2 pairs.
cudaError_t launch_pair_dense(const RunArgs& a, int num_workers, int64_t num_pages, MetaLaunchCache* cache,
                              cudaStream_t s) {
  if (num_workers < 2) return cudaErrorInvalidValue;
  if (!cache->attr_set[3]) {
    cudaError_t e = cudaFuncSetAttribute(pair_dense_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTotal);
    if (e != cudaSuccess) return e;
    cache->attr_set[3] = true;
  }
  CUtensorMap* k_map = reinterpret_cast<CUtensorMap*>(cache->pair_maps[0]);
  CUtensorMap* v_map = reinterpret_cast<CUtensorMap*>(cache->pair_maps[1]);
  const bool same = cache->pair_valid && cache->pk_pool == a.k_pool && cache->pv_pool == a.v_pool &&
                    cache->p_num_pages == num_pages && cache->p_page_stride == a.page_stride &&
                    cache->p_head_stride == a.head_stride && cache->p_token_stride == a.token_stride &&
                    cache->p_num_kv_heads == a.num_kv_heads && cache->p_page_size == a.page_size;
  if (!same) {
    cache->pair_valid = false;
    // K: boxes of at most 64 tokens (a CTA stages 64 keys of a tile); V: whole pages, 64 columns
    if (!encode_pool_map(k_map, a.k_pool, num_pages, a.num_kv_heads, a.page_size, a.page_stride, a.head_stride,
                         a.token_stride, false, a.page_size < 64 ? a.page_size : 64) ||
        !encode_pool_map(v_map, a.v_pool, num_pages, a.num_kv_heads, a.page_size, a.page_stride, a.head_stride,
                         a.token_stride, false))
      return cudaErrorInvalidValue;
    cache->pk_pool = a.k_pool;
    cache->pv_pool = a.v_pool;
    cache->p_num_pages = num_pages;
    cache->p_page_stride = a.page_stride;
    cache->p_head_stride = a.head_stride;
    cache->p_token_stride = a.token_stride;
    cache->p_num_kv_heads = a.num_kv_heads;
    cache->p_page_size = a.page_size;
    cache->pair_valid = true;
  }
  MetaParams P{a};
  cache->ctas = num_workers & ~1;
  pair_dense_kernel<<<num_workers & ~1, kThreads, kSmemTotal, s>>>(P, *k_map, *v_map);
  return cudaGetLastError();
}

}  // namespace xy

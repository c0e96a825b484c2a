#include "gemm_choice.h"

#include <algorithm>
#include <cmath>

namespace xy {
namespace {

// Time models, in us.  Fitted to 2 400 timed problems (N 64 .. 128256, K 256 .. 28672 in multiples of 64, 1 ..
// 1536 tokens, weights cycled through so that they come from HBM; B200, 148 SMs): 5 to 6 % rms for each
// kernel.  Terms that overlap are joined by the cube root of the sum of their cubes: their maximum with a
// rounded corner.
int div_up(int a, int b) { return (a + b - 1) / b; }
float join(float a, float b, float c = 0.f, float d = 0.f) { return std::cbrt(a * a * a + b * b * b + c * c * c + d * d * d); }

// Persistent whole-K tiles: waves of K chunks, all operand bytes, all (padded) flops, all stores.
struct TileModel {
  int tm, tn;
  float start, chunk, wave, store, hbm, out, pflops;  // us, us per chunk, per wave, per tile, TB/s, TB/s, PFLOP/s
};
constexpr TileModel kTile128{128, 128, 3.51f, 0.2583f, 0.00f, 0.98f, 7.61f, 2.21f, 1.465f};
constexpr TileModel kTile256{128, 256, 3.64f, 0.3797f, 1.28f, 1.06f, 6.58f, 2.22f, 1.667f};
constexpr TileModel kPair256{256, 256, 0.00f, 0.3214f, 0.00f, 4.92f, 6.06f, 1.91f, 1.756f};
float tile_us(const TileModel& m, int M, int N, int K, int slots) {
  const float fm = M, fn = N, fk = K, tiles = static_cast<float>(div_up(M, m.tm)) * div_up(N, m.tn);
  const float waves = std::ceil(tiles / slots), chunks = div_up(K, 64);
  return m.start + m.store * std::min(M, m.tm) / m.tm +
         join(waves * (chunks * m.chunk + m.wave), 2e-6f * (fn * fk + fm * fk + fm * fn) / m.hbm,
              2e-9f * tiles * m.tm * m.tn * fk / m.pflops, 2e-6f * fm * fn / m.out);
}

// 128 x 128 tiles, K over a cluster: one tile per cluster, so clusters beyond those that fit come as
// another wave (16 tiles of eight slices, of which 15 fit: 24 - 29 us, 15 tiles 17).
float splitk_us(int M, int N, int K, int splits, const GemmDevice& dev) {
  const int tiles = div_up(M, 128) * div_up(N, 128);
  const float waves = div_up(tiles, std::max(1, dev.clusters[splits - 1])), chunks = div_up(div_up(K, 64), splits);
  return 0.26f + join(waves * chunks * 0.2644f, 2e-6f * N * K / 6.86f) + waves * (2.67f * std::min(M, 128) / 128 + 3.83f);
}

// Split of K over a cluster for few tiles and up to 512 tokens (0: none).  Four or more slices pay off from
// 16 chunks per slice on; two or three only when the chain is long (32 chunks per slice), else the reduction
// costs what the shorter chain saves.
int cluster_splits(int M, int N, int K, int sms) {
  if (M > 512) return 0;
  const int64_t tiles = static_cast<int64_t>(div_up(M, 128)) * div_up(N, 128);
  const int k_chunks = div_up(K, 64);
  int splits = static_cast<int>(std::min<int64_t>(kClusterMaxCtas, sms / tiles));
  while (splits >= 2 && k_chunks / splits < (splits >= 4 ? 16 : 32)) --splits;
  return splits >= 2 ? splits : 0;
}

// The kernels that compute C row by row: what every call took before there were weight-major kernels, and
// what they have to beat.
GemmChoice token_major(int M, int N, int K, const GemmDevice& dev) {
  GemmChoice c;
  if (M > 128 && dev.sms >= 2) {
    // 256 x 256 tiles on CTA pairs when the padding of M to 256 rows stays under 15 % and the tiles
    // give at least half of the pairs work: measured best or level with the best from 1024 tokens
    // on (at 4096 tokens QKV 155 -> 143 us, OProj 105 -> 96, GateUp 667 -> 609, Down 369 -> 339).
    const int64_t mp = div_up(M, 256), np = div_up(N, 256);
    if ((mp * 256 - M) * 100 <= 15 * mp * 256 && mp * np * 4 >= dev.sms) {
      c.kernel = kGemmPair;
      c.tile_n = 256;
      c.us = tile_us(kPair256, M, N, K, dev.sms / 2);
      return c;
    }
  }
  c.splits = cluster_splits(M, N, K, dev.sms);
  if (c.splits >= 2) {
    c.kernel = kGemmSplitK;
    c.tile_n = 128;
    c.us = splitk_us(M, N, K, c.splits, dev);
    return c;
  }
  // 128 x 256 tiles read the least of A and W per flop; they are used when they give at least
  // half of the SMs a tile (measured: OProj at 1024 tokens, 128 such tiles, 28 us against 44 us
  // with 128 x 128).  Below that 128 x 128.
  c.splits = 1;
  c.tile_n = static_cast<int64_t>(div_up(M, 128)) * div_up(N, 256) * 2 >= dev.sms ? 256 : 128;
  c.us = tile_us(c.tile_n == 256 ? kTile256 : kTile128, M, N, K, dev.sms);
  return c;
}

// Weight-major kernel.  Per K chunk a CTA pair takes its MMAs (64 cycles per instruction at least) but no
// less than 0.2 us; every wave of tiles also takes its weights' time in HBM; the store of a tile's sums
// overlaps the next tile's chain when tensor memory holds two sets of them; splitting K costs the exchange
// of sums.  (Fitted when a tile's sums were stored by half as many warps: its time is an upper one, and the lines
// below keep to what was measured with it.)
float swap_us(int N, int K, const SwapPlan& p, int fit) {
  const int n_tiles = div_up(N, 256), tiles = p.m_tiles * n_tiles, chunks = div_up(div_up(K, 64), p.splits);
  const bool two_sets = 2 * p.tok <= 512;
  const float mma = 0.001764f * p.halves * std::max(64.f, 0.5f * p.tok / p.halves), mma2 = mma * mma;
  const float chain = chunks * std::sqrt(std::sqrt(mma2 * mma2 + 0.001673f));  // 0.202^4
  const float store = 0.56f + 4.12f * p.tok / 256;
  auto wave = [&](int t) {  // the token tiles of a weight tile share its bytes
    const float body = join(chain, 512e-6f * K * t / p.m_tiles / 6.65f);
    return two_sets ? join(body, store) : 1.19f * body + store;
  };
  const float all = (tiles / fit) * wave(fit) + (tiles % fit ? wave(tiles % fit) : 0.f);
  return 2.96f + join(all, 512e-9f * p.m_tiles * p.tok * n_tiles * K / 1.65f) + (two_sets ? store : 0.f) +
         (p.splits > 1 ? 1.59f : 0.f);
}

// Which cut of a problem the weight-major kernel takes.  These simpler terms find the better cuts (us, with
// them / with the model above: N 6144, K 4096 at 1216 tokens 49.5 / 54.0, N 3584, K 18944 at 820
// 93 / 101, N 16384, K 1024 at 352 16.6 / 18.7); the model above is closer to the kernel's time.  Per K
// chunk a pair takes its MMAs (1.3 of the nominal rate) or an intake of 50 B a clock, whichever is longer;
// splitting pays only while every cluster fits the device at once.
SwapPlan swap_plan(int M, int N, int K, int64_t workspace_bytes, const GemmDevice& dev) {
  SwapPlan best;
  float best_us = 1e30f;
  const int n_tiles = div_up(N, 256), k_chunks = div_up(K, 64);
  const int m_lo = div_up(M, 512);
  for (int m_tiles = m_lo; m_tiles <= m_lo + 4; ++m_tiles) {
    SwapPlan p;
    const int per = div_up(M, m_tiles);
    p.m_tiles = m_tiles;
    p.halves = per > 256 ? 2 : 1;
    p.tok = div_up(per, 16 * p.halves) * 16 * p.halves;
    if ((m_tiles - 1) * p.tok >= M) continue;
    for (p.splits = 1; p.splits <= kSwapMaxSplits; ++p.splits) {
      const int64_t tiles = static_cast<int64_t>(m_tiles) * n_tiles;
      const int cps = div_up(k_chunks, p.splits), fit = dev.pair_clusters[p.splits - 1];
      if (fit < 1) continue;
      if (p.splits > 1 && (tiles > fit || cps < 8 || (p.splits - 1) * cps >= k_chunks ||
                           tiles * p.splits * p.tok * 1024 > workspace_bytes))
        continue;
      const float mma = 4.f * p.halves * std::max(64.f, 0.5f * p.tok / p.halves) * 1.3f, intake = (16384.f + 64.f * p.tok) / 50.f;
      const float chain = cps * std::max(mma, intake) / 1900.f + (2 * p.tok > 512 ? p.tok * 0.010f : 0.f);
      auto wave = [&](int64_t t) { return std::max(chain, 512.f * K * t / (6.3e6f * m_tiles)); };
      const float us = (tiles / fit) * wave(fit) + (tiles % fit ? wave(tiles % fit) : 0.f) + p.tok * 0.006f +
                       (p.splits > 1 ? 1.5f + p.tok * 0.010f : 0.f) + 4.f;
      if (us < 0.98f * best_us) {
        best = p;
        best_us = us;
      }
    }
  }
  if (best.tok > 0) best.us = swap_us(N, K, best, dev.pair_clusters[best.splits - 1]);
  return best;
}

// Weight-streaming kernel: clusters of n CTAs, two CTAs on an SM, that run at once.  Clusters of an even number
// need whole SMs of a GPC, so that as many fit as clusters of half the size at one CTA per SM; the doubled
// answer for their own size is the safe count else.  Measured on a B200 (the first tile count that takes
// a second wave, less one): 148, 92, 71, 55, 45, 37, 33 clusters of 2 .. 8; this says 148, 90, 70, 52, 45, 30, 32.
int small_fit(const GemmDevice& dev, int n) {
  if (n == 1) return 2 * dev.sms;
  const int twice = 2 * dev.clusters[n - 1];
  return n % 2 ? twice : std::min(dev.clusters[n / 2 - 1], twice * 16 / 15);
}

// A CTA's chain of K chunks (what it takes in: 128 rows of W and all tokens, shared between the CTAs of an SM)
// or its wave's weights from HBM, then the exchange of sums or the store.
float small_us(int M, int N, int K, int splits, const GemmDevice& dev) {
  const int tiles = div_up(N, 128), chunks = div_up(div_up(K, 64), splits), tok = div_up(M, 16) * 16, fit = small_fit(dev, splits);
  const float after = splits > 1 ? 1.15f + 5.34f * tok / 128 : 4.50f * tok / 128;
  auto wave = [&](int n) {
    const float per_sm = std::min(2.f, std::max(1.f, static_cast<float>(n) * splits / dev.sms));
    return join(chunks * 0.00421f * (1.54f + per_sm) * (16.f + 0.128f * tok), 256e-6f * n * K / 6.47f) + after;
  };
  const float us = 1.33f + (tiles / fit) * wave(fit) + (tiles % fit ? wave(tiles % fit) : 0.f);
  return splits > 1 || tiles > dev.sms ? us : 1.1f * us;  // a whole chain alone on its SM
}

}  // namespace

GemmChoice choose_gemm(int M, int N, int K, int64_t workspace_bytes, const GemmDevice& dev) {
  if (workspace_bytes < gemm_scratch_bytes(dev.sms)) workspace_bytes = 0;
  GemmChoice c = token_major(M, N, K, dev);
  if (M <= 128) {
    // Up to 128 tokens are bound by the bytes of W, and the kernel that streams them is the faster one but for
    // short chains with many tokens, where its stores and its exchange of sums weigh (us, it / the other:
    // N 16384, K 1024, 128 tokens 14.4 / 10.2; N 12288, K 4096, 128 tokens 27.0 / 24.8).  Its K is cut by the
    // model, at least six chunks per CTA (N 12288, K 4096, 16 tokens: two slices 20.1, three 24.7, whose 96
    // clusters do not fit).  The line, over 640 problems: at 1.03 of the
    // models 7 are more than 2 % slower than the other kernel, at 1.0 one, but 11 that were faster go to the other.
    int best = 0;
    float best_us = 1.03f * c.us;
    const int k_chunks = div_up(K, 64);
    for (int sp = 1; sp <= kClusterMaxCtas && (sp == 1 || sp * 6 <= k_chunks); ++sp) {
      if (small_fit(dev, sp) < 1 || (sp - 1) * div_up(k_chunks, sp) >= k_chunks) continue;  // no CTA without a chunk
      const float us = small_us(M, N, K, sp, dev);
      if (us < best_us) {
        best = sp;
        best_us = us;
      }
    }
    if (best > 0) {
      c.kernel = kGemmSmall;
      c.splits = best;
      c.tile_n = 0;
      c.us = best_us;
    }
    return c;
  }
  if (M <= 1536) {
    // The weight-major kernel where its model is below that of the kernel that would run otherwise.  (From about
    // 1500 tokens on both are bound by the MMAs, and the 256 x 256 tiles overlap their stores.)  The line, from
    // 3 700 measured pairs on two devices: with two sets of sums the kernels are level at 0.97 of the models (0.94
    // - 0.96: 5 % faster, 0.98 - 1.0: 1 % slower), with one set, which power limits sooner, at 0.94 (0.94 - 0.96: 3 %
    // slower, up to 12 %).
    const SwapPlan p = swap_plan(M, N, K, workspace_bytes, dev);
    if (p.tok > 0 && p.us < (2 * p.tok > 512 ? 0.94f : 0.98f) * c.us) {
      c.kernel = kGemmSwap;
      c.swap = p;
      c.splits = p.splits;
      c.tile_n = 0;
      c.us = p.us;
    }
  }
  return c;
}

}  // namespace xy

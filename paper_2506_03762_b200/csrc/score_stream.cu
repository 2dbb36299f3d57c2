// Two walks over all tiles of a score matrix that, unlike the eviction score, need no second pass inside one kernel:
//
//   row statistics   per row of Q the log2 sum of 2^{c w} over the keys it sees, and for the row entropies (Eq. 6) the mean
//                    of x = c w - M under the softmax, M the row's largest c w: with Z = sum of 2^x and T = sum of 2^x x,
//                    H_i = - sum_j a_ij ln a_ij = ln 2 (log2 Z - T / Z).  Parts of a row are kept as (M, Z, T) and merged by
//                    differences of their M: a row's M may be hundreds, its entropy far below 1, and only differences may meet.
//   column sums      the score accumulated over every causal row (Eq. 2-3): per key the sum over all later rows of
//                    2^{c w - L}, L the row's statistic.
//
// One kernel serves both: a CTA keeps one 128-row operand tile (a block of queries; a tile of keys) in shared memory and
// streams the tiles of the other past it (keys; queries).  D = fixed . streamed^T by tcgen05.mma into four TMEM
// accumulators, TMA with 128-byte swizzle on both sides, a thread per TMEM lane: a row's statistics or a key's column sum
// never leave their thread until the run is over, and no CTA waits for another.
//
// What bounds it: 16384 exponentials a tile, 1024 cycles of an SM's special-function unit; products take 512 and the
// copies less.  A tile belongs to one of four groups of four softmax warps, so that four tiles are under way in four
// phases.  Runs (a fixed tile with a stretch of its stream) are dealt out statically, longest first, back and forth over
// the CTAs, which leaves them within a tile or two of one another.  Measured: row entropies of 64 heads x 128 rows x
// 32768 keys 123 us (warp-level products and a triple per tile in global memory: 615); all causal rows of 32 heads x
// 8192 tokens 812 us (64 launches of the two-pass kernel over half-masked tiles: 2150).
#include <cuda.h>

#include "ahakv_internal.cuh"
#include "tc_common.cuh"

namespace ahakv {
namespace {

using namespace tc;

enum Mode { kEntropy, kRowStats, kColumns };

constexpr int kSms = 148;                  // what runs are planned for
constexpr int kStages = 4;                 // streamed-tile ring depth
constexpr int kGroups = 4;                 // groups of four softmax warps
constexpr int kSubTileBytes = 128 * 128;   // 128 rows x 64 16-bit elements, 128-byte swizzled
constexpr int kTileBytes = 2 * kSubTileBytes;
constexpr int kThreads = 32 * (4 + 4 * kGroups);   // TMA, MMA, delivery, row constants; softmax

struct StreamArgs {
  int n, D, bf16, G, Hkv, n_blk;   // n_blk: 128-row tiles of the n tokens
  int rpu, n_runs;                 // runs per fixed tile, runs in all
  // entropy: row blocks of up to 128 stacked observation rows
  int r, hb, n_rb;
  int min_last;
  // all causal rows: heads g0 .. g0 + gs - 1 of each group, BH = B * Hkv
  int BH, g0, gs, n_pad;
  const float* ctab;               // [n_pad] lambda log2(e) per row, zero past n
  float* stat;                     // row statistics, one float a row: entropy [unit][rpu][128]; causal [rpu][BH * gs][n_pad]
  float *z, *t;                    // entropy: `stat` has the M of every part and row, these its Z and T
  const float* neg_l;              // columns: [BH * gs][n_pad], -L per row, -inf past n
  float* s;                        // columns: [bh][split][n]
  int splits, accumulate;
  float inv_g;
  int* status;                     // of the call; entropy: one word a CTA
  long long test_wait_ns;          // test build of the kernel only: what every bounded wait allows
  int test_withhold;               // test build only: the softmax warps of CTA 0 never hand their first run over
  float c[kMaxRows];               // entropy: lambda_i log2(e) per observation row
  int last[kMaxRows];              // and the last key it may see
};

struct Shared {
  float tab_c[4][128], tab_l[4][128];       // columns: constants of the streamed rows, per accumulator
  float stat[2][kGroups][128];              // by run parity: each group's share of a row's (a key's) result
  float z[2][kGroups][128], t[2][kGroups][128];   // entropy: Z and T beside it
  unsigned long long fix_full[2], fix_empty[2];
  unsigned long long str_full[kStages], str_empty[kStages];
  unsigned long long acc_empty[4];          // per accumulator
  // Per group: its m-th tile completes barrier m mod 4.  (A barrier per accumulator would not do: a group can come to wait for
  // a tile of an accumulator whose last tile, another group's, is not complete yet, and a wait by parity cannot tell the
  // phase before that from its own.)
  unsigned long long acc_full[kGroups][4], tab_full[kGroups][4];
  unsigned long long stat_full[2], stat_empty[2];
  uint32_t tmem_slot;
};

// Every wait is bounded; on expiry a role records AHAKV_ERR_TIMEOUT in the status word and leaves, and the others' own waits
// run out in turn.  Like the scoring kernel this one exists twice, for the test of that (ahakv_test_set_wait).
template <bool kTest> __device__ __forceinline__ long long wait_limit(const StreamArgs& a) {
  return kTest ? a.test_wait_ns : kWaitLimitNs;
}
// Row entropies: no kernel runs before this one to clear a status word, so every CTA clears and keeps one of its own, and
// entropy_finish gathers them into the first word of the scratch.
constexpr int kStatusBytes = 1024;
static_assert(kStatusBytes >= (1 + kSms) * (int)sizeof(int), "a word for the call and one for every CTA");

constexpr int kOffFix = 0;
constexpr int kOffStr = 2 * kTileBytes;
constexpr int kSmemTiles = kOffStr + kStages * kTileBytes;
constexpr int kSmemBytes = kSmemTiles + 1024 /*alignment slack*/ + (int)sizeof(Shared);
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");

// One run, decoded by every role for itself.
struct Work {
  int unit, rin, cnt;       // fixed tile, part of its stream, tiles in the part
  int b, fix_row, fix_head;
  int first;                // first tile of the part
  int per_head;             // columns: tiles a query head contributes
  int rows;                 // entropy: live rows
};
template <int kMode>
__device__ __forceinline__ Work decode(const StreamArgs& a, int run) {
  Work w = {};
  if (kMode == kEntropy) {
    w.unit = run / a.rpu;
    w.rin = run - w.unit * a.rpu;
    const int bh = w.unit / a.n_rb, rb = w.unit - bh * a.n_rb, h = bh % a.Hkv;
    w.b = bh / a.Hkv;
    w.rows = a.r <= 128 ? min(a.hb, a.G - rb * a.hb) * a.r : min(128, a.r - rb * 128);
    w.fix_head = a.r <= 128 ? h * a.G + rb * a.hb : h;
    w.fix_row = a.r <= 128 ? 0 : rb * 128;
    w.first = (int)((long long)w.rin * a.n_blk / a.rpu);
    w.cnt = (int)((long long)(w.rin + 1) * a.n_blk / a.rpu) - w.first;
  } else if (kMode == kRowStats) {
    const int heads = a.BH * a.gs, per = heads * a.rpu, k = run / per, rem = run - k * per;
    const int rb = a.n_blk - 1 - k, hd = rem / a.rpu, bh = hd / a.gs;   // the longest rows first
    w.rin = rem - hd * a.rpu;
    w.unit = hd;
    w.b = bh / a.Hkv;
    w.fix_head = (bh % a.Hkv) * a.G + a.g0 + hd % a.gs;
    w.fix_row = rb * 128;
    w.first = (int)((long long)w.rin * (rb + 1) / a.rpu);
    w.cnt = (int)((long long)(w.rin + 1) * (rb + 1) / a.rpu) - w.first;
  } else {
    const int per = a.BH * a.splits, j = run / per, rem = run - j * per;    // the earliest keys are seen by most rows
    w.unit = rem / a.splits;
    w.rin = rem - w.unit * a.splits;
    w.b = w.unit / a.Hkv;
    w.fix_head = w.unit % a.Hkv;
    w.fix_row = j * 128;
    w.per_head = a.n_blk - j;
    const int all = a.gs * w.per_head;
    w.first = (int)((long long)w.rin * all / a.splits);
    w.cnt = (int)((long long)(w.rin + 1) * all / a.splits) - w.first;
  }
  return w;
}
// f(work, ordinal) for the runs of this CTA: dealt out back and forth.  Runs without tiles get ordinal -1.
template <int kMode, typename F>
__device__ __forceinline__ void for_each_run(const StreamArgs& a, F f) {
  const int grid = gridDim.x;
  int k = 0;
  for (int round = 0; round * grid < a.n_runs; ++round) {
    const int run = round * grid + (round & 1 ? grid - 1 - (int)blockIdx.x : (int)blockIdx.x);
    if (run >= a.n_runs) continue;
    const Work w = decode<kMode>(a, run);
    if (!f(w, w.cnt > 0 ? k : -1)) return;
    if (w.cnt > 0) ++k;
  }
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, int bytes, void* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// ---- roles --------------------------------------------------------------------------------------------
template <int kMode, bool kTest>
__device__ __forceinline__ void producer(const StreamArgs& a, int* status, const CUtensorMap* fix, const CUtensorMap* str, Shared* sh, char* tiles) {
  const int n_sub = a.D / 64;
  const int fix_bytes = n_sub * 128 * (kMode == kEntropy && a.r <= 128 ? a.hb * a.r : 128), str_bytes = n_sub * kSubTileBytes;
  int tc = 0;
  bool ok = true;
  for_each_run<kMode>(a, [&](const Work& w, int k) {
    if (k < 0) return true;
    const int fb = k & 1;
    if (!(ok = mbar_wait(&sh->fix_empty[fb], ((k >> 1) & 1) ^ 1, status, wait_limit<kTest>(a)))) return false;
    mbar_expect_tx(&sh->fix_full[fb], fix_bytes);
    for (int s = 0; s < n_sub; ++s)
      tma_load_4d(tiles + kOffFix + fb * kTileBytes + s * kSubTileBytes, fix, &sh->fix_full[fb], s * 64, w.fix_row, w.fix_head, w.b);
    for (int t = 0; t < w.cnt; ++t, ++tc) {
      int row, head;
      if (kMode == kColumns) {
        const int g = (w.first + t) / w.per_head;
        row = w.fix_row + (w.first + t - g * w.per_head) * 128;
        head = w.fix_head * a.G + a.g0 + g;
      } else {
        row = (w.first + t) * 128;
        head = w.fix_head / a.G;
      }
      const int stage = tc % kStages;
      if (!(ok = mbar_wait(&sh->str_empty[stage], ((tc / kStages) & 1) ^ 1, status, wait_limit<kTest>(a)))) return false;
      mbar_expect_tx(&sh->str_full[stage], str_bytes);
      for (int s = 0; s < n_sub; ++s)
        tma_load_4d(tiles + kOffStr + stage * kTileBytes + s * kSubTileBytes, str, &sh->str_full[stage], s * 64, row, head, w.b);
    }
    return true;
  });
  if (!ok) {
    // a wait ran out: give copies already in flight a bounded time (1 ms) to land before the CTA exits
    const long long now = now_ns();
    while (now_ns() - now < 1000000) __nanosleep(1000);
  }
}

// Group g's number of tiles so far, mod 4 (two bits of `turns`), then one more.
__device__ __forceinline__ int take_turn(uint32_t& turns, int g) {
  const int at = 2 * g, now = (turns >> at) & 3;
  turns = (turns & ~(3u << at)) | (((now + 1) & 3u) << at);
  return now;
}

// Columns: the constants of every streamed tile's rows, into the place of the accumulator the tile will use.
template <bool kTest>
__device__ __forceinline__ void table_loader(const StreamArgs& a, int* status, Shared* sh) {
  int tc = 0;
  uint32_t turns = 0;                       // two bits per group: its tiles so far, mod 4
  bool ok = true;
  for_each_run<kColumns>(a, [&](const Work& w, int k) {
    if (k < 0) return true;
    for (int t = 0; t < w.cnt; ++t, ++tc) {
      const int acc = tc & 3, g = (w.first + t) / w.per_head, row = w.fix_row + (w.first + t - g * w.per_head) * 128;
      if (!(ok = mbar_wait(&sh->acc_empty[acc], ((tc >> 2) & 1) ^ 1, status, wait_limit<kTest>(a)))) return false;
      void* full = &sh->tab_full[t % kGroups][take_turn(turns, t % kGroups)];
      mbar_expect_tx(full, 2 * 512);
      bulk_load(sh->tab_c[acc], a.ctab + row, 512, full);
      bulk_load(sh->tab_l[acc], a.neg_l + (size_t)(w.unit * a.gs + g) * a.n_pad + row, 512, full);
    }
    return true;
  });
  if (!ok) {
    const long long now = now_ns();
    while (now_ns() - now < 1000000) __nanosleep(1000);
  }
}

// D[fixed rows x streamed rows].  The whole warp walks the runs, converged, and one elected lane issues; a tile's barriers
// are tested while the tile before it is being issued.
template <int kMode, bool kTest>
__device__ __forceinline__ void mma_warp(const StreamArgs& a, int* status, Shared* sh, char* tiles, uint32_t tmem_base) {
  const int nk = a.D / 16;
  const uint32_t idesc = umma_idesc(128, 128, a.bf16);
  int tc = 0;
  uint32_t turns = 0;
  for_each_run<kMode>(a, [&](const Work& w, int k) {
    if (k < 0) return true;
    const int fb = k & 1, cnt = __shfl_sync(0xffffffffu, w.cnt, 0);
    if (!__all_sync(0xffffffffu, mbar_wait(&sh->fix_full[fb], (k >> 1) & 1, status, wait_limit<kTest>(a)))) return false;
    const uint32_t a_lo = umma_desc_lo(smem_u32(tiles + kOffFix + fb * kTileBytes));
    bool s_ok = false, a_ok = false;
    for (int t = 0; t < cnt; ++t, ++tc) {
      const int stage = tc % kStages, acc = tc & 3;
      if (!s_ok && !__all_sync(0xffffffffu, mbar_wait(&sh->str_full[stage], (tc / kStages) & 1, status, wait_limit<kTest>(a)))) return false;
      if (!a_ok && !__all_sync(0xffffffffu, mbar_wait(&sh->acc_empty[acc], ((tc >> 2) & 1) ^ 1, status, wait_limit<kTest>(a)))) return false;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 128);
      const uint32_t b_lo = umma_desc_lo(smem_u32(tiles + kOffStr + stage * kTileBytes));
      if (t + 1 < cnt) {
        s_ok = __all_sync(0xffffffffu, mbar_test(&sh->str_full[(tc + 1) % kStages], ((tc + 1) / kStages) & 1));
        a_ok = __all_sync(0xffffffffu, mbar_test(&sh->acc_empty[(tc + 1) & 3], (((tc + 1) >> 2) & 1) ^ 1));
      }
      void* full = &sh->acc_full[t % kGroups][take_turn(turns, t % kGroups)];
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = (uint32_t)(((kk >> 2) * kSubTileBytes + (kk & 3) * 32) >> 4);
          if (kk < nk) {
            if (kk == 0) umma_step<0>(d_tmem, desc64(a_lo + off, kDescHi), desc64(b_lo + off, kDescHi), idesc);
            else umma_step<1>(d_tmem, desc64(a_lo + off, kDescHi), desc64(b_lo + off, kDescHi), idesc);
          }
        }
        tc_commit(full);
        tc_commit(&sh->str_empty[stage]);
        if (t + 1 == cnt) tc_commit(&sh->fix_empty[fb]);   // the fixed tile is free once the run's products are done
      }
      __syncwarp();
    }
    return true;
  });
}

// Like fold_chunk, with the sum T of 2^{x - M} (x - M) beside Z.  Masked exponents are finite and huge instead of -inf, so
// that their terms of T are 0, not NaN; the mask goes over the finished exponent, whatever the scale makes of a logit.
constexpr float kMaskedExp = -1e30f;
template <bool kMask>
__device__ __forceinline__ void exp_sums32(const float* v, float c, float neg, int j_first, int last, float& z, float& t) {
  const uint64_t c2 = pack2(c, c), neg2 = pack2(neg, neg);
  uint64_t za = pack2(0.f, 0.f), zb = za, ta = za, tb = za;
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    uint64_t xa = fma2(pack2(v[i], v[i + 1]), c2, neg2), xb = fma2(pack2(v[i + 2], v[i + 3]), c2, neg2);
    float x0, x1, x2, x3;
    unpack2(xa, x0, x1);
    unpack2(xb, x2, x3);
    if (kMask) {
      if (j_first + i > last) x0 = kMaskedExp;
      if (j_first + i + 1 > last) x1 = kMaskedExp;
      if (j_first + i + 2 > last) x2 = kMaskedExp;
      if (j_first + i + 3 > last) x3 = kMaskedExp;
      xa = pack2(x0, x1);
      xb = pack2(x2, x3);
    }
    const uint64_t ea = pack2(fast_exp2(x0), fast_exp2(x1)), eb = pack2(fast_exp2(x2), fast_exp2(x3));
    za = add2(za, ea);
    zb = add2(zb, eb);
    ta = fma2(ea, xa, ta);
    tb = fma2(eb, xb, tb);
  }
  float z0, z1, t0, t1;
  unpack2(add2(za, zb), z0, z1);
  unpack2(add2(ta, tb), t0, t1);
  z = z0 + z1;
  t = t0 + t1;
}
// Z and T of a row against its largest logit so far, v_max c.  The shift is the maximum itself and not, as where only Z is
// wanted, a value near it: the leading term is then 1 exactly, and log2 Z of a row with one key that matters is as small as it
// should be.  (Found before the exponentials, for 16 three-way maxima a chunk: with a second look only at chunks whose sum
// says that something exceeded the shift, some row of a warp nearly always does, 135 us a call
// of 64 heads x 128 rows x 32768 keys against 175.)  Where the shift is so large
// that rounding it could move an exponential by more than 2^{1/16}, the logits are taken relative to v_max before they are scaled.
constexpr float kWideShift = 1048576.f;   // 2^20
template <bool kMask>
__device__ __forceinline__ void fold_chunk_mean(const uint32_t* r, int j_first, int last, float c, float& v_max, float& Z, float& T) {
  float v[32], top[4] = {v_max, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    v[i] = __uint_as_float(r[i]);
    if (!kMask || j_first + i <= last) top[i & 3] = fmaxf(top[i & 3], v[i]);
  }
  const float mx = fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3]));
  float neg = -mx * c;
  const bool wide = fabsf(neg) > kWideShift;
  if (mx > v_max) {
    if (Z > 0.f) {
      const float d = wide ? (v_max - mx) * c : v_max * c + neg, s = fast_exp2(d);
      T = (T + Z * d) * s;
      Z *= s;
    }
    v_max = mx;
  }
  if (mx > -INFINITY) {
    if (wide) {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] -= mx;
      neg = 0.f;
    }
    float z, t;
    exp_sums32<kMask>(v, c, neg, j_first, last, z, t);
    Z += z;
    T += t;
  }
}

// Thirty-two rows of a key's column: adds 2^{c D - L} of each.  kDiagonal: only rows from the key's own on see it.
template <bool kDiagonal>
__device__ __forceinline__ void column_chunk(const uint32_t* r, const float* c, const float* neg_l, int row0, int key, uint64_t& za,
                                             uint64_t& zb) {
#pragma unroll
  for (int t = 0; t < 32; t += 4) {
    const float4 cc = *reinterpret_cast<const float4*>(c + t), ll = *reinterpret_cast<const float4*>(neg_l + t);
    float x0, x1, x2, x3;
    unpack2(fma2(pack2(__uint_as_float(r[t]), __uint_as_float(r[t + 1])), pack2(cc.x, cc.y), pack2(ll.x, ll.y)), x0, x1);
    unpack2(fma2(pack2(__uint_as_float(r[t + 2]), __uint_as_float(r[t + 3])), pack2(cc.z, cc.w), pack2(ll.z, ll.w)), x2, x3);
    if (kDiagonal) {
      if (row0 + t < key) x0 = -INFINITY;
      if (row0 + t + 1 < key) x1 = -INFINITY;
      if (row0 + t + 2 < key) x2 = -INFINITY;
      if (row0 + t + 3 < key) x3 = -INFINITY;
    }
    za = add2(za, pack2(fast_exp2(x0), fast_exp2(x1)));
    zb = add2(zb, pack2(fast_exp2(x2), fast_exp2(x3)));
  }
}

// Softmax warps: groups of four warps, a thread per TMEM lane; tile t of a run belongs to group t mod kGroups.
template <int kMode, bool kTest>
__device__ __forceinline__ void softmax_group(const StreamArgs& a, int* status, Shared* sh, uint32_t tmem_base, int g) {
  const int s = threadIdx.x & 127, quarter = (threadIdx.x >> 5) & 3;
  const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
  int tc0 = 0, mine = 0;   // tiles, own tiles so far
  for_each_run<kMode>(a, [&](const Work& w, int k) {
    if (k < 0) return true;
    float res = 0.f, Z = 0.f, T = 0.f;
    if (kMode == kColumns) {
      for (int t = g; t < w.cnt; t += kGroups, ++mine) {
        const int acc = (tc0 + t) & 3;
        if (!mbar_wait(&sh->tab_full[g][mine & 3], (mine >> 2) & 1, status, wait_limit<kTest>(a))) return false;
        if (!mbar_wait(&sh->acc_full[g][mine & 3], (mine >> 2) & 1, status, wait_limit<kTest>(a))) return false;
        tc_fence_after();
        const bool diagonal = (w.first + t) % w.per_head == 0;
        uint64_t za = pack2(0.f, 0.f), zb = za;
#pragma unroll 1
        for (int ch = 0; ch < 4; ++ch) {
          uint32_t ra[32];
          tmem_ld32_issue(lane_base + acc * 128 + 32 * ch, ra);
          tmem_ld_wait(ra);
          if (!diagonal) column_chunk<false>(ra, sh->tab_c[acc] + 32 * ch, sh->tab_l[acc] + 32 * ch, 32 * ch, s, za, zb);
          else column_chunk<true>(ra, sh->tab_c[acc] + 32 * ch, sh->tab_l[acc] + 32 * ch, 32 * ch, s, za, zb);
        }
        tc_fence_before();
        mbar_arrive(&sh->acc_empty[acc]);            // the accumulator and its rows' constants are free
        float z0, z1;
        unpack2(add2(za, zb), z0, z1);
        res += z0 + z1;
      }
    } else {
      float c;
      int last, min_last;
      if (kMode == kEntropy) {
        const int i = a.r <= 128 ? s % a.r : w.fix_row + s;
        c = a.c[i < a.r ? i : 0];
        last = s < w.rows ? a.last[i < a.r ? i : 0] : -1;
        min_last = a.min_last;
      } else {
        c = a.ctab[w.fix_row + s];
        last = w.fix_row + s < a.n ? w.fix_row + s : -1;
        min_last = w.fix_row;
      }
      const bool live = kMode == kRowStats || quarter * 32 < w.rows;
      float M = -INFINITY;                           // entropy: M in units of the raw logit until the run is over
      for (int t = g; t < w.cnt; t += kGroups, ++mine) {
        const int acc = (tc0 + t) & 3;
        if (!mbar_wait(&sh->acc_full[g][mine & 3], (mine >> 2) & 1, status, wait_limit<kTest>(a))) return false;
        tc_fence_after();
        const int j0 = (w.first + t) * 128;
        const bool full = j0 + 127 <= min_last && j0 + 128 <= a.n;
        if (live) {
#pragma unroll 1
          for (int ch = 0; ch < 4; ++ch) {
            uint32_t ra[32];
            tmem_ld32_issue(lane_base + acc * 128 + 32 * ch, ra);
            tmem_ld_wait(ra);
            if (ch == 3) {
              tc_fence_before();
              mbar_arrive(&sh->acc_empty[acc]);
            }
            if (kMode != kEntropy) fold_chunk(ra, full, j0 + 32 * ch, last, c, M, Z);
            else if (full) fold_chunk_mean<false>(ra, j0 + 32 * ch, last, c, M, Z, T);
            else fold_chunk_mean<true>(ra, j0 + 32 * ch, last, c, M, Z, T);
          }
        } else {
          mbar_arrive(&sh->acc_empty[acc]);
        }
      }
      if (kMode == kEntropy) res = last < 0 ? -INFINITY : M * c;
      else res = last < 0 ? -INFINITY : Z > 0.f ? M + log2f(Z) : Z == Z ? -INFINITY : Z;   // rows that do not exist weigh nothing
    }
    tc0 += w.cnt;
    const int slot = k & 1;
    if (!mbar_wait(&sh->stat_empty[slot], ((k >> 1) & 1) ^ 1, status, wait_limit<kTest>(a))) return false;
    sh->stat[slot][g][s] = res;
    if (kMode == kEntropy) {
      sh->z[slot][g][s] = Z;
      sh->t[slot][g][s] = T;
    }
    if (!(kTest && a.test_withhold && blockIdx.x == 0 && k == 0)) mbar_arrive(&sh->stat_full[slot]);
    return true;
  });
}

// (M, Z, T) of disjoint key sets into one, in order.  Nothing (Z = 0) weighs nothing; a NaN stays.
template <int N>
__device__ __forceinline__ void merge_parts(const float (&m)[N], const float (&z)[N], const float (&t)[N], float& M, float& Z, float& T) {
  float top = M;
#pragma unroll
  for (int i = 0; i < N; ++i) top = fmaxf(top, m[i]);
  if (top > -INFINITY) {
    if (Z != 0.f) {
      const float d = M - top, s = fast_exp2(d);
      T = (T + Z * d) * s;
      Z *= s;
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (z[i] != 0.f) {
        const float d = m[i] - top, s = fast_exp2(d);
        T += (t[i] + z[i] * d) * s;
        Z += z[i] * s;
      }
    M = top;
  }
}

// Delivery warp: the groups' shares of a run, in order, into the run's result; lane l has rows (keys) 4 l .. 4 l + 3.
template <int kMode, bool kTest>
__device__ __forceinline__ void delivery(const StreamArgs& a, int* status, Shared* sh) {
  const int lane = threadIdx.x & 31;
  for_each_run<kMode>(a, [&](const Work& w, int k) {
    float v[4], Z[4] = {}, T[4] = {};
    if (k >= 0) {
      const int slot = k & 1;
      if (!mbar_wait(&sh->stat_full[slot], (k >> 1) & 1, status, wait_limit<kTest>(a))) return false;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float x[kGroups], z[kGroups], t[kGroups];
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
          x[g] = sh->stat[slot][g][4 * lane + e];
          if (kMode == kEntropy) {
            z[g] = sh->z[slot][g][4 * lane + e];
            t[g] = sh->t[slot][g][4 * lane + e];
          }
        }
        if (kMode == kColumns) {
          v[e] = x[0];
#pragma unroll
          for (int g = 1; g < kGroups; ++g) v[e] += x[g];
        } else if (kMode == kRowStats) {
          float M = -INFINITY, sum = 0.f;
          merge_logs(x, M, sum);
          v[e] = M + log2f(sum);
        } else {
          v[e] = -INFINITY;
          merge_parts(x, z, t, v[e], Z[e], T[e]);
        }
      }
      mbar_arrive(&sh->stat_empty[slot]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = kMode == kColumns ? 0.f : -INFINITY;
    }
    if (kMode == kColumns) {
      float* to = a.s + ((size_t)w.unit * a.splits + w.rin) * a.n;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = w.fix_row + 4 * lane + e;
        if (j < a.n) to[j] = a.accumulate ? to[j] + v[e] * a.inv_g : v[e] * a.inv_g;
      }
    } else if (kMode == kRowStats) {
      // a single part is final: -L, and -inf for rows that do not exist
      if (a.rpu == 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = v[e] == -INFINITY ? v[e] : -v[e];
      }
      float* to = a.stat + ((size_t)w.rin * a.BH * a.gs + w.unit) * a.n_pad + w.fix_row + 4 * lane;
      *reinterpret_cast<float4*>(to) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      const size_t at = ((size_t)w.unit * a.rpu + w.rin) * 128 + 4 * lane;
      *reinterpret_cast<float4*>(a.stat + at) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4*>(a.z + at) = make_float4(Z[0], Z[1], Z[2], Z[3]);
      *reinterpret_cast<float4*>(a.t + at) = make_float4(T[0], T[1], T[2], T[3]);
    }
    return true;
  });
}

template <int kMode, bool kTest>
__global__ void __launch_bounds__(kThreads, 1)
stream_kernel(const __grid_constant__ CUtensorMap fix, const __grid_constant__ CUtensorMap str, const __grid_constant__ StreamArgs a) {
  extern __shared__ char smem_raw[];
  char* tiles = reinterpret_cast<char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  Shared* sh = reinterpret_cast<Shared*>(tiles + kSmemTiles);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&fix)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&str)) : "memory");
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sh->fix_full[s], 1);
      mbar_init(&sh->fix_empty[s], 1);
      mbar_init(&sh->stat_full[s], 128 * kGroups);
      mbar_init(&sh->stat_empty[s], 32);
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sh->str_full[s], 1);
      mbar_init(&sh->str_empty[s], 1);
    }
    for (int s = 0; s < 4; ++s) {
      mbar_init(&sh->acc_empty[s], 128);
      for (int g = 0; g < kGroups; ++g) {
        mbar_init(&sh->acc_full[g][s], 1);
        mbar_init(&sh->tab_full[g][s], 1);
      }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (kMode == kEntropy && (a.r <= 128 ? a.hb * a.r : 128) < 128) {   // rows the box never covers must read as zeros
    uint4* z = reinterpret_cast<uint4*>(tiles + kOffFix);
    for (int t = threadIdx.x; t < 2 * kTileBytes / 16; t += kThreads) z[t] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {   // all 512 TMEM columns: four 128-column accumulators
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sh->tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_slot;
  griddep_wait();

  int* const status = kMode == kEntropy ? a.status + 1 + blockIdx.x : a.status;
  if (kMode == kEntropy) {
    if (threadIdx.x == 0) *status = 0;
    __syncthreads();
  }

  if (warp == 0) {
    if (lane == 0) producer<kMode, kTest>(a, status, &fix, &str, sh, tiles);
  } else if (warp == 1) {
    mma_warp<kMode, kTest>(a, status, sh, tiles, __shfl_sync(0xffffffffu, tmem_base, 0));
  } else if (warp == 2) {
    delivery<kMode, kTest>(a, status, sh);
  } else if (warp == 3) {
    if (kMode == kColumns && lane == 0) table_loader<kTest>(a, status, sh);
  } else {
    softmax_group<kMode, kTest>(a, status, sh, tmem_base, (warp - 4) >> 2);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
}

// The parts of a row block's statistics into the rows' entropies, and the CTAs' status words into the call's.
__global__ void __launch_bounds__(128) entropy_finish(const __grid_constant__ StreamArgs a, float* __restrict__ out, int Hq) {
  griddep_wait();
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    bool expired = false;
    for (int i = threadIdx.x; i < min(a.n_runs, kSms); i += 32) expired |= a.status[1 + i] == (int)AHAKV_ERR_TIMEOUT;
    expired = __any_sync(0xffffffffu, expired);
    if (threadIdx.x == 0) a.status[0] = expired ? (int)AHAKV_ERR_TIMEOUT : 0;
  }
  const Work w = decode<kEntropy>(a, blockIdx.x * a.rpu);
  const int s = threadIdx.x;
  if (s >= w.rows) return;
  float M = -INFINITY, Z = 0.f, T = 0.f;
  const size_t at = (size_t)w.unit * a.rpu * 128 + s;
  for (int t0 = 0; t0 < a.rpu; t0 += 8) {
    float m[8], z[8], t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const size_t from = at + (size_t)(t0 + i) * 128;
      const bool there = t0 + i < a.rpu;
      m[i] = there ? a.stat[from] : -INFINITY;
      z[i] = there ? a.z[from] : 0.f;
      t[i] = there ? a.t[from] : 0.f;
    }
    merge_parts(m, z, t, M, Z, T);
  }
  const int head = a.r <= 128 ? w.fix_head + s / a.r : w.fix_head, i = a.r <= 128 ? s % a.r : w.fix_row + s;
  out[((size_t)w.b * Hq + head) * a.r + i] = 0.6931471805599453f * (log2f(Z) - T / Z);
}

// The parts of the causal rows' statistics into -L (-inf for rows that do not exist).
__global__ void __launch_bounds__(256) row_stats_finish(const float* stat, float* neg_l, int parts, size_t total) {
  griddep_wait();
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= total) return;
  float M = -INFINITY, Z = 0.f;
  for (int p = 0; p < parts; ++p) {
    const float x[1] = {stat[p * total + i]};
    merge_logs(x, M, Z);
  }
  const float L = M + log2f(Z);
  neg_l[i] = L == -INFINITY ? L : -L;
}

// Eq. 12 (or the call's scale) for every row of the cache, times log2(e); zero past the end.  Clears the status word.
__global__ void __launch_bounds__(256) row_scales(float* ctab, int n, int n_pad, int mode, double fixed, double first_tokens, double budget,
                                                  int d, int* status) {
  griddep_wait();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i == 0) *status = 0;
  if (i >= n_pad) return;
  double lam = fixed;
  if (mode == AHAKV_SCALE_ADAPTIVE_ROW) {
    const double ratio = (first_tokens + i) / budget;
    lam = ratio > 1.0 ? sqrt(2.0 * log(ratio) / (double)d) : 1.0 / sqrt((double)d);
  }
  ctab[i] = i < n ? (float)(lam * 1.4426950408889634) : 0.f;
}

// ---- host ------------------------------------------------------------------------------------------------
template <int kMode>
cudaError_t launch_stream(const CUtensorMap& fix, const CUtensorMap& str, StreamArgs& a, cudaStream_t st) {
  const TestHooks hooks = test_hooks();
  const bool test = hooks.wait_ns > 0 || hooks.withhold != 0;
  a.test_wait_ns = hooks.wait_ns > 0 ? hooks.wait_ns : kWaitLimitNs;
  a.test_withhold = hooks.withhold;
  // leave to use more than 48 KB of shared memory, asked for once per device
  constexpr int kMaxDevices = 64;
  static bool configured[kMaxDevices] = {};
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(stream_kernel<kMode, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(stream_kernel<kMode, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  count_launch();
  return launch_chained(test ? stream_kernel<kMode, true> : stream_kernel<kMode, false>, dim3(a.n_runs < kSms ? a.n_runs : kSms), dim3(kThreads), 1, kSmemBytes, st, fix, str, a);
}

// Parts per row block of the entropy's walk: the number that makes rounds x (tiles of a part + 1) smallest, a run boundary
// costing about a tile; at most 64, and at most sixteen rounds of runs.
constexpr int kMaxParts = 64, kMaxPartRuns = 16 * kSms;
int entropy_parts(const Plan& pl) {
  const long long units = (long long)pl.B * pl.Hkv * pl.n_rb;
  int best = 1;
  long long best_cost = -1;
  for (int p = 1; p <= pl.n_blk && p <= kMaxParts && (p == 1 || units * p <= kMaxPartRuns); ++p) {
    const long long cost = (units * p + kSms - 1) / kSms * ((pl.n_blk + p - 1) / p + 1);
    if (best_cost < 0 || cost < best_cost) { best = p; best_cost = cost; }
  }
  return best;
}

}  // namespace

// Room for as many parts as any call with these row blocks and tiles, or fewer, may be cut into: a larger batch or a longer
// context may want fewer parts, but scratch that was sized for it has to serve the smaller calls too.  One part more than
// there can be covers what a call with fewer than 128 keys keeps (entropy.cu: 16 bytes a row).
size_t entropy_tc_scratch_bytes(const Plan& pl) {
  const size_t units = (size_t)pl.B * pl.Hkv * pl.n_rb, most = units * (pl.n_blk < kMaxParts ? pl.n_blk : kMaxParts);
  const size_t runs = most < kMaxPartRuns ? most : units > kMaxPartRuns ? units : kMaxPartRuns;
  return kStatusBytes + (runs + units) * 128 * 3 * sizeof(float);
}

ahakv_status launch_entropy_tc(const Plan& pl, const void* q, const void* k, void* scratch, float* out, cudaStream_t st) {
  StreamArgs a = {};
  a.n = pl.n; a.D = pl.d; a.bf16 = pl.dtype == AHAKV_BF16; a.G = pl.G; a.Hkv = pl.Hkv; a.n_blk = pl.n_blk;
  a.r = pl.r; a.hb = pl.heads_per_rb; a.n_rb = pl.n_rb;
  a.rpu = entropy_parts(pl);
  const int units = pl.B * pl.Hkv * pl.n_rb;
  a.n_runs = units * a.rpu;
  a.min_last = pl.last[0];
  a.status = (int*)scratch;
  a.stat = (float*)((char*)scratch + kStatusBytes);
  a.z = a.stat + (size_t)units * a.rpu * 128;
  a.t = a.z + (size_t)units * a.rpu * 128;
  for (int i = 0; i < kMaxRows; ++i) { a.c[i] = pl.rows.c[i]; a.last[i] = pl.last[i]; }
  CUtensorMap qmap, kmap;
  const int box_rows = pl.r <= 128 ? pl.r : 128, box_heads = pl.r <= 128 ? pl.heads_per_rb : 1;
  if (!make_map(&qmap, q, a.bf16, pl.d, pl.r, pl.Hq, pl.B, pl.qs, pl.es, box_rows, box_heads) ||
      !make_map(&kmap, k, a.bf16, pl.d, pl.n, pl.Hkv, pl.B, pl.ks, pl.es, kKeyTile, 1))
    return AHAKV_ERR_CUDA;
  cudaError_t e = launch_stream<kEntropy>(qmap, kmap, a, st);
  if (e == cudaSuccess) e = launch_chained(entropy_finish, dim3(units), dim3(128), 1, 0, st, a, out, pl.Hq);
  count_launch();
  return cuda_ok(e);
}

// The room: row scales, -L per row of the query heads of a pass, the parts of their statistics, and the column sums of
// every split.  `pool` is what the workspace has for them.  As many query heads of each group a pass as fit.
ahakv_status launch_causal_tc(const Plan& pl, int scale_mode, double fixed, long long first_cached, const void* q, const long long qs[3],
                              const void* k, float* pool, size_t pool_bytes, float* sums, const float** slots_out, int* n_slots,
                              int* status, cudaStream_t st) {
  const int BH = pl.B * pl.Hkv;
  StreamArgs a = {};
  a.n = pl.n; a.D = pl.d; a.bf16 = pl.dtype == AHAKV_BF16; a.G = pl.G; a.Hkv = pl.Hkv; a.n_blk = pl.n_blk;
  a.BH = BH; a.n_pad = pl.n_blk * kKeyTile; a.status = status;
  a.inv_g = 1.f / (float)pl.G;
  float* ctab = pool;
  size_t room = pool_bytes / sizeof(float) - a.n_pad, head = (size_t)BH * a.n_pad;   // floats left; floats of one head of each group
  // Splits of a key tile's rows: enough runs for three a CTA, as far as the room goes (one needs none: it is `sums`).
  int splits = 1;
  while (splits < 8 && (long long)pl.n_blk * BH * splits < 3LL * kSms && room >= head + (size_t)BH * pl.n * splits * 2) splits *= 2;
  float* slots = sums;
  if (splits > 1) {
    slots = ctab + a.n_pad;
    const size_t used = ((size_t)BH * pl.n * splits + 63) / 64 * 64;
    room -= used;
    pool = slots + used;
  } else {
    pool = ctab + a.n_pad;
  }
  int gs = (int)(room / head);
  if (gs < 1) return AHAKV_ERR_WORKSPACE;
  if (gs > pl.G) gs = pl.G;
  // Parts of a row block's keys, likewise: their statistics need room beside the finished ones.
  int parts = 1;
  while (parts < 8 && (long long)pl.n_blk * BH * gs * parts < 3LL * kSms && room >= head * gs * (1 + 2 * parts)) parts *= 2;
  CUtensorMap qmap, kmap;
  if (!make_map(&qmap, q, a.bf16, pl.d, pl.n, pl.Hq, pl.B, qs, pl.es, kKeyTile, 1) ||
      !make_map(&kmap, k, a.bf16, pl.d, pl.n, pl.Hkv, pl.B, pl.ks, pl.es, kKeyTile, 1))
    return AHAKV_ERR_CUDA;
  a.ctab = ctab;
  cudaError_t e = launch_chained(row_scales, dim3((a.n_pad + 255) / 256), dim3(256), 1, 0, st, ctab, pl.n, a.n_pad, scale_mode, fixed,
                                 (double)(first_cached + 1), (double)pl.Bud, pl.d, status);
  count_launch();
  for (int g0 = 0; g0 < pl.G && e == cudaSuccess; g0 += gs) {
    a.g0 = g0;
    a.gs = pl.G - g0 < gs ? pl.G - g0 : gs;
    const size_t rows = head * a.gs;
    float* neg_l = pool;
    a.rpu = parts;
    a.stat = parts > 1 ? pool + rows : pool;
    a.n_runs = pl.n_blk * BH * a.gs * parts;
    e = launch_stream<kRowStats>(qmap, kmap, a, st);
    if (e == cudaSuccess && parts > 1) {
      e = launch_chained(row_stats_finish, dim3((unsigned)((rows + 255) / 256)), dim3(256), 1, 0, st, a.stat, neg_l, parts, rows);
      count_launch();
    }
    a.neg_l = neg_l;
    a.s = slots;
    a.splits = splits;
    a.accumulate = g0 > 0;
    a.n_runs = pl.n_blk * BH * splits;
    if (e == cudaSuccess) e = launch_stream<kColumns>(kmap, qmap, a, st);
  }
  *slots_out = slots;
  *n_slots = splits;
  return cuda_ok(e);
}

}  // namespace ahakv

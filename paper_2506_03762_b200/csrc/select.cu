// Value-prior refinement (Eq. 13-15) and budgeted selection (Algorithm 1).
//
// One cluster of C CTAs per (sequence, KV head), each CTA a contiguous piece of its tokens, each thread kPer adjacent ones,
// whose refined scores stay in registers from the first load to the last store.
//   refine: adds the row-block partial scores, smooths nu with the mean filter, normalises by the head-wide maximum,
//     multiplies, and adds the carried score.
//   select: the B_s-th largest candidate score by a histogram over the order-preserving integer image of the float: its
//     2048 bins cover the sixteen octaves below the largest raw score (128 an octave, so that few tokens meet in a bin),
//     it names the bin the threshold falls into, and the tokens of that bin are ranked against each other from a list;
//     as long as they are too many for the list, a histogram over the bin's own range comes first (at most three more).
//     Then every candidate above the threshold plus the lowest-indexed ones equal to it are emitted in ascending index
//     order (a prefix sum over the cluster), then the recent window; exact, ties lowest index first.
// What bounds it: for few heads the latency of its steps (about ten block-wide ones; the cluster adds four barriers), for
// many the instructions.  Adjacent tokens per thread make both cheaper than tokens dealt out in turn: a thread reads its
// filter window once, straight from L1 (a warp's loads together cover whole lines), and the ordered emission needs one
// prefix sum over threads instead of a ballot per token.
#include <cooperative_groups.h>

#include "ahakv_internal.cuh"
#include "select_common.cuh"

namespace ahakv {
namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 4 * kThreads;
constexpr int kList = kThreads;          // one list entry per thread
constexpr int kMaxPer = 16, kMaxCluster = 16;

struct SelectArgs {
  const float* s_raw;       // [unit][slots][n]
  const float* nu;          // [unit][n], or null: no value prior
  const float* prev;        // [unit][n], or null
  float* score;             // [unit][n] refined score out, or null
  float* score_out;         // [unit][n_keep] scores of the kept tokens, or null
  int32_t* kept;            // [unit][n_keep], or null: refinement only
  const int32_t* budgets;   // a budget per unit, or null
  // the gather of the kept rows, when this kernel does it too (one CTA per head): k_out null otherwise
  const char *k, *v;
  char *k_out, *v_out;
  int lanes;                // 16-byte pieces of a row
  int slots;
  int chunk;                // tokens per CTA, a multiple of kMaxPer
};

// The budget of one (sequence, KV head): the call's, or the caller's own for this head, held to [max(Br, 1), Bud].
__device__ __forceinline__ int head_budget(const Shape& pl, const int32_t* budgets, int unit) {
  if (budgets == nullptr) return pl.Bud;
  return min(max(budgets[unit], max(pl.Br, 1)), pl.Bud);
}

// Exclusive prefix sum of x over the block, and the block's total.  `tot` holds kWarps counts and is free again after the
// next block-wide barrier.
__device__ __forceinline__ unsigned block_scan(unsigned x, unsigned* tot, unsigned& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) tot[warp] = inc;
  __syncthreads();
  const unsigned y = lane < kWarps ? tot[lane] : 0u;
  total = __reduce_add_sync(0xffffffffu, y);
  return __reduce_add_sync(0xffffffffu, lane < warp ? y : 0u) + inc - x;
}

// kPer adjacent values from p + j0 (p: a head's row), zero from n on; `vec`: rows start on 16-byte boundaries.
template <int kPer>
__device__ __forceinline__ void load_run(const float* p, int j0, int n, bool vec, float (&v)[kPer]) {
  if (kPer >= 4 && vec && j0 + kPer <= n) {
#pragma unroll
    for (int e = 0; e < kPer; e += 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + j0 + e);
      v[e] = x.x; v[(e + 1) % kPer] = x.y; v[(e + 2) % kPer] = x.z; v[(e + 3) % kPer] = x.w;
    }
  } else {
#pragma unroll
    for (int e = 0; e < kPer; ++e) v[e] = j0 + e < n ? p[j0 + e] : 0.f;
  }
}

__device__ __noinline__ float pooled_any(const float* nu, int j, int n, int half, float inv_w, bool zero_pad) {
  return pooled(nu, j, n, half, inv_w, zero_pad);
}

// Rows out[0 .. count) of K and V to the dense outputs, by the one CTA that has just written the indices.
__device__ __forceinline__ void gather_rows(const SelectArgs& a, const Shape& pl, const int32_t* out, int unit, int count) {
  __syncthreads();                                     // the indices are there
  const long long b = unit / pl.Hkv, h = unit % pl.Hkv;
  const int sub = threadIdx.x % a.lanes, step = kThreads / a.lanes;
  const char* k = a.k + (b * pl.ks[0] + h * pl.ks[1]) * pl.es + sub * 16;
  const char* v = a.v + (b * pl.vs[0] + h * pl.vs[1]) * pl.es + sub * 16;
  const long long ktok = pl.ks[2] * pl.es, vtok = pl.vs[2] * pl.es, row = (long long)a.lanes * 16;
  char* ko = a.k_out + (size_t)unit * pl.n_keep * row + sub * 16;
  char* vo = a.v_out + (size_t)unit * pl.n_keep * row + sub * 16;
#pragma unroll 4
  for (int t = threadIdx.x / a.lanes; t < count; t += step) {
    const long long j = *(const volatile int32_t*)(out + t);
    const uint4 x = *reinterpret_cast<const uint4*>(k + j * ktok), y = *reinterpret_cast<const uint4*>(v + j * vtok);
    *reinterpret_cast<uint4*>(ko + t * row) = x;
    *reinterpret_cast<uint4*>(vo + t * row) = y;
  }
}

template <int kPer, bool kCluster>
__global__ void __launch_bounds__(kThreads, kPer > 8 ? 1 : 2)
refine_select_kernel(const __grid_constant__ SelectArgs a, const __grid_constant__ Shape pl) {
  __shared__ __align__(16) unsigned hist[kBins];
  __shared__ __align__(16) unsigned list_key[kList + 4];
  __shared__ unsigned scan_tot[2][kWarps], cta_count;
  __shared__ uint2 red[kWarps], cta_max;              // largest filtered norm, largest raw (plus carried) score
  __shared__ unsigned list_n, sh_bin, sh_need, sh_in_bin, sh_thr, sh_need_eq;
  cg::cluster_group cl = cg::this_cluster();
  const int C = kCluster ? (int)cl.num_blocks() : 1, rank = kCluster ? (int)cl.block_rank() : 0;
  const int unit = kCluster ? blockIdx.x / C : blockIdx.x, n = pl.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = rank * a.chunk, end = min(base + a.chunk, n);
  const int j0 = base + tid * kPer;                    // this thread's tokens: j0 .. j0 + kPer - 1, as far as below `end`
  const bool prior = a.nu != nullptr, vec = (n & 3) == 0;
  *reinterpret_cast<uint4*>(&hist[4 * tid]) = make_uint4(0, 0, 0, 0);
  if (tid == 0) list_n = 0;
  griddep_wait();

  // ---- this thread's tokens ----
  float s[kPer], g[kPer], p[kPer];
  float top = -INFINITY, m = 0.f;
#pragma unroll
  for (int e = 0; e < kPer; ++e) { s[e] = 0.f; g[e] = 0.f; p[e] = 0.f; }
  if (j0 < end) {
    const float* raw = a.s_raw + (size_t)unit * a.slots * n;
    load_run<kPer>(raw, j0, n, vec, s);
    if (a.prev) load_run<kPer>(a.prev + (size_t)unit * n, j0, n, vec, p);
    if (prior) {
      const float* nu = a.nu + (size_t)unit * n;
      const int half = pl.pool / 2;
      const float inv_w = 1.f / (float)pl.pool;
      const bool zero_pad = (pl.flags & AHAKV_FLAG_POOL_ZERO_PAD) != 0;
      if (half == 3) {
        // the usual width: the window's values read once, added in the order of pooled() (the zeros outside the head
        // change nothing)
        float w[kPer + 6], own[kPer];
        load_run<kPer>(nu, j0, n, vec, own);
        if (vec && kPer >= 4) {
          const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 l = j0 >= 4 ? *reinterpret_cast<const float4*>(nu + j0 - 4) : z;
          const float4 r = j0 + kPer + 4 <= n ? *reinterpret_cast<const float4*>(nu + j0 + kPer) : z;
          w[0] = l.y; w[1] = l.z; w[2] = l.w;
          w[kPer + 3] = r.x; w[kPer + 4] = r.y; w[kPer + 5] = r.z;
        } else {
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            w[e] = j0 - 3 + e >= 0 ? nu[j0 - 3 + e] : 0.f;
            w[kPer + 3 + e] = j0 + kPer + e < n ? nu[j0 + kPer + e] : 0.f;
          }
        }
#pragma unroll
        for (int e = 0; e < kPer; ++e) w[3 + e] = own[e];
#pragma unroll
        for (int e = 0; e < kPer; ++e)
          g[e] = (((((w[e] + w[e + 1]) + w[e + 2]) + w[e + 3]) + w[e + 4]) + w[e + 5]) + w[e + 6];
        if ((j0 >= 3 && j0 + kPer + 3 <= n) || (zero_pad && j0 + kPer <= n)) {
#pragma unroll
          for (int e = 0; e < kPer; ++e) g[e] *= inv_w;
        } else {                                       // near an end: over the taps inside the head
#pragma unroll
          for (int e = 0; e < kPer; ++e) {
            const int taps = 7 - max(3 - j0 - e, 0) - max(j0 + e + 4 - n, 0);
            g[e] = j0 + e >= n ? 0.f : taps == 7 || zero_pad ? g[e] * inv_w : g[e] / (float)taps;
          }
        }
      } else {
#pragma unroll
        for (int e = 0; e < kPer; ++e)
          if (j0 + e < n) g[e] = pooled_any(nu, j0 + e, n, half, inv_w, zero_pad);
      }
#pragma unroll
      for (int e = 0; e < kPer; ++e) m = fmaxf(m, g[e]);
    }
#pragma unroll 1
    for (int t = 1; t < a.slots; ++t) {                // in the order of combine_slots()
      raw += n;
      float x[kPer];
      load_run<kPer>(raw, j0, n, vec, x);
#pragma unroll
      for (int e = 0; e < kPer; ++e) s[e] = pl.group_max ? fmaxf(s[e], x[e]) : s[e] + x[e];
    }
#pragma unroll
    for (int e = 0; e < kPer; ++e) top = fmaxf(top, s[e] + p[e]);
  }

  // ---- head-wide maxima, as integers: the norms are not negative, so that their bits are ordered like they are, and the
  // scores go by their order keys ----
  unsigned mbits = __reduce_max_sync(0xffffffffu, __float_as_uint(m)), ktop = __reduce_max_sync(0xffffffffu, order_key(top));
  if (lane == 0) red[warp] = make_uint2(mbits, ktop);
  __syncthreads();
  {
    const uint2 x = lane < kWarps ? red[lane] : make_uint2(0u, 0u);
    mbits = __reduce_max_sync(0xffffffffu, x.x);
    ktop = __reduce_max_sync(0xffffffffu, x.y);
  }
  if (kCluster) {
    if (tid == 0) cta_max = make_uint2(mbits, ktop);
    cl.sync();
    const uint2 x = *cl.map_shared_rank(&cta_max, lane < C ? lane : 0);
    mbits = __reduce_max_sync(0xffffffffu, x.x);
    ktop = __reduce_max_sync(0xffffffffu, x.y);
  }

  uint32_t key[kPer];
  const float inv_gmax = prior ? __frcp_rn(__uint_as_float(mbits)) : 1.f;
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    if (prior) s[e] = __fmul_rn(__fmul_rn(g[e], inv_gmax), s[e]);
    if (a.prev) s[e] = __fadd_rn(s[e], p[e]);
    key[e] = order_key(s[e]);
  }
  if (a.score && j0 < end) {
    float* to = a.score + (size_t)unit * n + j0;
    if (kPer >= 4 && vec && j0 + kPer <= n) {
#pragma unroll
      for (int e = 0; e < kPer; e += 4)
        *reinterpret_cast<float4*>(to + e) = make_float4(s[e], s[(e + 1) % kPer], s[(e + 2) % kPer], s[(e + 3) % kPer]);
    } else {
#pragma unroll
      for (int e = 0; e < kPer; ++e)
        if (j0 + e < n) to[e] = s[e];
    }
  }
  if (a.kept == nullptr) {
    griddep_launch();
    if (kCluster) cl.sync();
    return;
  }

  // ---- what is kept whatever the scores ----
  int32_t* out = a.kept + (size_t)unit * pl.n_keep;
  float* so = a.score_out ? a.score_out + (size_t)unit * pl.n_keep : nullptr;
  const int bud = head_budget(pl, a.budgets, unit);
  if (rank == 0)
    for (int t = min(n, bud) + tid; t < pl.n_keep; t += kThreads) out[t] = -1;   // a head with a budget of its own
  const bool all = n <= bud;                                                   // nothing to evict
  const int n_cand = all ? 0 : n - pl.Br, Bs = all ? 0 : bud - pl.Br;
  if (j0 < end && j0 + kPer > n_cand) {
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int j = j0 + e;
      if (j >= n_cand && j < n) {                      // all of them, or the recent window
        out[Bs + j - n_cand] = j;
        if (so) so[Bs + j - n_cand] = s[e];
      }
    }
  }
  if (Bs == 0) {
    griddep_launch();
    if (!kCluster && a.k_out) gather_rows(a, pl, out, unit, min(n, bud));
    if (kCluster) cl.sync();
    return;
  }

  // ---- threshold ----
  const int mine = j0 < end ? min(kPer, n_cand - j0) : 0;   // this thread's candidates: its first `mine` tokens
  // keys in [lo, hi] are still in question; bin b holds those with (key - lo) >> shift == b, the first histogram's lowest
  // bin everything below it too and its highest everything above
  const unsigned span = (unsigned)kBins << 16;
  unsigned lo = ktop > 0xfffdffffu ? 0xffffffffu - span + 1u : ktop + 0x20000u > span ? ktop + 0x20000u - span : 0u;
  unsigned hi = 0xffffffffu, need = (unsigned)Bs, thr = 0;
  int need_eq = 0, shift = 16;
  for (bool wide = true;; wide = false) {
    // `wide`: the first histogram, whose outer bins are open.  Its lowest bin, which may hold nearly everything, is
    // counted in registers: atomics on one address are served one after the other.
    if (wide) {
      unsigned low = 0;
#pragma unroll
      for (int e = 0; e < kPer; ++e)
        if (e < mine) {
          const unsigned d = key[e] > lo ? (key[e] - lo) >> 16 : 0u;
          if (d == 0) ++low;
          else atomicAdd(&hist[min(d, (unsigned)kBins - 1u)], 1u);
        }
      low = __reduce_add_sync(0xffffffffu, low);
      if (lane == 0 && low) atomicAdd(&hist[0], low);
    } else {
#pragma unroll
      for (int e = 0; e < kPer; ++e)
        if (e < mine && key[e] - lo <= hi - lo) atomicAdd(&hist[(key[e] - lo) >> shift], 1u);
    }
    if (kCluster) cl.sync(); else __syncthreads();
    // thread t has bins 4 (511 - t) .. + 3, so that the prefix sum runs from the largest digit down
    const int b4 = 4 * (kThreads - 1 - tid);
    uint4 h = *reinterpret_cast<const uint4*>(&hist[b4]);
    if (kCluster) {
      for (int r = 1; r < C; ++r) {
        const int other = rank + r < C ? rank + r : rank + r - C;   // each CTA starts with another neighbour
        const uint4 x = *reinterpret_cast<const uint4*>(cl.map_shared_rank(&hist[b4], other));
        h.x += x.x; h.y += x.y; h.z += x.z; h.w += x.w;
      }
    }
    unsigned total;
    const unsigned sum = h.x + h.y + h.z + h.w, above = block_scan(sum, scan_tot[0], total);
    if (above < need && above + sum >= need) {          // exactly one thread
      unsigned higher = above, in = h.w;
      int d = b4 + 3;
      if (higher + in < need) { higher += in; in = h.z; --d; }
      if (higher + in < need && d == b4 + 2) { higher += in; in = h.y; --d; }
      if (higher + in < need && d == b4 + 1) { higher += in; in = h.x; --d; }
      sh_bin = (unsigned)d; sh_need = need - higher; sh_in_bin = in;
    }
    __syncthreads();
    const unsigned bin = sh_bin, in_bin = sh_in_bin;
    need = sh_need;
    {
      const unsigned first_key = lo + (bin << shift), last_key = first_key + ((1u << shift) - 1u);
      if (!(wide && bin == kBins - 1)) hi = min(hi, last_key);
      lo = wide && bin == 0 ? 0u : first_key;
    }
    if (lo == hi) {                                     // one key is left
      thr = lo;
      need_eq = (int)need;
      break;
    }
    if (in_bin == need && lo != 0) {                    // the whole bin is kept: everything from its smallest key up
      thr = lo - 1;
      break;
    }
    if (in_bin <= (unsigned)kList) {
      // rank the bin's tokens against each other: the list of the cluster's first CTA, then a copy in every CTA
      unsigned* ln = kCluster ? cl.map_shared_rank(&list_n, 0) : &list_n;
      unsigned* lk = kCluster ? cl.map_shared_rank(list_key, 0) : list_key;
#pragma unroll
      for (int e = 0; e < kPer; ++e)
        if (e < mine && key[e] - lo <= hi - lo) lk[atomicAdd(ln, 1u)] = key[e];
      if (kCluster) {
        cl.sync();
        if (rank != 0 && tid < (int)in_bin) list_key[tid] = lk[tid];
      } else {
        __syncthreads();
      }
      if (tid < 4) list_key[in_bin + tid] = 0u;         // read four at a time; a zero is greater than nothing
      __syncthreads();
      if (tid < (int)in_bin) {
        const unsigned k = list_key[tid];
        unsigned greater = 0, equal = 0;
#pragma unroll 2
        for (unsigned t = 0; t < in_bin; t += 4) {
          const uint4 o = *reinterpret_cast<const uint4*>(&list_key[t]);
          greater += (o.x > k) + (o.y > k) + (o.z > k) + (o.w > k);
          equal += (o.x == k) + (o.y == k) + (o.z == k) + (o.w == k);
        }
        // the key whose equals straddle rank `need`; several threads hold it and write the same two numbers
        if (greater < need && greater + equal >= need) { sh_thr = k; sh_need_eq = need - greater; }
      }
      __syncthreads();
      thr = sh_thr;
      need_eq = (int)sh_need_eq;
      break;
    }
    // too many for the list: a histogram over what is left
    if (kCluster) cl.sync(); else __syncthreads();
    *reinterpret_cast<uint4*>(&hist[4 * tid]) = make_uint4(0, 0, 0, 0);
    shift = max(0, 32 - __clz(hi - lo) - 11);
    __syncthreads();
  }

  // ---- ordered emission: greater and equal counts of a thread in one word (a CTA has at most 8192 tokens) ----
  unsigned own = 0;
#pragma unroll
  for (int e = 0; e < kPer; ++e)
    if (e < mine) own += key[e] > thr ? 1u : key[e] == thr ? 1u << 16 : 0u;
  unsigned total;
  const unsigned before = block_scan(own, scan_tot[1], total);
  int gt = (int)(before & 0xffffu), eq = (int)(before >> 16);
  if (kCluster) {
    if (tid == 0) cta_count = total;
    cl.sync();
    const unsigned x = lane < rank ? *cl.map_shared_rank(&cta_count, lane) : 0u;
    gt += __reduce_add_sync(0xffffffffu, (int)(x & 0xffffu));
    eq += __reduce_add_sync(0xffffffffu, (int)(x >> 16));
    cl.barrier_arrive();                                // done with the others' shared memory
  }
  griddep_launch();
  if (own != 0) {
    // this thread's kept tokens follow one another: those above the threshold and the equals still wanted
    const int at = gt + min(eq, need_eq), eq_end = need_eq - eq;
    int seen_eq = 0, k = at;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      if (e < mine && key[e] >= thr) {
        const bool keep = key[e] > thr || seen_eq < eq_end;
        seen_eq += key[e] == thr;
        if (keep) {
          out[k] = j0 + e;
          if (so) so[k] = s[e];
          ++k;
        }
      }
    }
  }
  if (!kCluster && a.k_out) gather_rows(a, pl, out, unit, min(n, bud));
  if (kCluster) cl.barrier_wait();                      // nobody leaves while its shared memory may still be read
}

// The accumulated score without value prior: no head-wide maximum, so a plain sweep over all tokens.
__global__ void __launch_bounds__(256) combine_kernel(const float* s_raw, const float* prev, float* score, const Shape pl,
                                                      const int slots) {
  griddep_wait();
  const int j = blockIdx.x * 256 + threadIdx.x, unit = blockIdx.y, n = pl.n;
  if (j < n) {
    float s = combine_slots(s_raw, (size_t)unit * slots * n + j, n, slots, pl.group_max);
    if (prev) s = __fadd_rn(s, prev[(size_t)unit * n + j]);
    score[(size_t)unit * n + j] = s;
  }
}

// ---- contexts beyond what a cluster holds: one CTA per head, passes over global memory ----
constexpr int kWideThreads = 1024;
constexpr int kWideWarps = kWideThreads / 32;


__device__ __forceinline__ float block_max(float x, float* red) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  float m = red[0];
  for (int w = 1; w < kWideWarps; ++w) m = fmaxf(m, red[w]);
  __syncthreads();
  return m;
}

__global__ void __launch_bounds__(kWideThreads) refine_kernel(const float* __restrict__ s_raw, const float* __restrict__ nu,
                                                          const float* __restrict__ prev, float* __restrict__ score,
                                                          const Shape pl, const int slots) {
  __shared__ float red[kWideWarps];
  const int unit = blockIdx.x, n = pl.n, half = pl.pool / 2;
  const bool prior = nu != nullptr;
  const float inv_w = 1.f / (float)pl.pool;
  const bool zero_pad = (pl.flags & AHAKV_FLAG_POOL_ZERO_PAD) != 0;
  const float* nu_u = prior ? nu + (size_t)unit * n : nullptr;
  float inv_gmax = 1.f;
  if (prior) {
    float m = 0.f;
    for (int j = threadIdx.x; j < n; j += kWideThreads) m = fmaxf(m, pooled(nu_u, j, n, half, inv_w, zero_pad));
    inv_gmax = __frcp_rn(block_max(m, red));
  }
  for (int j = threadIdx.x; j < n; j += kWideThreads) {
    float s = combine_slots(s_raw, (size_t)unit * slots * n + j, n, slots, pl.group_max);
    if (prior) s = __fmul_rn(__fmul_rn(pooled(nu_u, j, n, half, inv_w, zero_pad), inv_gmax), s);
    if (prev) s = __fadd_rn(s, prev[(size_t)unit * n + j]);
    score[(size_t)unit * n + j] = s;
  }
}

// The digit at which the count of keys, taken from the largest digit down, reaches `need`: a suffix scan of
// the 256-bin histogram by 256 threads.  Writes the extended prefix and how many keys of that digit are still
// needed; ends with a barrier.
__device__ __forceinline__ void find_digit(const unsigned* hist, unsigned need, unsigned prefix, int shift,
                                           unsigned* out_prefix, unsigned* out_need, unsigned* warp_tot) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  unsigned h = 0, inc = 0;
  if (t < 256) {
    h = hist[255 - t];                         // thread t looks at digit 255 - t
    inc = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) warp_tot[warp] = inc;
  }
  __syncthreads();
  if (t < 256) {
    for (int w = 0; w < warp; ++w) inc += warp_tot[w];
    if (inc >= need && inc - h < need) {       // exactly one digit crosses
      *out_prefix = prefix | ((unsigned)(255 - t) << shift);
      *out_need = need - (inc - h);
    }
  }
  __syncthreads();
}

// Entries of a head's index row beyond the tokens it keeps (heads with a budget of their own only).
__device__ __forceinline__ void pad_kept(int32_t* out, int kept_here, int n_keep) {
  for (int t = kept_here + threadIdx.x; t < n_keep; t += kWideThreads) out[t] = -1;
}

__global__ void __launch_bounds__(kWideThreads) select_kernel(const float* __restrict__ score, int32_t* __restrict__ kept,
                                                          const Shape pl, const int32_t* __restrict__ budgets) {
  __shared__ unsigned hist[256];
  __shared__ unsigned sh_prefix, sh_need, scan_tot[8];
  __shared__ int warp_gt[kWideWarps], warp_eq[kWideWarps];
  __shared__ int run_gt, run_eq;
  const int unit = blockIdx.x, n = pl.n;
  const float* s = score + (size_t)unit * n;
  int32_t* out = kept + (size_t)unit * pl.n_keep;
  const int bud = head_budget(pl, budgets, unit);
  pad_kept(out, min(n, bud), pl.n_keep);
  if (n <= bud) {                          // nothing to evict
    for (int j = threadIdx.x; j < n; j += kWideThreads) out[j] = j;
    return;
  }
  const int n_cand = n - pl.Br, Bs = bud - pl.Br;
  for (int t = threadIdx.x; t < pl.Br; t += kWideThreads) out[Bs + t] = n_cand + t;   // recent window
  if (Bs == 0) return;

  // ---- radix select: key of the Bs-th largest candidate --------------------
  unsigned prefix = 0, need = (unsigned)Bs;     // `need` elements still to take among keys matching prefix
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    const unsigned mask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
    if (threadIdx.x < 256) hist[threadIdx.x] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < n_cand; j += kWideThreads) {
      const unsigned key = order_key(s[j]);
      if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    find_digit(hist, need, prefix, shift, &sh_prefix, &sh_need, scan_tot);
    prefix = sh_prefix;
    need = sh_need;
    __syncthreads();
  }
  const unsigned thr = prefix;              // exact key of the threshold score
  const int need_eq = (int)need;            // how many keys equal to thr are kept (lowest index first)

  // ---- ordered emission ------------------------------------------------------
  if (threadIdx.x == 0) { run_gt = 0; run_eq = 0; }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int base = 0; base < n_cand; base += kWideThreads) {
    const int j = base + threadIdx.x;
    bool gt = false, eq = false;
    if (j < n_cand) {
      const unsigned key = order_key(s[j]);
      gt = key > thr;
      eq = key == thr;
    }
    const unsigned bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
    const unsigned below = (1u << lane) - 1u;
    if (lane == 0) { warp_gt[warp] = __popc(bg); warp_eq[warp] = __popc(be); }
    __syncthreads();
    int gt_before = run_gt + __popc(bg & below), eq_before = run_eq + __popc(be & below);
    for (int w = 0; w < warp; ++w) { gt_before += warp_gt[w]; eq_before += warp_eq[w]; }
    if (gt || (eq && eq_before < need_eq)) out[gt_before + min(eq_before, need_eq)] = j;
    __syncthreads();
    if (threadIdx.x == kWideThreads - 1) {
      run_gt = gt_before + (gt ? 1 : 0);
      run_eq = eq_before + (eq ? 1 : 0);
    }
    __syncthreads();
  }
}

template <int kPer, bool kCluster>
cudaError_t launch_as(const SelectArgs& a, const Shape& pl, int C, cudaStream_t st) {
  if (C > 8) {
    // leave to use clusters beyond the portable size, asked for once per device
    constexpr int kMaxDevices = 64;
    static bool configured[kMaxDevices] = {};
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
      e = cudaFuncSetAttribute(refine_select_kernel<kPer, kCluster>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
      configured[dev] = true;
    }
  }
  return launch_chained(refine_select_kernel<kPer, kCluster>, dim3(pl.B * pl.Hkv * C), dim3(kThreads), kCluster ? C : 1, 0, st, a, pl);
}

// One cluster per head.  False: no cluster holds a head.
bool launch_clustered(SelectArgs a, const Shape& pl, cudaStream_t st, cudaError_t* err) {
  if (pl.n > kMaxCluster * kThreads * kMaxPer) return false;   // 131072 tokens
  // Eight tokens a thread and two CTAs an SM while all heads' clusters fit on the GPU at once; beyond that sixteen, whose
  // smaller clusters exchange less (256 heads of 32768 tokens: 103 us against 115; 32 of 16384: 19 against 15).
  const long long ctas8 = (long long)pl.B * pl.Hkv * ((pl.n + kThreads * 8 - 1) / (kThreads * 8));
  const int per_cta = kThreads * (ctas8 > 2 * 148 ? 16 : 8);
  int C = (pl.n + per_cta - 1) / per_cta;
  if (C > kMaxCluster) C = kMaxCluster;
  a.chunk = ((pl.n + C - 1) / C + kMaxPer - 1) / kMaxPer * kMaxPer;
  const int per = (a.chunk + kThreads - 1) / kThreads;
  if (C == 1) {
    *err = per <= 1 ? launch_as<1, false>(a, pl, C, st) : per <= 2 ? launch_as<2, false>(a, pl, C, st)
         : per <= 4 ? launch_as<4, false>(a, pl, C, st) : per <= 8 ? launch_as<8, false>(a, pl, C, st) : launch_as<16, false>(a, pl, C, st);
  } else {
    *err = per <= 4 ? launch_as<4, true>(a, pl, C, st) : per <= 8 ? launch_as<8, true>(a, pl, C, st)
                                                                 : launch_as<kMaxPer, true>(a, pl, C, st);
  }
  return true;
}

}  // namespace

ahakv_status launch_refine(const Plan& pl, const float* s_raw, const float* nu, const float* score_prev,
                           float* score, int slots, cudaStream_t st) {
  SelectArgs a = {};
  a.s_raw = s_raw; a.nu = nu; a.prev = score_prev; a.score = score; a.slots = slots;
  const Shape& shape = pl;
  cudaError_t e = cudaSuccess;
  if (!nu) {
    e = launch_chained(combine_kernel, dim3((pl.n + 255) / 256, pl.B * pl.Hkv), dim3(256), 1, 0, st, s_raw, score_prev, score, shape, slots);
  } else if (!launch_clustered(a, pl, st, &e)) {
    refine_kernel<<<pl.B * pl.Hkv, kWideThreads, 0, st>>>(s_raw, nu, score_prev, score, pl, slots);
    e = cudaGetLastError();
  }
  count_launch();
  return cuda_ok(e);
}

ahakv_status launch_select(const Plan& pl, const float* score, int32_t* kept_idx, cudaStream_t st) {
  SelectArgs a = {};
  a.s_raw = score; a.kept = kept_idx; a.slots = 1;
  cudaError_t e = cudaSuccess;
  if (!launch_clustered(a, pl, st, &e)) {
    select_kernel<<<pl.B * pl.Hkv, kWideThreads, 0, st>>>(score, kept_idx, pl, nullptr);
    e = cudaGetLastError();
  }
  count_launch();
  return cuda_ok(e);
}

ahakv_status launch_refine_select(const Plan& pl, const float* s_raw, const float* nu, const float* score_prev,
                                  float* score, float** score_left, float* score_out, int32_t* kept_idx, int slots,
                                  const int32_t* budgets, const void* k, const void* v, void* k_out, void* v_out, bool* gathered,
                                  cudaStream_t st) {
  SelectArgs a = {};
  a.s_raw = s_raw; a.nu = nu; a.prev = score_prev; a.score_out = score_out; a.kept = kept_idx; a.budgets = budgets; a.slots = slots;
  // The CTA that selects a head also gathers its rows when that is a launch saved and little to move: one CTA a head, at
  // most 128 KB in and as much out (beyond, a gather spread over the whole GPU is faster).
  *gathered = pl.n <= kThreads * 8 && (size_t)2 * pl.n_keep * pl.d * pl.es <= 128 * 1024;
  if (*gathered) {
    a.k = (const char*)k; a.v = (const char*)v; a.k_out = (char*)k_out; a.v_out = (char*)v_out;
    a.lanes = pl.d * pl.es / 16;
  }
  cudaError_t e = cudaSuccess;
  if (launch_clustered(a, pl, st, &e)) {
    *score_left = nullptr;
    count_launch();
    return cuda_ok(e);
  }
  refine_kernel<<<pl.B * pl.Hkv, kWideThreads, 0, st>>>(s_raw, nu, score_prev, score, pl, slots);
  select_kernel<<<pl.B * pl.Hkv, kWideThreads, 0, st>>>(score, kept_idx, pl, budgets);
  *score_left = score;
  count_launch(2);
  return cuda_ok(cudaGetLastError());
}

}  // namespace ahakv

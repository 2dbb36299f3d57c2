// The generation phase one token at a time (Algorithm 1, Generation: A = q_t K^T, F_t = SGsoftmax(A) + F_{t-1},
// then S = TopK(F_t, B_s) U recent B_r and K <- K_S, V <- V_S before the next token).
//
// step_kernel: a cluster of C CTAs per (sequence, KV head), each a contiguous piece of the keys.  The G query rows of the
//   group (one new query per head) against the n cached keys is a matrix-vector product, bound by reading K once.
//   16-bit inputs: warp-level m16n8k16 products, the heads on the rows and eight keys on the columns; every warp keeps four
//   blocks of eight keys in flight and folds a block's logits into its running (shift, sum) as it goes.  float32 inputs:
//   half a warp (or a quarter, by row size) reads one key row with 16-byte loads, every lane keeps its slice of the G
//   queries in registers, and the partial dot products meet by shuffle.  The G x n logits stay in shared memory, so
//   that after one exchange of the warps' statistics the new score is written in a single sweep.  No scratch memory,
//   no second read of K.  At 128 heads x 2049 keys (67 MB): 16.7 us, 4.0 TB/s, of which the loads take 11; it was 21.7 with
//   one CTA a head, a straggling last round of loads and two sweeps over the logits between block-wide reductions.
//   8 heads: 8.2 us (17.5).  Asking the keys into L2 ahead of the launch's turn gained nothing.
//   For a cache kept as slots (kSlots) it also copies the new token's rows into the free slot and names the slot that
//   becomes free (smallest score outside the recent window).
//
// compact_inplace_kernel: a cluster of CTAs per (sequence, KV head).  kept_idx is ascending, so row t of the result comes
//   from row kept_idx[t] >= t: rows before the first evicted index do not move at all, and the others move in rounds
//   through registers (all loads of a round, a barrier over the cluster, all its stores), so no row is overwritten
//   before it has been read.  128 heads x 2049 rows of 256 bytes, half of them moving (67 MB each way): 26 us; one CTA a head
//   with batches through shared memory took 62.
#include <cooperative_groups.h>

#include <type_traits>

#include "ahakv_internal.cuh"
#include "mma_sync.cuh"
#include "select_common.cuh"

namespace ahakv {
namespace {

namespace cg = cooperative_groups;

constexpr int kStepThreads = 512;
constexpr int kStepWarps = kStepThreads / 32;
constexpr int kStepMaxG = 16;                  // query heads per KV head the step kernel takes
constexpr size_t kStepMaxLogitBytes = 160 * 1024;   // 40960 logits
constexpr int kStepMaxCluster = 8;
constexpr int kStepHeldG = 5;                  // float32: heads whose queries are held in registers

template <typename T> using Acc = typename std::conditional<std::is_same<T, float>::value, double, float>::type;

struct StepArgs {
  const void* q;             // [B,Hq,1,d]
  const void* k;             // the cache
  const float* prev;         // F_{t-1}, or null
  float* score;              // F_t
  double c;                  // lambda log2(e)
  int chunk;                 // keys per CTA, a multiple of 8
  // slots only
  const void *k_new, *v_new;
  void *k_out, *v_out;       // the cache again, to be written to
  int32_t *pos, *free_slot;
  int new_pos;
};

// A running softmax: Z = sum of 2^{x - M}.  M is a shift, not necessarily the maximum: it moves only when a logit outruns
// it by so much that the sum would suffer.
__device__ __forceinline__ void fold_logits(float x0, float x1, float& M, float& Z) {
  const float mx = fmaxf(x0, x1);
  if (mx > M + 32.f) {                              // the first logits of a thread always come this way: M = -inf
    Z = Z > 0.f ? Z * fast_exp2(M - mx) : 0.f;
    M = mx;
  }
  if (mx > -INFINITY) Z += fast_exp2(x0 - M) + fast_exp2(x1 - M);
}
__device__ __forceinline__ void merge_stats(float& M, float& Z, float m, float z) {
  const float t = fmaxf(M, m);
  Z = (Z > 0.f ? Z * fast_exp2(M - t) : 0.f) + (z > 0.f ? z * fast_exp2(m - t) : 0.f);
  M = t;
}

// The G x (k1 - k0) logits of this CTA's keys, in log2 units, into logit[g * pitch + j - k0], and every warp's statistics
// of every head into st[g][warp].  Key `slot` is read from `k_new`.
//
// The sum over d does not care in which order d is walked, so each thread takes one contiguous quarter of a row -- of its
// query head's row for the A operand, of its key's row for the B operand -- and hands its 32-bit words to the instruction in
// pairs: the k-slices the four threads of a group present side by side are then the same permutation of d for A and B.
template <typename T, int D, int kG>
__device__ __forceinline__ void step_logits_mma(const StepArgs& a, const Shape& pl, int b, int h, int k0, int k1, int slot,
                                                float* logit, int pitch, float2 (*st)[kStepWarps]) {
  constexpr int CH = D / 4, W = CH / 2, Q4 = CH / 8;           // a thread's quarter row: elements, 32-bit words, 16-byte loads
  constexpr int kAhead = 4;                                    // 8-key blocks in flight per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane >> 2, tig = lane & 3;
  const float c = (float)a.c;
  const T* kbase = (const T*)a.k + (long long)b * pl.ks[0] + (long long)h * pl.ks[1] + CH * tig;
  const T* fresh = (const T*)a.k_new + ((long long)b * pl.Hkv + h) * D + CH * tig;
  const int n_blocks = (k1 - k0 + 7) / 8;
  uint4 raw[kAhead][Q4];
  const auto load = [&](uint4 (&dst)[Q4], int blk) {
    const int j = k0 + blk * 8 + grp;
    const T* src = j == slot ? fresh : kbase + (long long)j * pl.ks[2];
#pragma unroll
    for (int t = 0; t < Q4; ++t) dst[t] = j < k1 ? *reinterpret_cast<const uint4*>(src + 8 * t) : make_uint4(0, 0, 0, 0);
  };
#pragma unroll
  for (int u = 0; u < kAhead; ++u) load(raw[u], warp + u * kStepWarps);

  // A: head `grp` (and `grp + 8` when there are more than eight) of the group's queries, this thread's quarter
  uint32_t qa[W], qb[W];
#pragma unroll
  for (int t = 0; t < W; ++t) { qa[t] = 0u; qb[t] = 0u; }
  const T* qrow = (const T*)a.q + (long long)b * pl.qs[0] + (long long)(h * pl.G + grp) * pl.qs[1] + CH * tig;
  if (grp < kG) {
#pragma unroll
    for (int t = 0; t < Q4; ++t) {
      const uint4 u = *reinterpret_cast<const uint4*>(qrow + 8 * t);
      qa[4 * t] = u.x; qa[4 * t + 1] = u.y; qa[4 * t + 2] = u.z; qa[4 * t + 3] = u.w;
    }
  }
  if (kG > 8 && grp + 8 < kG) {
#pragma unroll
    for (int t = 0; t < Q4; ++t) {
      const uint4 u = *reinterpret_cast<const uint4*>(qrow + 8 * pl.qs[1] + 8 * t);
      qb[4 * t] = u.x; qb[4 * t + 1] = u.y; qb[4 * t + 2] = u.z; qb[4 * t + 3] = u.w;
    }
  }
  float M0 = -INFINITY, Z0 = 0.f, M1 = -INFINITY, Z1 = 0.f;     // heads grp and grp + 8
  for (int blk0 = warp; blk0 < n_blocks; blk0 += kAhead * kStepWarps) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int blk = blk0 + u * kStepWarps;
      if (blk >= n_blocks) break;                                // uniform over the warp
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int t = 0; t < Q4; ++t) {
        // two k-steps a 16-byte load: words (0, 1) and (2, 3)
        Mma16816<T>::run(acc, qa[4 * t], qb[4 * t], qa[4 * t + 1], qb[4 * t + 1], raw[u][t].x, raw[u][t].y);
        Mma16816<T>::run(acc, qa[4 * t + 2], qb[4 * t + 2], qa[4 * t + 3], qb[4 * t + 3], raw[u][t].z, raw[u][t].w);
      }
      load(raw[u], blk + kAhead * kStepWarps);
      const int i = blk * 8 + 2 * tig;
      const bool v0 = k0 + i < k1, v1 = k0 + i + 1 < k1;
      if (grp < kG) {
        const float x0 = acc[0] * c, x1 = acc[1] * c;
        *reinterpret_cast<float2*>(&logit[grp * pitch + i]) = make_float2(x0, x1);
        fold_logits(v0 ? x0 : -INFINITY, v1 ? x1 : -INFINITY, M0, Z0);
      }
      if (kG > 8 && grp + 8 < kG) {
        const float x0 = acc[2] * c, x1 = acc[3] * c;
        *reinterpret_cast<float2*>(&logit[(grp + 8) * pitch + i]) = make_float2(x0, x1);
        fold_logits(v0 ? x0 : -INFINITY, v1 ? x1 : -INFINITY, M1, Z1);
      }
    }
  }
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    // both partners add in the same order: the lower thread's set first
    const float m0 = __shfl_xor_sync(0xffffffffu, M0, o), z0 = __shfl_xor_sync(0xffffffffu, Z0, o);
    const float m1 = __shfl_xor_sync(0xffffffffu, M1, o), z1 = __shfl_xor_sync(0xffffffffu, Z1, o);
    merge_stats(M0, Z0, m0, z0);                                 // a sum of two is the same either way round
    if (kG > 8) merge_stats(M1, Z1, m1, z1);
  }
  if (tig == 0 && grp < kG) st[grp][warp] = make_float2(M0, Z0);
  if (kG > 8 && tig == 0 && grp + 8 < kG) st[grp + 8][warp] = make_float2(M1, Z1);
}

// The same for float32 inputs, dot products in double.  LANES threads share a key row (16 bytes each); kG query heads.
template <typename T, int D, int kG>
__device__ __forceinline__ void step_logits_simt(const StepArgs& a, const Shape& pl, int b, int h, int k0, int k1, int slot,
                                                 float* logit, int pitch, float2 (*st)[kStepWarps]) {
  using A = Acc<T>;
  constexpr int V = Vec16<T>::N, LANES = D / V, KEYS_PER_WARP = 32 / LANES;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % LANES, which = lane / LANES;
  const A c = (A)a.c;
  // The group's queries in double, converted once (a conversion costs as much as four multiply-adds): this lane's slices in
  // registers, or, for more than kStepHeldG heads, the rows in shared memory.
  constexpr bool kHeld = kG <= kStepHeldG;
  __shared__ __align__(16) A q_sm[kHeld ? 1 : kG][D];
  A qreg[kHeld ? kG : 1][V];
  const auto query = [&](int g, A (&to)[V]) {
    float f[V];
    Vec16<T>::widen(*reinterpret_cast<const uint4*>((const T*)a.q + (long long)b * pl.qs[0] + (long long)(h * pl.G + g) * pl.qs[1] + sub * V), f);
#pragma unroll
    for (int e = 0; e < V; ++e) to[e] = (A)f[e];
  };
  const char* kbase = reinterpret_cast<const char*>((const T*)a.k + (long long)b * pl.ks[0] + (long long)h * pl.ks[1] + sub * V);
  // where the new token's row lies, seen from there
  const long long fresh = reinterpret_cast<intptr_t>((const T*)a.k_new + ((long long)b * pl.Hkv + h) * D + sub * V) - reinterpret_cast<intptr_t>(kbase);
  constexpr int kUnroll = 4;                                     // key rows in flight per lane
  const int stride = kStepWarps * KEYS_PER_WARP;
  uint4 raw[kUnroll];
  const auto load = [&](int j0) {
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int j = j0 + u * stride;
      raw[u] = make_uint4(0, 0, 0, 0);
      if (j < k1) raw[u] = *reinterpret_cast<const uint4*>(kbase + (j == slot ? fresh : (long long)j * pl.ks[2] * (long long)sizeof(T)));
    }
  };
  load(k0 + warp * KEYS_PER_WARP + which);
  if (kHeld) {
#pragma unroll
    for (int g = 0; g < kG; ++g) query(g, qreg[kHeld ? g : 0]);
  } else {
    for (int g = threadIdx.x / LANES; g < kG; g += kStepThreads / LANES) {
      A x[V];
      query(g, x);
#pragma unroll
      for (int e = 0; e < V; ++e) q_sm[kHeld ? 0 : g][sub * V + e] = x[e];
    }
    __syncthreads();
  }
  // The next rows are asked for before this round's are multiplied (the stores of the logits keep the compiler from doing so by
  // itself), and the reductions of four keys run side by side.  Without either, 512 heads of four queries x 513 keys of 512
  // bytes took 180 us, now 78; 128 x 1025 72, now 34.
  for (int j0 = k0 + warp * KEYS_PER_WARP + which; j0 - which < k1; j0 += stride * kUnroll) {
    A kv[kUnroll][V];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      float f[V];
      Vec16<T>::widen(raw[u], f);
#pragma unroll
      for (int e = 0; e < V; ++e) kv[u][e] = (A)f[e];
    }
    load(j0 + stride * kUnroll);
#pragma unroll
    for (int g = 0; g < kG; ++g) {
      A acc[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        acc[u] = 0;
#pragma unroll
        for (int e = 0; e < V; ++e) acc[u] = fma(kHeld ? qreg[kHeld ? g : 0][e] : q_sm[kHeld ? 0 : g][sub * V + e], kv[u][e], acc[u]);
      }
#pragma unroll
      for (int o = LANES / 2; o; o >>= 1) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
      }
      // every lane has the sums of its four rows: lane u of a row stores that of key u
      A mine = acc[0];
#pragma unroll
      for (int u = 1; u < kUnroll; ++u) mine = sub == u ? acc[u] : mine;
      const int j = j0 + sub * stride;
      if (sub < kUnroll && j < k1) logit[g * pitch + j - k0] = (float)(mine * c);    // log2 units
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int g = 0; g < kG; ++g) {
    float M = -INFINITY, Z = 0.f;
    for (int i = threadIdx.x; i < k1 - k0; i += kStepThreads) fold_logits(logit[g * pitch + i], -INFINITY, M, Z);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float m = __shfl_xor_sync(0xffffffffu, M, o), z = __shfl_xor_sync(0xffffffffu, Z, o);
      merge_stats(M, Z, m, z);
    }
    if (lane == 0) st[g][warp] = make_float2(M, Z);
  }
}

// (M, Z) pairs of kG heads, `count` <= 16 of each, from at(g, i): every warp ends up with the heads' totals in every lane.
template <int kG, typename F>
__device__ __forceinline__ void reduce_stats(int count, F at, float (&M)[kG], float (&Z)[kG]) {
  const int lane = threadIdx.x & 31, half = lane >> 4, i = lane & 15;
#pragma unroll
  for (int g0 = 0; g0 < kG; g0 += 2) {
    float m = -INFINITY, z = 0.f;
    if (g0 + half < kG && i < count) {
      const float2 x = at(g0 + half, i);
      m = x.x; z = x.y;
    }
    float mx = m;
#pragma unroll
    for (int o = 8; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    z = z > 0.f ? z * fast_exp2(m - mx) : 0.f;
#pragma unroll
    for (int o = 8; o; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    M[g0] = __shfl_sync(0xffffffffu, mx, 0);
    Z[g0] = __shfl_sync(0xffffffffu, z, 0);
    if (g0 + 1 < kG) {
      M[(g0 + 1) % kG] = __shfl_sync(0xffffffffu, mx, 16);
      Z[(g0 + 1) % kG] = __shfl_sync(0xffffffffu, z, 16);
    }
  }
}

template <typename T, int D, int kG, bool kSlots, bool kCluster>
__global__ void __launch_bounds__(kStepThreads, std::is_same<T, float>::value && kG == 1 ? 2 : 1) step_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ Shape pl) {
  extern __shared__ __align__(16) float logit[];                 // [kG][chunk]
  __shared__ float2 st[kG][kStepWarps], cta_st[kG];
  __shared__ unsigned long long best[kStepWarps], cta_best;
  cg::cluster_group cl = cg::this_cluster();
  const int C = kCluster ? (int)cl.num_blocks() : 1, rank = kCluster ? (int)cl.block_rank() : 0;
  const int unit = kCluster ? blockIdx.x / C : blockIdx.x, b = unit / pl.Hkv, h = unit % pl.Hkv, n = pl.n;
  const int k0 = min(rank * a.chunk, n), k1 = min(k0 + a.chunk, n), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  griddep_wait();
  int slot = -1;
  if (kSlots) {
    slot = a.free_slot[unit];
    if (slot < 0 || slot >= n) return;                           // the caller's table is broken: touch nothing
    if (slot >= k0 && slot < k1) {                               // the new token moves in; below its key is read from k_new
      constexpr int V = Vec16<T>::N, LANES = D / V;
      if (threadIdx.x < 2 * LANES) {
        const int sub = threadIdx.x % LANES;
        const bool is_v = threadIdx.x >= LANES;
        const T* src = (const T*)(is_v ? a.v_new : a.k_new) + ((long long)b * pl.Hkv + h) * D + sub * V;
        T* dst = is_v ? (T*)a.v_out + (long long)b * pl.vs[0] + (long long)h * pl.vs[1] + (long long)slot * pl.vs[2] + sub * V
                      : (T*)a.k_out + (long long)b * pl.ks[0] + (long long)h * pl.ks[1] + (long long)slot * pl.ks[2] + sub * V;
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
      }
    }
  }
  // the first tokens' carried scores (and positions) while the keys are on their way
  constexpr int kPre = 4;
  const float* prev = kSlots ? a.score : a.prev;
  float f[kPre];
  int ps[kPre];
#pragma unroll
  for (int t = 0; t < kPre; ++t) {
    const int j = k0 + t * kStepThreads + (int)threadIdx.x;
    f[t] = prev && j < k1 ? prev[(size_t)unit * n + j] : 0.f;
    if (kSlots) ps[t] = j < k1 ? a.pos[(size_t)unit * n + j] : 0;
  }
  if constexpr (std::is_same<T, float>::value) step_logits_simt<T, D, kG>(a, pl, b, h, k0, k1, slot, logit, a.chunk, st);
  else step_logits_mma<T, D, kG>(a, pl, b, h, k0, k1, slot, logit, a.chunk, st);
  griddep_launch();
  __syncthreads();

  // shift and normaliser of every head
  float M[kG], Z[kG];
  reduce_stats<kG>(kStepWarps, [&](int g, int i) { return st[g][i]; }, M, Z);
  if (kCluster) {
    if (threadIdx.x == 0) {
#pragma unroll
      for (int g = 0; g < kG; ++g) cta_st[g] = make_float2(M[g], Z[g]);
    }
    cl.sync();
    reduce_stats<kG>(C, [&](int g, int i) { return *cl.map_shared_rank(&cta_st[g], i); }, M, Z);
  }
  const float inv_g = pl.group_max ? 1.f : 1.f / (float)kG;
#pragma unroll
  for (int g = 0; g < kG; ++g) Z[g] = inv_g / Z[g];

  // F_t = SGsoftmax(A_t) + F_{t-1}, and for slots the candidate to leave: smallest score, then largest position
  const int oldest_protected = a.new_pos - pl.Br + 1;            // positions from here on are the recent window
  unsigned long long mine = ~0ull;
  int mine_j = -1;
  const auto update = [&](int j, float old, int pj) {
    const int i = j - k0;
    float s = fast_exp2(logit[i] - M[0]) * Z[0];
#pragma unroll
    for (int g = 1; g < kG; ++g) {
      const float w = fast_exp2(logit[g * a.chunk + i] - M[g]) * Z[g];
      s = pl.group_max ? fmaxf(s, w) : s + w;
    }
    if (kSlots) {
      if (j == slot) pj = a.new_pos;                             // a new token starts at zero
      else s = __fadd_rn(s, old);
      if (pj < oldest_protected) {
        // ascending in (score, -position): the position is below 2^31, so its complement orders it downwards within 32 bits
        const unsigned long long key = ((unsigned long long)order_key(s) << 32) | (unsigned)(0x7fffffff - pj);
        if (key < mine) { mine = key; mine_j = j; }
      }
    } else if (prev) {
      s = __fadd_rn(s, old);
    }
    a.score[(size_t)unit * n + j] = s;
  };
#pragma unroll
  for (int t = 0; t < kPre; ++t) {
    const int j = k0 + t * kStepThreads + (int)threadIdx.x;
    if (j < k1) update(j, f[t], kSlots ? ps[t] : 0);
  }
  for (int j = k0 + kPre * kStepThreads + (int)threadIdx.x; j < k1; j += kStepThreads)
    update(j, prev ? prev[(size_t)unit * n + j] : 0.f, kSlots ? a.pos[(size_t)unit * n + j] : 0);
  if (!kSlots) {
    if (kCluster) cl.sync();
    return;
  }
  // the smallest key of the block, then of the cluster; positions are distinct, so one thread has it
  unsigned long long win = mine;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, win, o);
    if (y < win) win = y;
  }
  if (lane == 0) best[warp] = win;
  __syncthreads();
  win = best[lane & (kStepWarps - 1)];
#pragma unroll
  for (int o = 8; o; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, win, o);
    if (y < win) win = y;
  }
  if (kCluster) {
    if (threadIdx.x == 0) cta_best = win;
    cl.sync();
    win = *cl.map_shared_rank(&cta_best, lane < C ? lane : 0);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, win, o);
      if (y < win) win = y;
    }
    cl.barrier_arrive();
  }
  if (win == ~0ull) {                                            // no slot outside the recent window: a broken position table
    if (rank == 0 && threadIdx.x == 0) a.free_slot[unit] = -1;
  } else {
    const bool leaves = mine == win;
    if (threadIdx.x == 0 && slot >= k0 && slot < k1) a.pos[(size_t)unit * n + slot] = a.new_pos;
    __syncthreads();                                             // the new token itself may be the one to leave
    if (leaves) {
      a.pos[(size_t)unit * n + mine_j] = -1;
      a.free_slot[unit] = mine_j;
    }
  }
  if (kCluster) cl.barrier_wait();                               // nobody leaves while its shared memory may still be read
}

template <typename T, int D, int kG, bool kSlots, bool kCluster>
ahakv_status launch_step_as(const StepArgs& a, const Shape& pl, int C, cudaStream_t st) {
  const size_t smem = (size_t)kG * a.chunk * sizeof(float);
  if (smem > 24 * 1024) {                                        // beside up to 18 KB of static shared memory
    constexpr int kMaxDevices = 64;
    static bool configured[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return AHAKV_ERR_CUDA;
    if (!configured[dev]) {
      if (cudaFuncSetAttribute(step_kernel<T, D, kG, kSlots, kCluster>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kStepMaxLogitBytes + 8 * kStepMaxG * (int)sizeof(float)) != cudaSuccess)
        return AHAKV_ERR_CUDA;
      configured[dev] = true;
    }
  }
  const cudaError_t e = launch_chained(step_kernel<T, D, kG, kSlots, kCluster>, dim3(pl.B * pl.Hkv * C), dim3(kStepThreads), C, smem, st, a, pl);
  count_launch();
  return cuda_ok(e);
}

template <typename T, int D, bool kSlots, bool kCluster>
ahakv_status launch_step_g(const StepArgs& a, const Shape& pl, int C, cudaStream_t st) {
  switch (pl.G) {
    case 1: return launch_step_as<T, D, 1, kSlots, kCluster>(a, pl, C, st);
    case 2: return launch_step_as<T, D, 2, kSlots, kCluster>(a, pl, C, st);
    case 3: return launch_step_as<T, D, 3, kSlots, kCluster>(a, pl, C, st);
    case 4: return launch_step_as<T, D, 4, kSlots, kCluster>(a, pl, C, st);
    case 5: return launch_step_as<T, D, 5, kSlots, kCluster>(a, pl, C, st);
    case 6: return launch_step_as<T, D, 6, kSlots, kCluster>(a, pl, C, st);
    case 7: return launch_step_as<T, D, 7, kSlots, kCluster>(a, pl, C, st);
    case 8: return launch_step_as<T, D, 8, kSlots, kCluster>(a, pl, C, st);
    case 12: return launch_step_as<T, D, 12, kSlots, kCluster>(a, pl, C, st);
    case 16: return launch_step_as<T, D, 16, kSlots, kCluster>(a, pl, C, st);
    default: return AHAKV_ERR_UNSUPPORTED;
  }
}

template <bool kSlots>
ahakv_status launch_step(StepArgs a, const Shape& pl, cudaStream_t st) {
  // A head's keys are split over as many CTAs as SMs allow (one CTA an SM: its loads in flight take half the registers),
  // as long as each keeps 256 keys: below that the exchanges of the cluster (1 us each) cost more than the shorter chain
  // of loads saves.
  const int units = pl.B * pl.Hkv;
  int C = 1;
  while (C < kStepMaxCluster && units * C * 2 <= 148 && pl.n >= 512 * C) C *= 2;
  a.chunk = ((pl.n + C - 1) / C + 7) / 8 * 8;
  const bool d64 = pl.d == 64;
#define AHAKV_STEP(T) \
  (C > 1 ? (d64 ? launch_step_g<T, 64, kSlots, true>(a, pl, C, st) : launch_step_g<T, 128, kSlots, true>(a, pl, C, st)) \
         : (d64 ? launch_step_g<T, 64, kSlots, false>(a, pl, C, st) : launch_step_g<T, 128, kSlots, false>(a, pl, C, st)))
  switch (pl.dtype) {
    case AHAKV_F32: return AHAKV_STEP(float);
    case AHAKV_F16: return AHAKV_STEP(__half);
    default: return AHAKV_STEP(__nv_bfloat16);
  }
#undef AHAKV_STEP
}

// ---- in-place compaction ------------------------------------------------------------------------------------------
constexpr int kMoveThreads = 256;
constexpr int kMoveVecs = 8;                    // 16-byte pieces of K, and as many of V, a thread holds per round
constexpr int kMovePieces = kMoveThreads * kMoveVecs;   // and a CTA
constexpr int kMoveCluster = 8;                 // at most

// Two CTAs an SM: the rows in flight take 64 registers, and with the 80 that three CTAs leave a thread 20 of them were spilled
// (128 heads x 2049: 32 us against 26; 2048 heads x 513 by one CTA each: 114 against 98).
template <int LANES>                            // 16-byte pieces of a row
__global__ void __launch_bounds__(kMoveThreads, 2) compact_inplace_kernel(char* k, char* v, float* score, const int32_t* kept,
                                                                          const __grid_constant__ Shape pl) {
  constexpr int kRowsCta = kMovePieces / LANES;                // rows a CTA holds per round
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int unit = blockIdx.x / C, n_keep = pl.n_keep, tid = threadIdx.x;
  const long long b = unit / pl.Hkv, h = unit % pl.Hkv;
  const int32_t* idx = kept + (size_t)unit * n_keep;
  const int sub = tid % LANES, row = tid / LANES;
  constexpr int kStep = kMoveThreads / LANES;
  char* kb = k + (b * pl.ks[0] + h * pl.ks[1]) * pl.es + sub * 16;
  char* vb = v + (b * pl.vs[0] + h * pl.vs[1]) * pl.es + sub * 16;
  const long long ktok = pl.ks[2] * pl.es, vtok = pl.vs[2] * pl.es;
  float* sc = score ? score + (size_t)unit * pl.n : nullptr;
  griddep_wait();

  // Rows before the first evicted index stay where they are: the indices are ascending, so idx[t] == t up to there and
  // nowhere after.  Found by probing at a stride, then within the stride.
  int t_begin = 0;
  for (int step = (n_keep + kMoveThreads - 1) / kMoveThreads, span = n_keep;;) {
    const int t = t_begin + tid * step;
    const int same = __syncthreads_count(tid * step < span && t < n_keep && idx[t] == t);
    if (step == 1) { t_begin += same; break; }
    t_begin += max(same - 1, 0) * step;           // the last probe that has not moved (or the start): the first moved row lies behind
    span = step;
    step = (step + kMoveThreads - 1) / kMoveThreads;
  }
  griddep_launch();

  for (int t0 = t_begin; t0 < n_keep; t0 += C * kRowsCta) {
    // this round's rows, in equal pieces: CTA `rank` has rows [lo, hi)
    const int rows = min(C * kRowsCta, n_keep - t0), per = (rows + C - 1) / C;
    const int lo = t0 + min(rank * per, rows), hi = t0 + min((rank + 1) * per, rows);
    uint4 kr[kMoveVecs], vr[kMoveVecs];
    float sr = 0.f;
#pragma unroll
    for (int e = 0; e < kMoveVecs; ++e) {
      const int t = lo + row + e * kStep;
      if (t < hi) {
        const long long j = idx[t];
        kr[e] = *reinterpret_cast<const uint4*>(kb + j * ktok);
        vr[e] = *reinterpret_cast<const uint4*>(vb + j * vtok);
      }
    }
    if (sc && lo + tid < hi) sr = sc[idx[lo + tid]];
    static_assert(kRowsCta <= kMoveThreads, "one thread per row's score");
    cl.sync();                                    // every row of the round has been read; later rounds read rows written by none
#pragma unroll
    for (int e = 0; e < kMoveVecs; ++e) {
      const int t = lo + row + e * kStep;
      if (t < hi) {
        *reinterpret_cast<uint4*>(kb + t * ktok) = kr[e];
        *reinterpret_cast<uint4*>(vb + t * vtok) = vr[e];
      }
    }
    if (sc && lo + tid < hi) sc[lo + tid] = sr;
  }
}

}  // namespace

bool step_score_fits(const Plan& pl) {
  if (pl.r != 1 || pl.G > kStepMaxG || (size_t)pl.G * pl.n * sizeof(float) > kStepMaxLogitBytes) return false;
  return pl.G <= 8 || pl.G == 12 || pl.G == 16;
}

ahakv_status launch_step_score(const Plan& pl, const void* q, const void* k, const float* prev, float* score,
                               cudaStream_t st) {
  StepArgs a = {};
  a.q = q; a.k = k; a.prev = prev; a.score = score;
  a.c = pl.lambda[0] * 1.4426950408889634;
  a.k_new = k;                                    // never read: no key is in the slot -1
  return launch_step<false>(a, pl, st);
}

ahakv_status launch_step_slots(const Plan& pl, const void* q, const void* k_new, const void* v_new, void* k, void* v,
                               float* score, int32_t* pos, int32_t* free_slot, int new_pos, cudaStream_t st) {
  StepArgs a = {};
  a.q = q; a.k = k; a.prev = score; a.score = score;
  a.c = pl.lambda[0] * 1.4426950408889634;
  a.k_new = k_new; a.v_new = v_new; a.k_out = k; a.v_out = v;
  a.pos = pos; a.free_slot = free_slot; a.new_pos = new_pos;
  return launch_step<true>(a, pl, st);
}

ahakv_status launch_compact_inplace(const Plan& pl, void* k, void* v, float* score, const int32_t* kept_idx,
                                    cudaStream_t st) {
  const Shape& shape = pl;
  // CTAs a head: eight while that is little more than the GPU holds.  Otherwise a barrier of a cluster between loads and stores
  // costs more than it spreads: no more CTAs than heads need to fill the GPU a few times over, nor than two rounds of rows
  // need.  us with eight / by this rule, rows of 128 bytes: 2048 heads x 513 177 / 53, 256 heads that keep 512 rows 26 / 10,
  // 1024 heads x 1025 105 / 55; 128 heads x 2049 16 / 15; 8 heads x 2049 5 either way, 14 with one.
  const int lanes = pl.d * pl.es / 16;
  const long long heads = (long long)pl.B * pl.Hkv;
  int C = kMoveCluster;
  while (C > 1 && (heads * C > 1024 || (heads * C > 2 * 148 && 2LL * C * (kMovePieces / lanes) > pl.n_keep))) C /= 2;
  const dim3 grid((unsigned)(heads * C)), block(kMoveThreads);
  cudaError_t e;
  switch (lanes) {
    case 8: e = launch_chained(compact_inplace_kernel<8>, grid, block, C, 0, st, (char*)k, (char*)v, score, kept_idx, shape); break;
    case 16: e = launch_chained(compact_inplace_kernel<16>, grid, block, C, 0, st, (char*)k, (char*)v, score, kept_idx, shape); break;
    default: e = launch_chained(compact_inplace_kernel<32>, grid, block, C, 0, st, (char*)k, (char*)v, score, kept_idx, shape);
  }
  count_launch();
  return cuda_ok(e);
}

}  // namespace ahakv

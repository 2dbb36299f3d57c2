// Internal declarations shared by the translation units of libahakv.so.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ahakv.h"

namespace ahakv {

constexpr int kMaxRows = 256;   // G * r, the stacked observation rows of one KV head
constexpr int kKeyTile = 128;   // keys per scoring tile
constexpr float kLog2e = 1.4426950408889634f;

// Per observation row i: c[i] = lambda_i * log2(e), so that e^{lambda w} = 2^{c w}.
struct RowScale {
  float c[kMaxRows];
};

// The sizes and strides of a call: the part of the plan that the small kernels take by value.
struct Shape {
  int B, Hq, Hkv, G, d, n, r, Br, Bud, Bs, n_keep, dtype, es, pool;
  unsigned flags;
  long long n_total;
  int R;          // G * r
  int n_blk;      // ceil(n / kKeyTile)
  int group_max;  // pool the query heads of a KV head by maximum instead of mean (and G > 1)
  long long qs[3], ks[3], vs[3];  // element strides: batch, head, token
};

// Everything the host derives from ahakv_params once per call.
struct Plan : Shape {
  int n_rb;       // row blocks of 128 stacked rows (tensor-core path)
  int heads_per_rb;  // query heads per row block (tensor-core path)
  bool use_tc;    // tensor-core scoring path applies
  RowScale rows;
  double lambda[kMaxRows];   // lambda_i itself, in double (the float32 path scales its logits in double)
  int last[kMaxRows];        // per observation row: the last cache row it may see (n - r + i unless positions are given)
  int n_eff;                 // last[r - 1] + 1: keys beyond are seen by no row
  // workspace layout, byte offsets
  size_t off_status, off_sync, off_sraw, off_nu, off_partial, off_final, off_score, ws_total;   // ws_total: what a call needs
  size_t ws_wanted;          // ws_total and room for the softmax numerators of the FP32-pipe kernels at off ws_total
};

// api.cu
// `obs_pos` (nullable, host, r ascending logical positions) places the observation rows; by default they are the
// last r positions.
ahakv_status make_plan(const ahakv_params* p, Plan* plan, const int64_t* obs_pos = nullptr);
void count_launch(int n = 1);

// Launchers.  Each returns AHAKV_OK or AHAKV_ERR_CUDA and queues work on `st` only.
// Both also stream V and write nu when the value prior is on (v and nu non-null), and clear the status word.
// `kept` (nullable): room for simt_kept_floats() floats, with which the logits are formed once instead of twice.
size_t simt_kept_floats(const Plan& pl);
ahakv_status launch_score_simt(const Plan& pl, const void* q, const void* k, const void* v, float* s_raw, float* nu, float2* partial,
                               float* kept, int* status, cudaStream_t st);
ahakv_status launch_score_tc(const Plan& pl, const void* q, const void* k, const void* v, float* s_raw, float* nu,
                             float* partial, float* off, int* counters, int* status, void* ones, size_t ones_bytes, cudaStream_t st);
bool score_tc_available();
// See ahakv_test_set_wait: the limit of the tensor-core kernels' bounded waits (0: their own), and whether a fault is planted.
struct TestHooks {
  long long wait_ns;
  int withhold;
};
void set_test_hooks(long long wait_ns, int withhold);
TestHooks test_hooks();
// The generation phase one token at a time (decode.cu): the score update of one new query per head without
// scratch memory, and compaction in place.
bool step_score_fits(const Plan& pl);
ahakv_status launch_step_slots(const Plan& pl, const void* q, const void* k_new, const void* v_new, void* k, void* v,
                               float* score, int32_t* pos, int32_t* free_slot, int new_pos, cudaStream_t st);
ahakv_status launch_step_score(const Plan& pl, const void* q, const void* k, const float* prev, float* score,
                               cudaStream_t st);
ahakv_status launch_compact_inplace(const Plan& pl, void* k, void* v, float* score, const int32_t* kept_idx,
                                    cudaStream_t st);
// Row entropy of the SG-softmax (entropy.cu): out [B, Hq, r]; `scratch` of entropy_scratch_bytes().
size_t entropy_scratch_bytes(const Plan& pl);
ahakv_status launch_entropy(const Plan& pl, const void* q, const void* k, void* scratch, float* out, cudaStream_t st);
// The same on the tensor cores (score_stream.cu; plans with use_tc).
size_t entropy_tc_scratch_bytes(const Plan& pl);
ahakv_status launch_entropy_tc(const Plan& pl, const void* q, const void* k, void* scratch, float* out, cudaStream_t st);
// Accumulation over every causal row on the tensor cores (score_stream.cu; plans with use_tc).  Leaves *n_slots partial sums
// per head in *slots (`sums` if there is one: [B * Hkv][n]); `pool` is scratch, 256-byte aligned: the room a plan with use_tc has
// for raw scores and partials, over 2 n_rb floats for every row of the 128-row tiles of each head, always suffices.
ahakv_status launch_causal_tc(const Plan& pl, int scale_mode, double fixed, long long first_cached, const void* q, const long long qs[3],
                              const void* k, float* pool, size_t pool_bytes, float* sums, const float** slots, int* n_slots,
                              int* status, cudaStream_t st);
// All ones into `bytes` (a multiple of 16) from `to` (16-byte aligned) on (clear.cu).
ahakv_status launch_clear(void* to, size_t bytes, cudaStream_t st);
ahakv_status launch_vnorm(const Plan& pl, const void* v, float* nu, cudaStream_t st);
// `slots` partial scores per head (row blocks, or query heads when pooling by maximum) are combined here.
ahakv_status launch_refine(const Plan& pl, const float* s_raw, const float* nu, const float* score_prev,
                           float* score, int slots, cudaStream_t st);
ahakv_status launch_select(const Plan& pl, const float* score, int32_t* kept_idx, cudaStream_t st);
// Both steps.  Writes the kept tokens' scores to score_out (nullable) itself when a head fits in a cluster; otherwise leaves
// the refined scores in `score`.  *score_left says which: null, or `score` for the caller to gather from.  Gathers the kept
// rows too where they are few (*gathered).
ahakv_status launch_refine_select(const Plan& pl, const float* s_raw, const float* nu, const float* score_prev,
                                  float* score, float** score_left, float* score_out, int32_t* kept_idx, int slots,
                                  const int32_t* budgets, const void* k, const void* v, void* k_out, void* v_out, bool* gathered,
                                  cudaStream_t st);
ahakv_status launch_compact(const Plan& pl, const void* k, const void* v, const float* score,
                            const int32_t* kept_idx, void* k_out, void* v_out, float* score_out,
                            cudaStream_t st);

// profile.cu: event marks around the stages of a call (no-ops unless profiling is enabled).
int profile_begin_call(cudaStream_t st);             // returns a slot, or -1
void profile_mark(int slot, int boundary, cudaStream_t st);   // boundary b closes stage b-1, opens stage b

// An error is reported once: cudaLaunchKernelEx leaves it behind as the thread's last error too, where the next
// cudaGetLastError() of a call that went well would find it.
inline ahakv_status cuda_ok(cudaError_t e) {
  if (e == cudaSuccess) return AHAKV_OK;
  cudaGetLastError();
  return AHAKV_ERR_CUDA;
}

// Launches `kernel` so that it may start its prologue while the kernel before it in the stream still runs (programmatic
// dependent launch; the kernel calls griddep_wait() before it touches anything), as clusters of `cluster` CTAs.
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, int cluster, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// ---- device helpers ---------------------------------------------------------
template <typename T> __device__ __forceinline__ float to_f32(T x);
template <> __device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f32<__half>(__half x) { return __half2float(x); }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

// 16 bytes of T widened to float.
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  static constexpr int N = 4;
  static __device__ __forceinline__ void widen(const uint4& u, float* f) {
    f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y);
    f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
  }
};
template <> struct Vec16<__half> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void widen(const uint4& u, float* f) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&w[t]));
      f[2 * t] = p.x; f[2 * t + 1] = p.y;
    }
  }
};
template <> struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void widen(const uint4& u, float* f) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {  // a bfloat16 is the high half of a float
      f[2 * t] = __uint_as_float(w[t] << 16);
      f[2 * t + 1] = __uint_as_float(w[t] & 0xffff0000u);
    }
  }
};

// Programmatic dependent launch: wait for the kernel before this one in the stream (no effect without the launch
// attribute), and let the one after it start its prologue.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float fast_exp2(float x) {  // 2 ulp over the whole range; 2^-inf = 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace ahakv

// Argument structures shared by the two arithmetic paths of the update block (fp32 on the plain ALUs, bf16 on the
// tensor cores).
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "launch.cuh"
#include "layout.h"

namespace mava {

struct UpdNet {
  const float *W1, *b1, *W2, *b2;  // caller layout [out][in]
  const float *W1t, *W2t;          // [in][out] copies
  const float *Wa, *ba, *Wv, *bv;  // heads (nullptr when the net has none of that kind)
  int Din, H;
  size_t oW1, ob1, oW2, ob2, oWa, oba, oWv, obv;  // offsets of the gradients in the flat array
};
struct UpdRows {
  const float *x;                  // [n][Din]
  const int32_t *actions;          // [n]          (actor)
  const float *logp_old, *adv;     // [n]          (actor)
  const float *value_old, *ret;    // [n * vstride] (value), element r at r * vstride
  int vstride;
  long long n;
  // a minibatch of environments: row q of the batch is (step, env_ids[i], slot) with q = (step * n_ids + i) * per_env + slot;
  // nullptr = every environment in order (row q is row q of the arrays)
  const int32_t *env_ids;
  int n_ids, E, per_env;
};

// Row of the trajectory arrays behind row q of the batch; -1 when the environment index is out of range.  U holds the batch's
// row numbers: 32 bits for what is cut from a trajectory without repetition (a row is 340 bytes of observation alone, so
// fewer than 2^31 fit a GPU); a minibatch that repeats environments may be longer than its trajectory and need 64.  The
// tensor-core kernels are compiled for either (choosing at run time cost H <= 128 0.5 to 0.9 us a minibatch, H = 256 2 %).
template <class U>
__device__ __forceinline__ long long real_row(const UpdRows &rows, long long row) {
  if (!rows.env_ids) return row;
  const U q = static_cast<U>(row), per_env = static_cast<U>(rows.per_env), per_step = static_cast<U>(rows.n_ids) * per_env;
  const U t = q / per_step, rem = q - t * per_step, i = rem / per_env, slot = rem - i * per_env;
  const int e = rows.env_ids[i];
  if (e < 0 || e >= rows.E) return -1;
  return static_cast<long long>((t * static_cast<uint32_t>(rows.E) + static_cast<uint32_t>(e)) * per_env + slot);
}
__host__ __device__ __forceinline__ bool rows_need_64_bits(const UpdRows &rows, long long n) { return rows.env_ids && (n >> 32) != 0; }
__device__ __forceinline__ long long real_row_any(const UpdRows &rows, long long row) {
  return rows_need_64_bits(rows, rows.n) ? real_row<uint64_t>(rows, row) : real_row<uint32_t>(rows, row);
}

// A predicated load (zero otherwise), in program order with its like: the compiler neither branches around it nor puts a use
// of one between two of them, so a batch costs one round trip (with plain conditional loads a batch of 48 took 22 k cycles).
__device__ __forceinline__ float ldg_if(const float *p, bool pred) {
  float v;
  asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\nmov.f32 %0, 0f00000000;\n@q ld.global.L1::no_allocate.f32 %0, [%1];\n}"
               : "=f"(v)
               : "l"(p), "r"(static_cast<uint32_t>(pred)));
  return v;
}
// The same for lines that another load of the warp reads as well.
__device__ __forceinline__ float ldg_if_cached(const float *p, bool pred) {
  float v;
  asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\nmov.f32 %0, 0f00000000;\n@q ld.global.f32 %0, [%1];\n}" : "=f"(v) : "l"(p), "r"(static_cast<uint32_t>(pred)));
  return v;
}
// real_row in two parts, so that the look-up of the environment can be on its way while other work goes on: the row is
// at + e * per_env for an e that is one of the environments.
struct RowLookup { int at, e; };
template <class U>
__device__ __forceinline__ RowLookup row_lookup(const UpdRows &rows, long long row, bool valid) {
  if (!rows.env_ids) return RowLookup{static_cast<int>(row), valid ? 0 : -1};
  const U q = static_cast<U>(row), per_env = static_cast<U>(rows.per_env), per_step = static_cast<U>(rows.n_ids) * per_env;
  const U t = q / per_step, rem = q - t * per_step, i = rem / per_env, slot = rem - i * per_env;
  const int e = __float_as_int(ldg_if_cached(reinterpret_cast<const float *>(rows.env_ids) + (valid ? i : 0), valid));
  return RowLookup{static_cast<int>(static_cast<uint32_t>(t) * static_cast<uint32_t>(rows.E) * static_cast<uint32_t>(rows.per_env) + static_cast<uint32_t>(slot)), valid ? e : -1};
}
__device__ __forceinline__ int row_found(const UpdRows &rows, RowLookup l) { return l.e >= 0 && l.e < rows.E ? l.at + l.e * rows.per_env : -1; }
// ---- two accumulator columns at a time: the epilogues of the tensor-core kernels --------------------------------------------
// All-ones in each half of the result whose bf16 in `v` is positive.
__device__ __forceinline__ uint32_t positive_mask(uint32_t v) {
  const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162 *>(&v);
  return __hgt2_mask(x, __floats2bfloat162_rn(0.0f, 0.0f));
}
// All-ones in each half of the result whose sign bit (15, 31) is set in `v`.
__device__ __forceinline__ uint32_t sign_mask(uint32_t v) {
  uint32_t m;
  asm("prmt.b32 %0, %1, %1, 0xBB99;" : "=r"(m) : "r"(v));
  return m;
}
__device__ __forceinline__ void add2(uint32_t &lo, uint32_t &hi, float blo, float bhi) {
  asm("{\n.reg .b64 a, b;\nmov.b64 a, {%0, %1};\nmov.b64 b, {%2, %3};\nadd.rn.f32x2 a, a, b;\nmov.b64 {%0, %1}, a;\n}"
      : "+r"(lo), "+r"(hi)
      : "r"(__float_as_uint(blo)), "r"(__float_as_uint(bhi)));
}
__device__ __forceinline__ float4 lds_float4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// ---- mean and population std of a vector, by the first kMomentBlocks blocks (256 threads each) of a kernel: block
// partial sums of x and x^2 in double; the block that finishes last adds them.  Fixed orders throughout: the same bytes on
// every call, and from every kernel that does it.
constexpr int kMomentBlocks = 256;
struct Moments {
  const float *x;      // nullptr: nothing to do
  long long n;
  UpdRows map;         // which elements (env_ids == nullptr: all n)
  double *part;        // [kMomentBlocks][2]
  double *out;         // mean, std
  unsigned *finished;  // zero before and after
};
// Sums of a and b over the block's first 256 threads, in thread 0.
__device__ __forceinline__ void block_sum2(double &a, double &b) {
  __shared__ double sa[8], sb[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { a += __shfl_xor_sync(0xFFFFFFFFu, a, o); b += __shfl_xor_sync(0xFFFFFFFFu, b, o); }
  __syncthreads();  // (the arrays may still be read from the last time)
  if ((threadIdx.x & 31) == 0 && threadIdx.x < 256) { sa[threadIdx.x >> 5] = a; sb[threadIdx.x >> 5] = b; }
  __syncthreads();
  if (threadIdx.x != 0) return;
  a = b = 0.0;
#pragma unroll
  for (int w = 0; w < 8; ++w) { a += sa[w]; b += sb[w]; }
}
__device__ __forceinline__ void moments_finish(const Moments &m, double a, double b) {
  static_assert(kMomentBlocks == 256, "one partial sum per thread of the last block");
  __shared__ bool last;
  const int t = threadIdx.x;
  block_sum2(a, b);
  if (t == 0) {
    m.part[2 * blockIdx.x] = a; m.part[2 * blockIdx.x + 1] = b;
    __threadfence();
    last = atomicInc(m.finished, kMomentBlocks - 1) == kMomentBlocks - 1;  // (wraps to zero)
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  a = t < 256 ? __ldcg(m.part + 2 * t) : 0.0; b = t < 256 ? __ldcg(m.part + 2 * t + 1) : 0.0;
  block_sum2(a, b);
  if (t != 0) return;
  const double mean = a / static_cast<double>(m.n), var = fmax(b / static_cast<double>(m.n) - mean * mean, 0.0);
  m.out[0] = mean; m.out[1] = sqrt(var);
}
template <class U>
__device__ __forceinline__ void moments_block(const Moments &m) {
  constexpr int kBatch = 8;  // loads in flight per thread (one at a time: 44 us for 16.8 million elements)
  constexpr long long kStep = 256LL * kMomentBlocks;
  double a = 0.0, b = 0.0;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < m.n; i += kBatch * kStep) {
    float v[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const long long q = i + k * kStep, row = real_row<U>(m.map, q < m.n ? q : i);  // (loads without a branch around them)
      v[k] = __ldcg(m.x + (row >= 0 ? row : 0));
      if (q >= m.n || row < 0) v[k] = 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) { a += v[k]; b += static_cast<double>(v[k]) * v[k]; }
  }
  moments_finish(m, a, b);
}
// What a gradient call starts with: the advantages' moments and, by the other blocks, the weight image (prep(i, n): thread i
// of n).
template <class U, class Prep>
__global__ void __launch_bounds__(256) prologue_kernel(Moments m, Prep prep) {
  dependents_may_start();
  const int first = m.x ? kMomentBlocks : 0, b = static_cast<int>(blockIdx.x);
  wait_for_predecessor();
  if (b < first) {
    moments_block<U>(m);
    return;
  }
  prep((b - first) * 256 + static_cast<int>(threadIdx.x), (static_cast<int>(gridDim.x) - first) * 256);
}
template <class Prep>
cudaError_t launch_prologue(const Moments &m, const Prep &prep, int prep_blocks, cudaStream_t stream) {
  return launch_dependent(rows_need_64_bits(m.map, m.n) ? prologue_kernel<uint64_t, Prep> : prologue_kernel<uint32_t, Prep>, (m.x ? kMomentBlocks : 0) + prep_blocks, 256, 0, stream, m, prep);
}

struct UpdHyper { float clip_eps, ent_coef, vf_coef; };

// Tensor-core path (update_tc.cu): shared-torso nets with H <= 128 and D <= 80.
bool ppo_tc_supported(const mava_config_t &cfg, int D);
size_t ppo_tc_image_bytes();
size_t ppo_tc_slice_floats();
struct TermSums;
struct AdamArgs;
// Enqueues the prologue (moments of the advantages, weight image; not if launch_step_tc has left both), the loss/gradient kernel and
// the reduction of its slices into `grad`, the loss terms and the gradient's sums of squares; `partial` holds `slices` slices of
// ppo_tc_slice_floats() floats (one per CTA), `term_partial` 4 x 3 doubles per slice.
cudaError_t launch_ppo_net_tc(mava_rollout *h, const float *params_dev, const ParamLayout &L, const UpdRows &rows, const UpdHyper &hp,
                              const Moments &adv, bool prepared, void *image, float *partial, double *term_partial, int slices, float *grad,
                              const TermSums &terms, double *squares);
// The sums of squares that launch_ppo_net_tc leaves, of a gradient that comes from elsewhere: the same order of additions.
cudaError_t launch_grad_squares_tc(mava_rollout *h, const ParamLayout &L, const float *grad, double *squares);
// An optimiser step with what the next gradient starts with: its weight image and its advantages' moments (`next`).
cudaError_t launch_step_tc(mava_rollout *h, const AdamArgs &adam, const ParamLayout &L, const Moments &next, void *image);

// Where the loss-term sums of a call lie, [n][3] doubles (surrogate, entropy, value) per list: the actor's list gives the
// first two, the value net's the third (one net with both heads: the same list).
struct TermSums {
  const double *actor, *value;
  int n_actor_part, n_value_part;
  long long n_actor, n_value;  // rows behind the means
  UpdHyper hp;
  float *out;                  // [4] total, actor, entropy, value; nullptr: not wanted
};
// Called by one whole block, done by its first kTermThreads threads at most: each adds every nt-th entry, eight loads in flight, then a tree
// (a fixed order for a block size; one thread adding 256 shares took longer than the rest of the reduction).
constexpr int kTermThreads = 512;
__device__ __forceinline__ void loss_terms(const TermSums &t) {
  constexpr int kBatch = 8;
  const int nt = min(static_cast<int>(blockDim.x), kTermThreads);
  __shared__ double st[3][16];
  if (!t.out) return;
  const int i = static_cast<int>(threadIdx.x);
  double a = 0.0, e = 0.0, v = 0.0;
  if (i < nt) {
    for (int k0 = i; k0 < t.n_actor_part; k0 += kBatch * nt) {
      double x[kBatch], y[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) { const int k = min(k0 + q * nt, t.n_actor_part - 1); x[q] = t.actor[3 * k]; y[q] = t.actor[3 * k + 1]; }
#pragma unroll
      for (int q = 0; q < kBatch; ++q)
        if (k0 + q * nt < t.n_actor_part) { a += x[q]; e += y[q]; }
    }
    for (int k0 = i; k0 < t.n_value_part; k0 += kBatch * nt) {
      double x[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) x[q] = t.value[3 * min(k0 + q * nt, t.n_value_part - 1) + 2];
#pragma unroll
      for (int q = 0; q < kBatch; ++q)
        if (k0 + q * nt < t.n_value_part) v += x[q];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xFFFFFFFFu, a, o); e += __shfl_xor_sync(0xFFFFFFFFu, e, o); v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    }
    if ((i & 31) == 0) { st[0][i >> 5] = a; st[1][i >> 5] = e; st[2][i >> 5] = v; }
  }
  __syncthreads();
  if (i != 0) return;
  a = e = v = 0.0;
  for (int w = 0; w < nt / 32; ++w) { a += st[0][w]; e += st[1][w]; v += st[2][w]; }
  const double actor = -a / static_cast<double>(t.n_actor), ent = e / static_cast<double>(t.n_actor), val = v / static_cast<double>(t.n_value);
  t.out[0] = static_cast<float>(actor - t.hp.ent_coef * ent + t.hp.vf_coef * val);
  t.out[1] = static_cast<float>(actor);
  t.out[2] = static_cast<float>(ent);
  t.out[3] = static_cast<float>(val);
}

// ---- optimiser step.  The gradient's 2-norm comes as kMomentBlocks sums of squares from the kernel in front; every block adds them
// for itself (when the last block of that kernel did, the step started 4 us later).
struct AdamArgs {
  float *params;
  const float *grad;
  float *m, *v;
  const double *squares;  // [kMomentBlocks]
  float max_norm, lr, beta1, beta2, eps, corr1, corr2;
};
// The factor that takes the gradient to max_norm at most (by a whole block of 256 threads, after its wait).
__device__ __forceinline__ float adam_scale(const AdamArgs &a) {
  __shared__ float scale;
  double none = 0.0, b = __ldcg(a.squares + threadIdx.x);
  block_sum2(none, b);
  if (threadIdx.x == 0) scale = a.max_norm / fmaxf(static_cast<float>(sqrt(b)), a.max_norm);
  __syncthreads();
  return scale;
}
// A parameter and its moments: the parts of a step that do not need the gradient can come before the wait for it.
struct AdamState { float p, m, v; };
__device__ __forceinline__ AdamState adam_load(const AdamArgs &a, size_t i) { return AdamState{__ldcg(a.params + i), __ldcg(a.m + i), __ldcg(a.v + i)}; }
__device__ __forceinline__ float adam_element(const AdamArgs &a, const AdamState &s, float grad, float scale, size_t i) {
  const float g = grad * scale;
  const float mi = a.beta1 * s.m + (1.0f - a.beta1) * g, vi = a.beta2 * s.v + (1.0f - a.beta2) * g * g;
  a.m[i] = mi; a.v[i] = vi;
  const float p = s.p - a.lr * (mi / a.corr1) / (sqrtf(vi / a.corr2) + a.eps);
  a.params[i] = p;
  return p;
}

__device__ __forceinline__ double squares_of_group(const double *warps) { return ((warps[0] + warps[1]) + warps[2]) + warps[3]; }

// grad[map(j)] = sum of element j over the CTAs' slices of `len` floats, in a fixed order, and the sum of squares of each group of
// kGradLanes elements (the 2-norm is what an optimiser step needs next); a block of its own turns the term sums into the loss terms.
// Four threads per element take a quarter of the slices each, 20 loads in flight; two groups per block, so that all blocks run at
// once: behind a kernel that fills the SMs only one block per SM was resident, and of 257 blocks of one group the last 109 started
// when the first were done (six reductions of 28 k elements over 148 slices: 346 -> 338 us with the loads of the step before its wait).
constexpr int kGradLanes = 128, kGroups = 2;  // elements per group; groups per block and round
constexpr int kReduceBlocks = kMomentBlocks / kGroups + 1, kReduceThreads = 4 * kGradLanes * kGroups;
struct IdentityMap {
  __device__ __forceinline__ long long operator()(int j) const { return j; }
};
template <class Map>
__global__ void __launch_bounds__(kReduceThreads) reduce_slices_kernel(const float *partial, int len, int n_slices, float *grad, TermSums terms,
                                                            double *squares, Map map) {
  dependents_may_start();
  wait_for_predecessor();
  if (blockIdx.x == kMomentBlocks / kGroups) {
    loss_terms(terms);
    return;
  }
  constexpr int kBatch = 20;
  __shared__ float quarter[kGroups][4][kGradLanes];
  __shared__ double warp_squares[kGroups][kGradLanes / 32];
  const int col = threadIdx.x % kGradLanes, q = threadIdx.x / kGradLanes % 4, g = threadIdx.x / (4 * kGradLanes);
  const int group = static_cast<int>(blockIdx.x) * kGroups + g;
  const int c_lo = n_slices * q / 4, c_hi = n_slices * (q + 1) / 4;
  double b = 0.0;
  for (int r0 = 0; r0 < len; r0 += kMomentBlocks * kGradLanes) {
    const int j = r0 + group * kGradLanes + col;
    const long long out = j < len ? map(j) : -1;
    const float *src = partial + (out >= 0 ? j : 0);
    float s = 0.0f;
    for (int c0 = c_lo; c0 < c_hi; c0 += kBatch) {
      float v[kBatch];
#pragma unroll
      for (int k = 0; k < kBatch; ++k) v[k] = __ldcg(src + static_cast<size_t>(min(c0 + k, c_hi - 1)) * len);  // (no branch around a load)
#pragma unroll
      for (int k = 0; k < kBatch; ++k) s = c0 + k < c_hi ? s + v[k] : s;
    }
    quarter[g][q][col] = s;
    __syncthreads();
    if (q == 0 && out >= 0) {
      s = (s + quarter[g][1][col]) + (quarter[g][2][col] + quarter[g][3][col]);
      grad[out] = s;
      b += static_cast<double>(s) * s;
    }
    __syncthreads();
  }
  if (q == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
    if ((col & 31) == 0) warp_squares[g][col >> 5] = b;
  }
  __syncthreads();
  if (q == 0 && col == 0) squares[group] = squares_of_group(warp_squares[g]);
}
// The same sums of squares of a gradient that comes from elsewhere, with the additions of reduce_slices_kernel: a group per block.
template <class Map>
__global__ void __launch_bounds__(kGradLanes) grad_squares_kernel(const float *grad, double *squares, int len, Map map) {
  dependents_may_start();
  wait_for_predecessor();
  __shared__ double warp_squares[kGradLanes / 32];
  const int col = threadIdx.x;
  double b = 0.0;
  for (int j = static_cast<int>(blockIdx.x) * kGradLanes + col; j < len; j += kMomentBlocks * kGradLanes) {
    const long long p = map(j);
    const float v = p >= 0 ? __ldcg(grad + p) : 0.0f;
    if (p >= 0) b += static_cast<double>(v) * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
  if ((col & 31) == 0) warp_squares[col >> 5] = b;
  __syncthreads();
  if (col == 0) squares[blockIdx.x] = squares_of_group(warp_squares);
}

// Tensor-core path for H = 256 (update_tc256.cu): a net with hidden width 256 whose first layer takes `slabs` observation
// slabs of width 64 < D <= 95 side by side (1: the actor / shared-torso net; n_agents: the centralised critic).  Offsets are
// those of the net's layers in the flat parameter array.  Writes the net's gradient and, after the net with the value head,
// the loss terms.
struct Tc256Net {
  size_t W1, b1, W2, b2, Wa, ba, Wv, bv;
  int slabs;
  bool has_actor, has_value;
};
struct Tc256Need { size_t scratch, ring; };  // bytes for a batch of n_rows rows
bool ppo_tc256_supported(const mava_config_t &cfg, int D);
Tc256Need ppo_tc256_need(long long n_rows, int sms, int slabs);
cudaError_t launch_ppo_net_tc256(mava_rollout *h, const float *params_dev, const Tc256Net &net, const UpdRows &rows, const UpdHyper &hp,
                                 const Moments &adv, const double *adv_stats, void *scratch, void *ring, int sms, float *grad, TermSums &terms);

}  // namespace mava

// Update block, fp32 path on the plain ALUs, and the optimiser step of all paths: the multi-agent PPO loss of one minibatch (all rows
// of the last rollout), its gradient with respect to every parameter, and the Adam step.
//   loss:  rho = exp(logp_new(a) - logp_old);  Ahat = (A - mean A) / (std A + 1e-8);
//          L = -mean min(rho Ahat, clip(rho, 1 +- eps) Ahat) - c_ent mean H
//              + c_val 0.5 mean max((V - R)^2, (Vold + clip(V - Vold, +-eps) - R)^2)
// A CTA of H threads (thread j = hidden unit j) walks over tiles of 32 rows: forward through the two hidden
// layers with the activations of the tile in shared memory, heads and per-row loss derivatives by one warp per
// row, backward through the layers, and the tile's contribution to every weight gradient added into the CTA's
// own slice of a partial-gradient array (reductions without a return value: an address is only ever added to by
// one thread, in program order; a last kernel adds the slices in a fixed order, so the result does not depend
// on scheduling).  Sums that decide a mean are kept in double.
// This is the validation path of the update block, as rollout_simt.cu is the rollout's; update_tc.cu and update_tc256.cu are
// the tensor-core paths.
#include "common.cuh"
#include "layout.h"
#include "update_common.cuh"

namespace mava {
namespace {

constexpr int kUpdRows = 32;       // rows per tile
constexpr int kUpdTS = kUpdRows;   // row stride of the transposed d z tiles [unit][row] (read by 16-byte broadcasts; the few
                                   // stores that fill them collide on banks, which costs less than the room padding takes)

__global__ void transpose_kernel(const float *__restrict__ W, float *__restrict__ Wt, int out, int in) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < out * in; i += gridDim.x * blockDim.x) {
    const int o = i / in, k = i - o * in;
    Wt[static_cast<size_t>(k) * out + o] = W[i];
  }
}

// HT = hidden width = threads per CTA; the register budget is set for the CTAs per SM that the shared memory allows.
template <int HT>
__global__ void __launch_bounds__(HT, HT == 256 ? 1 : (HT == 128 ? 3 : 4))
ppo_net_kernel(UpdNet net, UpdRows rows, UpdHyper hp, const double *__restrict__ adv_stats,
                               float *__restrict__ partial, size_t n_params, double *__restrict__ term_partial, int *status) {
  extern __shared__ __align__(16) float smf[];
  constexpr int H = HT;
  const int Din = net.Din, j = threadIdx.x, lane = j & 31, warp = j >> 5, n_warps = H >> 5;
  const int Dp = (Din + 3) & ~3;  // row stride of the input tile; the pad columns hold zeros
  // every inner product below reads four operands per shared-memory access (16-byte broadcast loads)
  // d z1 takes the place of h2, which is dead by then: three CTAs fit an SM at H = 128
  float *xs = smf, *h1s = xs + kUpdRows * Dp, *h2s = h1s + kUpdRows * H, *dz2t = h2s + kUpdRows * H, *dz1t = h2s,
        *dl = dz2t + H * kUpdTS;  // dl [32][8]: d logits (6), d value
  long long *rmap = reinterpret_cast<long long *>(dl + kUpdRows * 8);  // trajectory row of every row of the tile
  auto ld4 = [](const float *p) { return *reinterpret_cast<const float4 *>(p); };
  const int HH = H >> 1, up = j % HH, r0 = (j / HH) * (kUpdRows / 2);  // the two-unit mapping of the dense loops
  float *part = partial + static_cast<size_t>(blockIdx.x) * n_params;
  const bool has_actor = net.Wa != nullptr, has_value = net.Wv != nullptr;
  const float mean = has_actor ? static_cast<float>(adv_stats[0]) : 0.0f;
  const float inv_std = has_actor ? 1.0f / (static_cast<float>(adv_stats[1]) + 1e-8f) : 0.0f;
  const float inv_n = 1.0f / static_cast<float>(rows.n);
  float gWa[kActions], gWv = 0.0f, gb1 = 0.0f, gb2 = 0.0f, gbh = 0.0f;
#pragma unroll
  for (int k = 0; k < kActions; ++k) gWa[k] = 0.0f;
  double t_actor = 0.0, t_ent = 0.0, t_value = 0.0;  // lane 0 of every warp
  const long long n_tiles = (rows.n + kUpdRows - 1) / kUpdRows;
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const long long row0 = tile * kUpdRows;
    const int n_valid = static_cast<int>(min(static_cast<long long>(kUpdRows), rows.n - row0));
    if (j < kUpdRows) {
      const long long row = j < n_valid ? real_row_any(rows, row0 + j) : -1;
      rmap[j] = row;
      if (j < n_valid && row < 0) atomicExch(status, kStatusBadIndex);
    }
    __syncthreads();
    for (int r = warp; r < kUpdRows; r += n_warps) {  // a warp per row: consecutive lanes, consecutive floats
      const long long row = rmap[r];
      for (int k = lane; k < Dp; k += 32) xs[r * Dp + k] = (row >= 0 && k < Din) ? rows.x[row * Din + k] : 0.0f;
    }
    __syncthreads();
    // hidden layer 1 and 2.  Here a thread computes two units (up, up + H/2) of half the tile's rows, so that one
    // 16-byte broadcast read of the activations feeds eight multiply-adds.
    auto dense2 = [&](const float *src, int stride, int K, int k_valid, const float *Wt, const float *bias, float *dst) {
      float a0[kUpdRows / 2], a1[kUpdRows / 2];
#pragma unroll
      for (int r = 0; r < kUpdRows / 2; ++r) a0[r] = a1[r] = 0.0f;
      for (int k = 0; k < K; k += 4) {
        float w0[4], w1[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const bool ok = k + q < k_valid;
          w0[q] = ok ? Wt[static_cast<size_t>(k + q) * H + up] : 0.0f;
          w1[q] = ok ? Wt[static_cast<size_t>(k + q) * H + up + HH] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < kUpdRows / 2; ++r) {
          const float4 x = ld4(src + (r0 + r) * stride + k);
          a0[r] = fmaf(x.x, w0[0], fmaf(x.y, w0[1], fmaf(x.z, w0[2], fmaf(x.w, w0[3], a0[r]))));
          a1[r] = fmaf(x.x, w1[0], fmaf(x.y, w1[1], fmaf(x.z, w1[2], fmaf(x.w, w1[3], a1[r]))));
        }
      }
      const float b0 = bias[up], b1v = bias[up + HH];
#pragma unroll
      for (int r = 0; r < kUpdRows / 2; ++r) {
        dst[(r0 + r) * H + up] = fmaxf(a0[r] + b0, 0.0f);
        dst[(r0 + r) * H + up + HH] = fmaxf(a1[r] + b1v, 0.0f);
      }
    };
    dense2(xs, Dp, Dp, Din, net.W1t, net.b1, h1s);
    __syncthreads();
    dense2(h1s, H, H, H, net.W2t, net.b2, h2s);
    __syncthreads();
    // heads and the per-row derivatives of the loss: one warp per row
    for (int r = warp; r < kUpdRows; r += n_warps) {
      float s[kActions + 1];
#pragma unroll
      for (int k = 0; k <= kActions; ++k) s[k] = 0.0f;
      for (int i = lane; i < H; i += 32) {
        const float hv = h2s[r * H + i];
        if (has_actor) {
#pragma unroll
          for (int k = 0; k < kActions; ++k) s[k] = fmaf(hv, net.Wa[k * H + i], s[k]);
        }
        if (has_value) s[kActions] = fmaf(hv, net.Wv[i], s[kActions]);
      }
#pragma unroll
      for (int k = 0; k <= kActions; ++k)
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], o);
      if (lane == 0) {
        float d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) d[k] = 0.0f;
        if (rmap[r] >= 0) {
          const long long row = rmap[r];
          if (has_actor) {
            float l[kActions], m = -INFINITY, sum = 0.0f;
#pragma unroll
            for (int k = 0; k < kActions; ++k) { l[k] = s[k] + net.ba[k]; m = fmaxf(m, l[k]); }
#pragma unroll
            for (int k = 0; k < kActions; ++k) sum += expf(l[k] - m);
            const float lse = m + logf(sum);
            const int a = rows.actions[row];
            float ent = 0.0f, p[kActions], lp[kActions], lpa = 0.0f;
#pragma unroll
            for (int k = 0; k < kActions; ++k) {
              lp[k] = l[k] - lse; p[k] = expf(lp[k]); ent -= p[k] * lp[k];
              if (k == a) lpa = lp[k];
            }
            const float rho = expf(lpa - rows.logp_old[row]);
            const float ahat = (rows.adv[row] - mean) * inv_std;
            const float clipped = fminf(fmaxf(rho, 1.0f - hp.clip_eps), 1.0f + hp.clip_eps);
            const float s1 = rho * ahat, s2 = clipped * ahat;
            const bool inside = rho >= 1.0f - hp.clip_eps && rho <= 1.0f + hp.clip_eps;
            const float d_logp = (inside || s1 < s2) ? -s1 * inv_n : 0.0f;  // the clipped branch is constant in rho
#pragma unroll
            for (int k = 0; k < kActions; ++k)
              d[k] = d_logp * ((k == a ? 1.0f : 0.0f) - p[k]) + hp.ent_coef * inv_n * p[k] * (lp[k] + ent);
            t_actor += fminf(s1, s2);
            t_ent += ent;
          }
          if (has_value) {
            const float v = s[kActions] + net.bv[0], vo = rows.value_old[row * rows.vstride], rt = rows.ret[row * rows.vstride];
            const float u = v - rt, uc = vo + fminf(fmaxf(v - vo, -hp.clip_eps), hp.clip_eps) - rt;
            const bool in_range = fabsf(v - vo) <= hp.clip_eps;
            d[kActions] = (in_range || u * u > uc * uc) ? hp.vf_coef * u * inv_n : 0.0f;
            t_value += 0.5 * fmaxf(u * u, uc * uc);
          }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) dl[r * 8 + k] = d[k];
      }
    }
    __syncthreads();
    // back through the heads: d h2, head gradients (kept in registers over all tiles), d z2
    float dzr[kUpdRows];
#pragma unroll
    for (int r = 0; r < kUpdRows; ++r) {
      const float hv = h2s[r * H + j];
      float dh = 0.0f;
      if (has_actor) {
#pragma unroll
        for (int k = 0; k < kActions; ++k) {
          const float dk = dl[r * 8 + k];
          dh = fmaf(dk, net.Wa[k * H + j], dh);
          gWa[k] = fmaf(dk, hv, gWa[k]);
        }
      }
      if (has_value) {
        const float dv = dl[r * 8 + kActions];
        dh = fmaf(dv, net.Wv[j], dh);
        gWv = fmaf(dv, hv, gWv);
      }
      const float dz = hv > 0.0f ? dh : 0.0f;
      dzr[r] = dz;
      gb2 += dz;
      if (j < 8) gbh += dl[r * 8 + j];  // threads 0..6: the heads' biases
    }
#pragma unroll
    for (int r = 0; r < kUpdRows; r += 4)
      *reinterpret_cast<float4 *>(dz2t + j * kUpdTS + r) = make_float4(dzr[r], dzr[r + 1], dzr[r + 2], dzr[r + 3]);
    __syncthreads();
    // d h1 = d z2 . W2 (rows of W2 are contiguous in the unit index), d z1: again two units and half the rows per thread
    {
      float a0[kUpdRows / 2], a1[kUpdRows / 2];
#pragma unroll
      for (int r = 0; r < kUpdRows / 2; ++r) a0[r] = a1[r] = 0.0f;
      for (int i = 0; i < H; i += 4) {
        float w0[4], w1[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          w0[q] = net.W2[static_cast<size_t>(i + q) * H + up];
          w1[q] = net.W2[static_cast<size_t>(i + q) * H + up + HH];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
          for (int r = 0; r < kUpdRows / 2; r += 4) {
            const float4 d = ld4(dz2t + (i + q) * kUpdTS + r0 + r);
            a0[r] = fmaf(d.x, w0[q], a0[r]); a0[r + 1] = fmaf(d.y, w0[q], a0[r + 1]);
            a0[r + 2] = fmaf(d.z, w0[q], a0[r + 2]); a0[r + 3] = fmaf(d.w, w0[q], a0[r + 3]);
            a1[r] = fmaf(d.x, w1[q], a1[r]); a1[r + 1] = fmaf(d.y, w1[q], a1[r + 1]);
            a1[r + 2] = fmaf(d.z, w1[q], a1[r + 2]); a1[r + 3] = fmaf(d.w, w1[q], a1[r + 3]);
          }
        }
      }
      // d z1 takes h2's place: h2 was last read before the barrier that precedes this loop
#pragma unroll
      for (int r = 0; r < kUpdRows / 2; r += 4) {
        float4 z0, z1;
        z0.x = h1s[(r0 + r) * H + up] > 0.0f ? a0[r] : 0.0f; z0.y = h1s[(r0 + r + 1) * H + up] > 0.0f ? a0[r + 1] : 0.0f;
        z0.z = h1s[(r0 + r + 2) * H + up] > 0.0f ? a0[r + 2] : 0.0f; z0.w = h1s[(r0 + r + 3) * H + up] > 0.0f ? a0[r + 3] : 0.0f;
        z1.x = h1s[(r0 + r) * H + up + HH] > 0.0f ? a1[r] : 0.0f; z1.y = h1s[(r0 + r + 1) * H + up + HH] > 0.0f ? a1[r + 1] : 0.0f;
        z1.z = h1s[(r0 + r + 2) * H + up + HH] > 0.0f ? a1[r + 2] : 0.0f; z1.w = h1s[(r0 + r + 3) * H + up + HH] > 0.0f ? a1[r + 3] : 0.0f;
        *reinterpret_cast<float4 *>(dz1t + up * kUpdTS + r0 + r) = z0;
        *reinterpret_cast<float4 *>(dz1t + (up + HH) * kUpdTS + r0 + r) = z1;
      }
    }
    __syncthreads();
    // bias gradient of layer 1: thread j sums d z1 of unit j over the tile's rows
#pragma unroll
    for (int r = 0; r < kUpdRows; r += 4) {
      const float4 d = ld4(dz1t + j * kUpdTS + r);
      gb1 += (d.x + d.y) + (d.z + d.w);
    }
    // Weight gradients, G[i][c] += sum_r dz[r][i] v[r][c]: a thread keeps two columns c of v (all 32 rows) in registers
    // and walks over half of the units i, so that every address is added to by one thread only and a broadcast read of
    // d z feeds eight multiply-adds.
    auto weight_grad = [&](const float *dzt, const float *v, int v_stride, int n_cols, size_t g_off) {
      const int i0 = (j / HH) * HH;
      for (int cb = 0; cb < n_cols; cb += H) {
        const int c0 = cb + up, c1 = cb + up + HH;
        if (c0 >= n_cols) break;
        const bool two = c1 < n_cols;
        float v0[kUpdRows], v1[kUpdRows];
#pragma unroll
        for (int r = 0; r < kUpdRows; ++r) {
          v0[r] = v[r * v_stride + c0];
          v1[r] = two ? v[r * v_stride + c1] : 0.0f;
        }
        for (int i = i0; i < i0 + HH; ++i) {
          float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
          for (int r = 0; r < kUpdRows; r += 4) {
            const float4 d = ld4(dzt + i * kUpdTS + r);
            s0 = fmaf(d.x, v0[r], fmaf(d.y, v0[r + 1], fmaf(d.z, v0[r + 2], fmaf(d.w, v0[r + 3], s0))));
            s1 = fmaf(d.x, v1[r], fmaf(d.y, v1[r + 1], fmaf(d.z, v1[r + 2], fmaf(d.w, v1[r + 3], s1))));
          }
          // results unused: fire-and-forget reductions, no load to wait for
          atomicAdd(part + g_off + static_cast<size_t>(i) * n_cols + c0, s0);
          if (two) atomicAdd(part + g_off + static_cast<size_t>(i) * n_cols + c1, s1);
        }
      }
    };
    weight_grad(dz2t, h1s, H, H, net.oW2);    // d W2[i][j] = sum_r d z2[r][i] h1[r][j]
    weight_grad(dz1t, xs, Dp, Din, net.oW1);  // d W1[i][k] = sum_r d z1[r][i] x[r][k]
    __syncthreads();
  }
  // what was kept in registers over all tiles
  part[net.ob1 + j] += gb1;
  part[net.ob2 + j] += gb2;
  if (has_actor) {
#pragma unroll
    for (int k = 0; k < kActions; ++k) part[net.oWa + static_cast<size_t>(k) * H + j] += gWa[k];
    if (j < kActions) part[net.oba + j] += gbh;
  }
  if (has_value) {
    part[net.oWv + j] += gWv;
    if (j == kActions) part[net.obv] += gbh;
  }
  if (lane == 0) {
    double *tp = term_partial + (static_cast<size_t>(blockIdx.x) * 8 + warp) * 3;
    tp[0] += t_actor; tp[1] += t_ent; tp[2] += t_value;
  }
}

template <class U>
__global__ void __launch_bounds__(256) moments_kernel(Moments m) {  // of the advantages
  dependents_may_start();
  wait_for_predecessor();
  moments_block<U>(m);
}

__global__ void __launch_bounds__(256) adam_kernel(AdamArgs a, size_t n) {
  dependents_may_start();
  wait_for_predecessor();
  const float scale = adam_scale(a);
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += static_cast<size_t>(gridDim.x) * blockDim.x) adam_element(a, adam_load(a, i), __ldcg(a.grad + i), scale, i);
}

// Scratch of the update block, made on first use: the head (two places for the advantages' moments, their counters, and the partial sums of
// one, the gradient's sums of squares, the partial sums of the other), then [weight image][term partials][transposed
// weights][partial gradients: one slice per CTA].  The image directly behind the head: a step finds it without knowing the slices.
size_t upd_smem_bytes(int Din, int H) {
  return sizeof(float) * (static_cast<size_t>(kUpdRows) * ((Din + 3) & ~3) + 2 * static_cast<size_t>(kUpdRows) * H +
                          static_cast<size_t>(H) * kUpdTS + kUpdRows * 8 + kUpdRows * 2);
}

// The head of the scratch, the same in every layout of the rest.
constexpr size_t kHeadBytes = 128 + 3 * sizeof(double) * 2 * kMomentBlocks;
Moments adv_moments_of(mava_rollout *h, int place, const UpdRows &rows) {  // (`place`, 0 or 1: see launch_ppo_grad)
  unsigned char *p = static_cast<unsigned char *>(h->d_upd);
  const int which = 2 * place;
  return Moments{h->buf.adv, rows.n, rows, reinterpret_cast<double *>(p + 128) + which * 2 * kMomentBlocks, reinterpret_cast<double *>(p) + 4 * which,
                 reinterpret_cast<unsigned *>(p + 96) + which};
}
// The gradient's sums of squares, between the two places of the moments' partial sums.
double *grad_squares_of(mava_rollout *h) { return reinterpret_cast<double *>(static_cast<unsigned char *>(h->d_upd) + 128) + 2 * kMomentBlocks; }

struct UpdScratch {
  double *term_part;
  float *wt, *partial;
  unsigned char *image;  // weight image of the tensor-core paths
  int slices;
};
size_t image_room() {
  return (ppo_tc_image_bytes() + 255) / 256 * 256;
}
UpdScratch carve(mava_rollout *h, size_t n_params, int slices) {
  unsigned char *p = static_cast<unsigned char *>(h->d_upd);
  UpdScratch s{};
  p += kHeadBytes;
  s.image = p; p += image_room();  // (the same place for every number of slices: a step leaves it to the next minibatch)
  s.term_part = reinterpret_cast<double *>(p); p += sizeof(double) * 3 * 8 * slices;
  s.wt = reinterpret_cast<float *>(p); p += sizeof(float) * ((n_params + 3) / 4 * 4);
  s.partial = reinterpret_cast<float *>(p);
  s.slices = slices;
  return s;
}

}  // namespace

// A bf16 handle takes the tensor-core kernels for the shapes they serve, unless it asked for the fp32 path.
bool update_takes_tensor_cores(const mava_config_t &cfg, int D) {
  return cfg.precision == MAVA_PRECISION_BF16 && (cfg.flags & MAVA_FLAG_UPDATE_FP32) == 0 && ppo_tc_supported(cfg, D);
}
bool update_takes_tensor_cores_256(const mava_config_t &cfg, int D) {
  return cfg.precision == MAVA_PRECISION_BF16 && (cfg.flags & MAVA_FLAG_UPDATE_FP32) == 0 && ppo_tc256_supported(cfg, D);
}

// Scratch that only grows, kept until destroy.
static cudaError_t ensure_bytes(void **p, size_t *have, size_t bytes) {
  if (*p && *have >= bytes) return cudaSuccess;
  cudaFree(*p);
  *p = nullptr;
  *have = 0;
  const cudaError_t err = cudaMalloc(p, bytes);
  if (err == cudaSuccess) *have = bytes;
  return err;
}
static cudaError_t ensure_update_bytes(mava_rollout *h, size_t bytes) {
  const void *had = h->d_upd;
  const size_t had_bytes = h->upd_bytes;
  const cudaError_t err = ensure_bytes(&h->d_upd, &h->upd_bytes, bytes);
  if (err != cudaSuccess || (h->d_upd == had && h->upd_bytes == had_bytes)) return err;
  return cudaMemsetAsync(h->d_upd, 0, 128, h->stream);  // the counters of the moments
}
static cudaError_t ensure_update_ring(mava_rollout *h, size_t bytes) { return ensure_bytes(&h->d_upd_ring, &h->upd_ring_bytes, bytes); }
static size_t update_scratch_bytes(size_t n_params, int slices) {
  return kHeadBytes + sizeof(double) * 3 * 8 * slices + sizeof(float) * ((n_params + 3) / 4 * 4) + image_room() + sizeof(float) * n_params * slices;
}

// How a gradient over the rows of `n_env` environments is cut up, and what it and the optimiser step behind it need.
using Fp32Kernel = void (*)(UpdNet, UpdRows, UpdHyper, const double *, float *, size_t, double *, int *);
struct UpdPlan {
  int sms, slices;
  Tc256Need net, critic;  // H = 256 on the tensor cores
  Fp32Kernel kern;        // fp32 path
  size_t scratch, ring;
};
static cudaError_t plan_update(const mava_rollout *h, int n_env, UpdPlan &plan) {
  const mava_config_t &cfg = h->cfg;
  const int N = cfg.n_agents, H = cfg.hidden;
  const size_t P = param_layout(cfg, h->D, 1).total;
  const long long S = static_cast<long long>(h->last_T) * n_env, R = S * N;  // environment-steps, rows
  const bool central = cfg.net_kind == MAVA_NET_CENTRAL_CRITIC;
  plan = UpdPlan{};
  cudaError_t err = cudaDeviceGetAttribute(&plan.sms, cudaDevAttrMultiProcessorCount, h->device);
  if (err != cudaSuccess) return err;
  const auto at_most = [](long long tiles, long long ctas) { return static_cast<int>(tiles < ctas ? tiles : ctas); };
  if (update_takes_tensor_cores(cfg, h->D)) {  // H <= 128: one CTA (= one gradient slice) per SM over tiles of 128 rows
    plan.slices = at_most((R + 127) / 128, plan.sms);
    plan.scratch = update_scratch_bytes(ppo_tc_slice_floats(), plan.slices);
  } else if (update_takes_tensor_cores_256(cfg, h->D)) {
    plan.net = ppo_tc256_need(R, plan.sms, 1);
    if (central) plan.critic = ppo_tc256_need(S, plan.sms, N);
    plan.scratch = kHeadBytes + plan.net.scratch + plan.critic.scratch;
    plan.ring = plan.net.ring > plan.critic.ring ? plan.net.ring : plan.critic.ring;
  } else {  // fp32: as many CTAs (= gradient slices) as are resident at once with the larger of the two nets' shared-memory needs
    const size_t smem_max = upd_smem_bytes(central ? N * h->D : h->D, H);
    plan.kern = H == 64 ? ppo_net_kernel<64> : (H == 128 ? ppo_net_kernel<128> : (H == 256 ? ppo_net_kernel<256> : nullptr));
    if (!plan.kern) return cudaErrorNotSupported;
    // (the most of any shape: the attribute belongs to the kernel, and another thread may be launching it for another shape)
    err = cudaFuncSetAttribute(plan.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(upd_smem_bytes(kMaxAgents * (kObsFixed + kMaxAgents), 256)));
    if (err != cudaSuccess) return err;
    int per_sm = 1;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, plan.kern, H, smem_max);
    if (err != cudaSuccess) return err;
    plan.slices = at_most((R + kUpdRows - 1) / kUpdRows, static_cast<long long>(plan.sms) * (per_sm < 1 ? 1 : per_sm));
    plan.scratch = update_scratch_bytes(P, plan.slices);
  }
  const size_t step = update_scratch_bytes(P, 1);  // launch_adam_step
  if (plan.scratch < step) plan.scratch = step;
  return cudaSuccess;
}
static cudaError_t ensure_update(mava_rollout *h, const UpdPlan &plan) {
  const cudaError_t err = ensure_update_bytes(h, plan.scratch);
  return err == cudaSuccess && plan.ring > 0 ? ensure_update_ring(h, plan.ring) : err;
}
cudaError_t reserve_update(mava_rollout *h, int n_small, int n_large) {
  UpdPlan small, plan;
  cudaError_t err = plan_update(h, n_small, small);
  if (err == cudaSuccess) err = plan_update(h, n_large, plan);
  if (err != cudaSuccess) return err;
  if (plan.scratch < small.scratch) plan.scratch = small.scratch;
  if (plan.ring < small.ring) plan.ring = small.ring;
  return ensure_update(h, plan);
}

// The rows of a minibatch of environments (nullptr: all) of the last run.
static UpdRows rows_of(const mava_rollout *h, const int32_t *env_ids_dev, int n_env) {
  UpdRows rows{};
  rows.x = h->buf.obs; rows.actions = h->buf.actions; rows.logp_old = h->buf.logp; rows.adv = h->buf.adv;
  rows.n = static_cast<long long>(h->last_T) * n_env * h->cfg.n_agents;
  rows.env_ids = env_ids_dev; rows.n_ids = n_env; rows.E = h->cfg.n_envs; rows.per_env = h->cfg.n_agents;
  if (h->cfg.net_kind != MAVA_NET_CENTRAL_CRITIC) { rows.value_old = h->buf.values; rows.ret = h->buf.ret; rows.vstride = 1; }
  return rows;
}

// `prepared`: the step directly in front, itself directly behind a gradient, was told of this minibatch (the `next` of launch_adam_step)
// and leaves its weight image and its advantages' moments.  The gradient kernel lets its successors start only after its own wait,
// so whatever was launched before the gradient in front is complete when that step starts: the step may take the moments, and
// this call fetch its first rows, before their waits.  The gradient in front may still read its own moments then, so the two
// have different places (`place`, 0 or 1).
cudaError_t launch_ppo_grad(mava_rollout *h, const float *params_dev, const mava_ppo_hyper_t &hyper, float *grad_dev,
                            float *terms_dev, const int32_t *env_ids_dev, int32_t n_ids, int place, bool prepared) {
  const mava_config_t &cfg = h->cfg;
  const int T = h->last_T, E = cfg.n_envs, N = cfg.n_agents, D = h->D, H = cfg.hidden;
  const ParamLayout L = param_layout(cfg, D, 1);
  const size_t P = L.total;
  const int n_env = env_ids_dev ? n_ids : E;  // environments in the minibatch
  UpdPlan plan;
  cudaError_t err = plan_update(h, n_env, plan);
  if (err == cudaSuccess) err = ensure_update(h, plan);
  if (err != cudaSuccess) return err;
  const int slices = plan.slices;
  const long long R = static_cast<long long>(T) * n_env * N, S = static_cast<long long>(T) * n_env;
  const bool central = cfg.net_kind == MAVA_NET_CENTRAL_CRITIC;
  const UpdHyper hp{hyper.clip_eps, hyper.ent_coef, hyper.vf_coef};
  cudaStream_t st = h->stream;
  const UpdRows rows = rows_of(h, env_ids_dev, n_env);

  if (update_takes_tensor_cores(cfg, D)) {
    const UpdScratch sc = carve(h, ppo_tc_slice_floats(), slices);
    const TermSums terms{sc.term_part, sc.term_part, 4 * slices, 4 * slices, R, R, hp, terms_dev};
    return launch_ppo_net_tc(h, params_dev, L, rows, hp, adv_moments_of(h, place, rows), prepared, sc.image, sc.partial, sc.term_part, slices, grad_dev, terms,
                             grad_squares_of(h));
  }

  UpdRows crows{};  // the centralised critic's: a row is an environment-step
  crows.x = h->buf.obs; crows.value_old = h->buf.values; crows.ret = h->buf.ret; crows.vstride = N; crows.n = S;
  crows.env_ids = env_ids_dev; crows.n_ids = n_env; crows.E = E; crows.per_env = 1;

  // H = 256 on the tensor cores: the actor / shared-torso net and, one input slab per agent, the centralised critic's
  if (update_takes_tensor_cores_256(cfg, D)) {
    const int sms = plan.sms;
    unsigned char *p = static_cast<unsigned char *>(h->d_upd) + kHeadBytes;
    const Moments adv = adv_moments_of(h, place, rows);
    const double *stats = adv.out;
    TermSums terms{nullptr, nullptr, 0, 0, R, central ? S : R, hp, terms_dev};
    if (!central) {
      const Tc256Net net{L.W1, L.b1, L.W2, L.b2, L.Wa, L.ba, L.Wv, L.bv, 1, true, true};
      return launch_ppo_net_tc256(h, params_dev, net, rows, hp, adv, stats, p, h->d_upd_ring, sms, grad_dev, terms);
    }
    const Tc256Net anet{L.W1, L.b1, L.W2, L.b2, L.Wa, L.ba, 0, 0, 1, true, false};
    err = launch_ppo_net_tc256(h, params_dev, anet, rows, hp, adv, stats, p, h->d_upd_ring, sms, grad_dev, terms);
    if (err != cudaSuccess) return err;
    const Tc256Net cnet{L.C1, L.c1, L.C2, L.c2, 0, 0, L.Cv, L.cv, N, false, true};
    return launch_ppo_net_tc256(h, params_dev, cnet, crows, hp, Moments{}, stats, p + plan.net.scratch, h->d_upd_ring, sms, grad_dev, terms);
  }

  const int joint = N * D;
  const Fp32Kernel kern = plan.kern;
  const UpdScratch sc = carve(h, P, slices);
  // transposed copies of the hidden layers' weights, in the parameters' own order
  auto tr = [&](size_t off, int out, int in) {
    transpose_kernel<<<64, 256, 0, st>>>(params_dev + off, sc.wt + off, out, in);
    h->launches += 1;
  };
  tr(L.W1, H, D); tr(L.W2, H, H);
  if (central) { tr(L.C1, H, joint); tr(L.C2, H, H); }
  const Moments adv = adv_moments_of(h, place, rows);
  err = launch_dependent(rows_need_64_bits(rows, R) ? moments_kernel<uint64_t> : moments_kernel<uint32_t>, kMomentBlocks, 256, 0, st, adv);
  h->launches += 1;
  if (err == cudaSuccess) err = cudaMemsetAsync(sc.term_part, 0, sizeof(double) * 3 * 8 * slices, st);
  if (err == cudaSuccess) err = cudaMemsetAsync(sc.partial, 0, sizeof(float) * P * slices, st);
  if (err != cudaSuccess) return err;
  auto run_net = [&](const UpdNet &net, const UpdRows &rows) {
    const size_t smem = upd_smem_bytes(net.Din, net.H);
    kern<<<slices, net.H, smem, st>>>(net, rows, hp, adv.out, sc.partial, P, sc.term_part, h->d_status);
    h->launches += 1;
    return cudaGetLastError();
  };
  UpdNet actor{};
  actor.W1 = params_dev + L.W1; actor.b1 = params_dev + L.b1; actor.W2 = params_dev + L.W2; actor.b2 = params_dev + L.b2;
  actor.W1t = sc.wt + L.W1; actor.W2t = sc.wt + L.W2;
  actor.Wa = params_dev + L.Wa; actor.ba = params_dev + L.ba;
  actor.Din = D; actor.H = H;
  actor.oW1 = L.W1; actor.ob1 = L.b1; actor.oW2 = L.W2; actor.ob2 = L.b2; actor.oWa = L.Wa; actor.oba = L.ba;
  if (!central) {
    actor.Wv = params_dev + L.Wv; actor.bv = params_dev + L.bv; actor.oWv = L.Wv; actor.obv = L.bv;
    err = run_net(actor, rows);
  } else {
    err = run_net(actor, rows);
    if (err != cudaSuccess) return err;
    UpdNet critic{};
    critic.W1 = params_dev + L.C1; critic.b1 = params_dev + L.c1; critic.W2 = params_dev + L.C2; critic.b2 = params_dev + L.c2;
    critic.W1t = sc.wt + L.C1; critic.W2t = sc.wt + L.C2;
    critic.Wv = params_dev + L.Cv; critic.bv = params_dev + L.cv;
    critic.Din = joint; critic.H = H;
    critic.oW1 = L.C1; critic.ob1 = L.c1; critic.oW2 = L.C2; critic.ob2 = L.c2; critic.oWv = L.Cv; critic.obv = L.cv;
    err = run_net(critic, crows);
  }
  if (err != cudaSuccess) return err;
  const TermSums terms{sc.term_part, sc.term_part, 8 * slices, 8 * slices, R, central ? S : R, hp, terms_dev};
  h->launches += 1;
  return launch_dependent(reduce_slices_kernel<IdentityMap>, kReduceBlocks, kReduceThreads, 0, st, static_cast<const float *>(sc.partial), static_cast<int>(P), slices,
                          grad_dev, terms, grad_squares_of(h), IdentityMap{});
}

cudaError_t launch_adam_step(mava_rollout *h, float *params_dev, const float *grad_dev, float *m_dev, float *v_dev, int32_t step,
                             const mava_ppo_hyper_t &hp, bool norm_known, const NextMinibatch *next) {
  const ParamLayout L = param_layout(h->cfg, h->D, 1);
  const size_t P = L.total;
  const bool tc = update_takes_tensor_cores(h->cfg, h->D);
  cudaError_t err = ensure_update_bytes(h, update_scratch_bytes(P, 1));
  if (err != cudaSuccess) return err;
  double *squares = grad_squares_of(h);
  if (!norm_known) {
    err = tc ? launch_grad_squares_tc(h, L, grad_dev, squares)
             : launch_dependent(grad_squares_kernel<IdentityMap>, kMomentBlocks, kGradLanes, 0, h->stream, grad_dev, squares, static_cast<int>(P), IdentityMap{});
    if (err != cudaSuccess) return err;
    h->launches += 1;
  }
  const float corr1 = static_cast<float>(1.0 - pow(static_cast<double>(hp.beta1), step));
  const float corr2 = static_cast<float>(1.0 - pow(static_cast<double>(hp.beta2), step));
  const AdamArgs adam{params_dev, grad_dev, m_dev, v_dev, squares, hp.max_grad_norm, hp.lr, hp.beta1, hp.beta2, hp.adam_eps, corr1, corr2};
  if (next && tc)
    return launch_step_tc(h, adam, L, adv_moments_of(h, next->place, rows_of(h, next->env_ids, next->n)), carve(h, ppo_tc_slice_floats(), 1).image);
  h->launches += 1;
  const int blocks = static_cast<int>((P + 255) / 256 < 2 * 148 ? (P + 255) / 256 : 2 * 148);
  return launch_dependent(adam_kernel, blocks, 256, 0, h->stream, adam, P);
}

// Whether a gradient call leaves the gradient's sums of squares behind (update_takes_tensor_cores_256: its reduction does not).
bool ppo_grad_leaves_norm(const mava_rollout *h) { return !update_takes_tensor_cores_256(h->cfg, h->D); }
// Whether a step prepares the minibatch that it is told of.
bool adam_step_prepares(const mava_rollout *h) { return update_takes_tensor_cores(h->cfg, h->D); }

}  // namespace mava

// Update block on the tensor cores (sm_100a, tcgen05): the multi-agent PPO loss of one minibatch and its gradient for the
// shared-torso nets with H <= 128 and D <= 80, bf16 operands with fp32 accumulation in tensor memory.
//
// One persistent CTA per SM walks over tiles of 128 rows.  Every matrix of a tile lives once in shared memory as a bf16
// tile in the canonical core-matrix layout [row][feature] (core matrix = 8 rows x 16 bytes; feature chunks 128 bytes
// apart, 8-row groups C*16 bytes apart for a tile of C features).  Read with the feature index as K it is the K-major
// A operand of the per-row products (forward layers, d h = d z . W); read with the row index as K it is an MN-major
// operand of the products that sum over rows (d W = d z^T . input), so no transposed copy is ever written.  The same
// holds for the weights: W2 [out][in] is the K-major B operand of the forward layer and, read the other way, the
// MN-major B operand of d h1 = d z2 . W2.
//   per tile:  x -> z1 -> h1 -> z2 -> h2 -> logits, value -> loss and its per-row derivatives (fp32, thread = row)
//              -> d h2 -> d z2 -> d h1 -> d z1, and on the side d Wh^T += h2^T . dhead, d W2 += d z2^T . h1,
//              d W1 += d z1^T . x, d b2 += d z2^T . 1, d b1 += d z1^T . 1 (the ones are column 7 of the dhead tile).
// The weight-gradient accumulators stay in tensor memory for all tiles of the CTA and are written once, into the CTA's
// own slice of the partial-gradient array; a last kernel adds the slices in a fixed order (reduce_slices_kernel: four quarters of
// them, each in slice order), so the gradient is the same bytes on every call.  Rounding points are those of the bf16-operand
// mode of the float64 oracle.
// A hidden width below 128 is padded with zero units (their activations, gates and gradients are exactly zero).
// MMAs are issued by one elected lane; tcgen05.commit tracks all MMAs issued before it, so a tile buffer may be rewritten as
// soon as a later commit has been waited for.  Every mbarrier wait is bounded.
#include <cuda_bf16.h>

#include "common.cuh"
#include "layout.h"
#include "tc_common.cuh"
#include "update_common.cuh"

namespace mava {
namespace {

constexpr int kUR = 128;        // rows per tile (M of the per-row products, K of the weight-gradient products)
constexpr int kUH = 128;        // hidden width, padded
constexpr int kUK1 = 80;        // input width, padded to the MMA's K step
constexpr int kUHeads = 16;     // six logits, the value, a column of ones, eight columns of zeros
constexpr int kUMain = 256;     // threads of the epilogues: thread = (row, column half)
constexpr int kULoaders = 3;    // warps that bring the rows in (with a fourth, 13 warps would leave 128 registers per thread, which spill)
constexpr int kUThreads = kUMain + 32 * kULoaders + 32;  // and one that issues the MMAs

// weight image: bf16 tiles W1 [H][K1], W2 [H][H], Wh [16][H]; then fp32 b1 [H], b2 [H], bh [8]
constexpr uint32_t kImgW1 = 0, kImgW2 = kImgW1 + kUH * kUK1 * 2, kImgWh = kImgW2 + kUH * kUH * 2;
constexpr uint32_t kImgB1 = kImgWh + kUHeads * kUH * 2, kImgB2 = kImgB1 + kUH * 4, kImgBh = kImgB2 + kUH * 4;
constexpr uint32_t kImgBytes = kImgBh + 32;
static_assert(kImgBytes % 16 == 0, "one bulk copy");

// tensor-memory columns
constexpr uint32_t kColAcc = 0, kColDW2 = 128, kColDW1 = 256, kColHead = 352, kColDWh = 384, kColDB2 = 416, kColDB1 = 448;
constexpr uint32_t kTmemCols = 512;

struct UtcSmem {
  alignas(128) unsigned char img[(kImgBytes + 127) / 128 * 128];
  alignas(128) unsigned char x[2][(kUR / 8) * (kUK1 / 8) * kALbo];  // feature chunks 144 bytes apart (see a_offset): the
                                                                    // converter's 2-byte stores then spread over the banks
  alignas(128) unsigned char h1[kUR * kUH * 2];
  alignas(128) unsigned char h2[kUR * kUH * 2];   // d z1 once h2's last reader is done
  alignas(128) unsigned char dz2[kUR * kUH * 2];
  alignas(128) unsigned char dhead[kUR * kUHeads * 2];
  int rmap[kUR];  // trajectory rows of the tile that is being fetched
  float red[4][8];
  alignas(8) uint64_t bar_load, bar_mma, bar_end, x_full[2];
  uint32_t tmem_base;
  int abort;  // the main threads gave up
};

struct PrepImage {
  const float *params;
  unsigned char *image;
  ParamLayout L;
  int D, H;
  __device__ void operator()(int tid, int nth) const;
};
// One element per thread: a kernel that everything behind it waits for (as loops over the parts with 8 k threads it took 3 us more).
constexpr int kPrepW1 = kUH * kUK1, kPrepW2 = kUH * kUH, kPrepWh = kUHeads * kUH, kPrepTotal = kPrepW1 + kPrepW2 + kPrepWh + 2 * kUH + 8;
constexpr int kPrepBlocks = (kPrepTotal + 255) / 256;
__device__ __forceinline__ void PrepImage::operator()(int tid, int nth) const {
  for (int i = tid; i < kPrepTotal; i += nth) {
    size_t src = 0, at;    // parameter, place in the image
    bool real, wide = false;  // whether there is such a parameter; fp32 instead of bf16
    int j = i;
    if (j < kPrepW1) {
      const int n = j / kUK1, k = j - n * kUK1;
      real = n < H && k < D; src = L.W1 + static_cast<size_t>(n) * D + k; at = kImgW1 + canon_offset(n, k, kUK1);
    } else if ((j -= kPrepW1) < kPrepW2) {
      const int n = j / kUH, k = j - n * kUH;
      real = n < H && k < H; src = L.W2 + static_cast<size_t>(n) * H + k; at = kImgW2 + canon_offset(n, k, kUH);
    } else if ((j -= kPrepW2) < kPrepWh) {
      const int n = j / kUH, k = j - n * kUH;
      real = k < H && n <= kActions; src = n < kActions ? L.Wa + static_cast<size_t>(n) * H + k : L.Wv + k; at = kImgWh + canon_offset(n, k, kUH);
    } else if ((j -= kPrepWh) < 2 * kUH) {
      const int n = j % kUH;
      real = n < H; src = (j < kUH ? L.b1 : L.b2) + n; at = (j < kUH ? kImgB1 : kImgB2) + 4 * n; wide = true;
    } else {
      j -= 2 * kUH;
      real = j <= kActions; src = j < kActions ? L.ba + j : L.bv; at = kImgBh + 4 * j; wide = true;
    }
    const float v = real ? __ldcg(params + src) : 0.0f;
    if (wide) *reinterpret_cast<float *>(image + at) = v;
    else *reinterpret_cast<__nv_bfloat16 *>(image + at) = __float2bfloat16_rn(v);
  }
}

// Descriptor of a canonical tile of C features read with the feature index as K (step k = features 16 k ..).
__device__ __forceinline__ uint64_t desc_k(uint32_t tile, int C, int k) { return smem_desc(tile + k * 256, 128, C * 16); }
// The same tile read with the row index as K (step k = rows 16 k ..): the 8-row groups are the K groups, the feature
// chunks the MN groups: the descriptor's leading-dimension offset is then the step between K groups (C*16 bytes) and
// its stride offset the step between MN groups (128 bytes).
__device__ __forceinline__ uint64_t desc_mn(uint32_t tile, int C, int k) { return smem_desc(tile + k * 2 * C * 16, C * 16, 128); }
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;  // operand is MN-major

// A CTA's slice of the partial gradients, matrices as [column / 4][unit][4] so that the lanes of a warp (= units) write whole
// lines (written row by row in the parameters' order, a slice took 33 k cycles to leave; like this 2 k):
// d W2 [128 columns], d W1 [80 columns], d Wh^T [8 columns], then d b2 [128], d b1 [128], the heads' biases [8].
constexpr int kSlW2 = 0, kSlW1 = kSlW2 + kUH * kUH, kSlWh = kSlW1 + kUK1 * kUH, kSlB2 = kSlWh + 8 * kUH, kSlB1 = kSlB2 + kUH, kSlBh = kSlB1 + kUH,
              kSlice = kSlBh + 8;
// The parameter behind a slice's element, -1 for padding.
struct SliceMap {
  ParamLayout L;
  int D, H;
  __device__ __forceinline__ long long operator()(int j) const {
    if (j < kSlB2) {
      const int e = j < kSlW1 ? j : (j < kSlWh ? j - kSlW1 : j - kSlWh), c = e / (4 * kUH) * 4 + (e & 3), unit = (e >> 2) % kUH;
      if (unit >= H) return -1;
      if (j < kSlW1) return c < H ? static_cast<long long>(L.W2) + unit * H + c : -1;
      if (j < kSlWh) return c < D ? static_cast<long long>(L.W1) + unit * D + c : -1;
      return c < kActions ? static_cast<long long>(L.Wa) + c * H + unit : (c == kActions ? static_cast<long long>(L.Wv) + unit : -1);
    }
    if (j < kSlBh) {
      const int unit = (j - kSlB2) % kUH;
      return unit < H ? static_cast<long long>(j < kSlB1 ? L.b2 : L.b1) + unit : -1;
    }
    const int k = j - kSlBh;
    return k < kActions ? static_cast<long long>(L.ba) + k : (k == kActions ? static_cast<long long>(L.bv) : -1);
  }
};

template <class U>  // row numbers of the batch (real_row)
__global__ void __launch_bounds__(kUThreads, 1)
ppo_net_tc_kernel(const unsigned char *image, UpdRows rows, UpdHyper hp, const double *adv_stats,
                  float *partial, double *term_partial, int *status, int D, bool rows_ready) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  UtcSmem &sm = *reinterpret_cast<UtcSmem *>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & (kUR - 1), half = tid >> 7;
  const int role = __shfl_sync(0xFFFFFFFFu, warp, 0);  // (uniform to the compiler)
  const uint32_t bar_load = smem_u32(&sm.bar_load), bar_mma = smem_u32(&sm.bar_mma), bar_end = smem_u32(&sm.bar_end), x_full0 = smem_u32(&sm.x_full[0]);
  if (tid == 0) {
    sm.abort = 0;
    mbar_init(bar_load, 1); mbar_init(bar_mma, 1); mbar_init(bar_end, 1); mbar_init(x_full0, kULoaders); mbar_init(x_full0 + 8, kULoaders);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the x tiles' pad columns and the dhead tile's upper eight columns stay zero for the whole run
  for (int i = tid; i < static_cast<int>(sizeof(sm.x) / 16); i += kUThreads) sts_zero16(smem_u32(sm.x) + 16u * i);
  for (int i = tid; i < static_cast<int>(sizeof(sm.dhead) / 16); i += kUThreads) sts_zero16(smem_u32(sm.dhead) + 16u * i);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // barrier of the main threads and the MMA warp; `any`: also whether one of them has given up
  auto step_barrier = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kUMain + 32) : "memory"); };
  auto step_any = [&](bool pred) {
    uint32_t out;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}"
                 : "=r"(out) : "r"(static_cast<uint32_t>(pred)), "n"(kUMain + 32) : "memory");
    return out != 0;
  };
  // The loaders need neither the weights nor the moments: the first tile's rows come while both are on their way.
  const bool loader = role >= kUMain / 32 && role < kUMain / 32 + kULoaders;
  bool timed_out = false;
  if (!loader || !rows_ready) wait_for_predecessor();
  if (!loader) {
    dependents_may_start();  // (after the wait: launch_ppo_grad)
    if (tid == 0) {
      mbar_expect_tx(bar_load, kImgBytes);
      constexpr uint32_t kChunk = 16384;
      for (uint32_t o = 0; o < kImgBytes; o += kChunk) bulk_load(smem_u32(sm.img + o), image + o, min(kChunk, kImgBytes - o), bar_load);
    }
    timed_out = step_any(!mbar_wait(bar_load, 0));
    if (timed_out) *reinterpret_cast<volatile int *>(&sm.abort) = 1;
  }

  const uint32_t tmem = sm.tmem_base;
  const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
  const uint32_t w1 = smem_u32(sm.img + kImgW1), w2 = smem_u32(sm.img + kImgW2), wh = smem_u32(sm.img + kImgWh);
  const uint32_t h1t = smem_u32(sm.h1), h2t = smem_u32(sm.h2), dz2t = smem_u32(sm.dz2), dz1t = h2t,
                 dht = smem_u32(sm.dhead);
  const uint32_t b1 = smem_u32(sm.img + kImgB1), b2 = smem_u32(sm.img + kImgB2);
  const float *bh = reinterpret_cast<const float *>(sm.img + kImgBh);
  const float mean = loader ? 0.0f : static_cast<float>(__ldcg(adv_stats));
  const float inv_std = loader ? 0.0f : 1.0f / (static_cast<float>(__ldcg(adv_stats + 1)) + 1e-8f);
  const float inv_n = 1.0f / static_cast<float>(rows.n);
  const long long n_tiles = (rows.n + kUR - 1) / kUR;
  const int my_tiles = blockIdx.x < n_tiles ? static_cast<int>((n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
  auto tile_of = [&](int i) { return static_cast<long long>(blockIdx.x) + static_cast<long long>(i) * gridDim.x; };

  uint32_t ph_mma = 0;
  double t_actor = 0.0, t_ent = 0.0, t_value = 0.0;
  float gbh[kActions + 1];  // gradient of the heads' biases, this thread's rows
#pragma unroll
  for (int k = 0; k <= kActions; ++k) gbh[k] = 0.0f;

  // d W1 [out][in] += d z1^T . x and d b1 [out] += d z1^T . ones (K = rows) of a tile, one lane
  auto weight_grad_1 = [&](uint32_t xt, uint32_t keep) {
#pragma unroll
    for (int k = 0; k < kUR / 16; ++k)
      mma_bf16(tmem + kColDW1, desc_mn(dz1t, kUH, k), smem_desc(xt + k * 2 * (kUK1 / 8) * kALbo, (kUK1 / 8) * kALbo, kALbo),
               instr_desc(kUH, kUK1) | kAmn | kBmn, keep | (k > 0));
#pragma unroll
    for (int k = 0; k < kUR / 16; ++k)
      mma_bf16(tmem + kColDB1, desc_mn(dz1t, kUH, k), desc_mn(dht, kUHeads, k), instr_desc(kUH, kUHeads) | kAmn | kBmn, keep | (k > 0));
    mma_commit(bar_end);
  };
  // hidden-layer epilogue: this thread's 64 accumulator columns + bias -> ReLU -> bf16 -> its row of `dst`; one gate bit per
  // unit out (pair i of 32 columns: bits 15 - i and 31 - i of gate[columns / 32]).  Two columns per instruction throughout
  // (column by column, with the gate bits shifted in one by one, an epilogue took 1.5 k cycles).
  auto fwd_epilogue = [&](uint32_t bias, uint32_t dst, uint32_t *gate) {
    uint32_t r[64];
    tmem_ld32_nowait(tmem + kColAcc + lane_off + 64u * half, r);
    tmem_ld32_nowait(tmem + kColAcc + lane_off + 64u * half + 32u, r + 32);
    tmem_ld_wait();
    const uint32_t drow = dst + static_cast<uint32_t>((row >> 3) * (kUH * 16) + (row & 7) * 16 + half * 8 * 128);
    gate[0] = gate[1] = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 ba = lds_float4(bias + 256u * half + 32u * q), bb = lds_float4(bias + 256u * half + 32u * q + 16u);
      add2(r[8 * q], r[8 * q + 1], ba.x, ba.y); add2(r[8 * q + 2], r[8 * q + 3], ba.z, ba.w);
      add2(r[8 * q + 4], r[8 * q + 5], bb.x, bb.y); add2(r[8 * q + 6], r[8 * q + 7], bb.z, bb.w);
      uint32_t pk[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        pk[e] = relu_pack_bf16(r[8 * q + 2 * e], r[8 * q + 2 * e + 1]);
        gate[q / 4] |= positive_mask(pk[e]) & (0x80008000u >> (4 * (q & 3) + e));
      }
      sts_v4(drow + static_cast<uint32_t>(q * 128), pk[0], pk[1], pk[2], pk[3]);
    }
  };
  // backward epilogue: d h (accumulator) gated by the layer's ReLU -> bf16 -> this thread's row of `dst`
  auto bwd_epilogue = [&](const uint32_t *gate, uint32_t dst) {
    uint32_t r[64];
    tmem_ld32_nowait(tmem + kColAcc + lane_off + 64u * half, r);
    tmem_ld32_nowait(tmem + kColAcc + lane_off + 64u * half + 32u, r + 32);
    tmem_ld_wait();
    const uint32_t drow = dst + static_cast<uint32_t>((row >> 3) * (kUH * 16) + (row & 7) * 16 + half * 8 * 128);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      uint32_t pk[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        pk[e] = pack_bf16(__uint_as_float(r[8 * q + 2 * e]), __uint_as_float(r[8 * q + 2 * e + 1])) & sign_mask(gate[q / 4] << (4 * (q & 3) + e));
      sts_v4(drow + static_cast<uint32_t>(q * 128), pk[0], pk[1], pk[2], pk[3]);
    }
  };

  if (timed_out) {
    // nothing was started
  } else if (loader) {
    // ---- the rows: sixteen at a time, the warps in turn, consecutive lanes consecutive features; a
    // tile ahead of the products (with the conversion on the main threads' chain a tile of 11 k cycles took 17 k)
    const int lw = role - kUMain / 32;
    const bool third = lane + 64 < D;
    for (int i = 0; i < my_tiles && !timed_out; ++i) {
      __syncwarp();
#pragma unroll
      for (int e = lane; e < 64; e += 32) {  // where this warp's rows lie (both look-ups in flight, before the wait)
        const int c = lw + kULoaders * (e / 16);
        const long long q = tile_of(i) * kUR + 16 * c + (e & 15);
        if (c < kUR / 16) sm.rmap[16 * c + (e & 15)] = static_cast<int>(q < rows.n ? real_row<U>(rows, q) : -1);
      }
      __syncwarp();
      if (i >= 2) timed_out = !mbar_wait_warp(bar_end, static_cast<uint32_t>(i) & 1u);  // d W1 of tile i - 2 has read this x tile
      if (timed_out || *reinterpret_cast<volatile int *>(&sm.abort)) break;
#pragma unroll 1
      for (int c = lw; c < kUR / 16; c += kULoaders) {
        const uint32_t rmap = smem_u32(&sm.rmap[16 * c]);
        const uint32_t my_col = smem_u32(sm.x[i & 1]) + a_offset<kUK1>(16 * c, lane);
        float v[16][3];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const int src = lds_s32(rmap + 4u * static_cast<uint32_t>(r));
          const float *p = rows.x + static_cast<long long>(src) * D + lane;
          v[r][0] = ldg_if(p, src >= 0);  // (D > 64: the first two are columns of every row)
          v[r][1] = ldg_if(p + 32, src >= 0);
          v[r][2] = ldg_if(p + 64, src >= 0 && third);
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) {  // (a chunk of eight features is 144 bytes on: 32 features are 576)
          const uint32_t at = my_col + static_cast<uint32_t>(r >> 3) * ((kUK1 / 8) * kALbo) + (r & 7) * 16;
          sts_u16(at, bf16_bits(v[r][0]));
          sts_u16(at + 576u, bf16_bits(v[r][1]));
          if (third) sts_u16(at + 1152u, bf16_bits(v[r][2]));
        }
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(x_full0 + 8u * (i & 1)) : "memory");
    }
  } else if (role == kUMain / 32 + kULoaders) {
    // ---- the MMAs, in the order of the chain; the products that only the weight gradients need follow the one that the chain
    // waits for.  tcgen05.commit covers everything issued before it, so a main thread that has waited for a later product
    // knows that the earlier ones have read their tiles.
    for (int i = 0; i < my_tiles && !timed_out; ++i) {
      const uint32_t xt = smem_u32(sm.x[i & 1]);
      const uint32_t keep = i > 0 ? 1u : 0u;  // the weight-gradient accumulators start at the CTA's first tile
      timed_out = !mbar_wait_warp(x_full0 + 8u * (i & 1), static_cast<uint32_t>(i >> 1) & 1u);
      tc_fence_after();
      if (elect_one()) {  // z1
#pragma unroll
        for (int k = 0; k < kUK1 / 16; ++k)
          mma_bf16(tmem + kColAcc, smem_desc(xt + k * 2 * kALbo, kALbo, (kUK1 / 8) * kALbo), desc_k(w1, kUK1, k), instr_desc(kUR, kUH), k > 0);
        mma_commit(bar_mma);
        if (i > 0) weight_grad_1(smem_u32(sm.x[(i - 1) & 1]), i > 1 ? 1u : 0u);
      }
      __syncwarp();
      step_barrier();
      tc_fence_after();
      if (elect_one()) {  // z2
#pragma unroll
        for (int k = 0; k < kUH / 16; ++k) mma_bf16(tmem + kColAcc, desc_k(h1t, kUH, k), desc_k(w2, kUH, k), instr_desc(kUR, kUH), k > 0);
        mma_commit(bar_mma);
      }
      __syncwarp();
      step_barrier();
      tc_fence_after();
      if (elect_one()) {  // heads
#pragma unroll
        for (int k = 0; k < kUH / 16; ++k) mma_bf16(tmem + kColHead, desc_k(h2t, kUH, k), desc_k(wh, kUH, k), instr_desc(kUR, kUHeads), k > 0);
        mma_commit(bar_mma);
      }
      __syncwarp();
      step_barrier();
      tc_fence_after();
      if (elect_one()) {
        // d h2 = dhead . Wh (K = the 16 head columns)
        mma_bf16(tmem + kColAcc, desc_k(dht, kUHeads, 0), desc_mn(wh, kUH, 0), instr_desc(kUR, kUH) | kBmn, 0);
        mma_commit(bar_mma);
        // d Wh^T [unit][head column] += h2^T . dhead (K = rows)
#pragma unroll
        for (int k = 0; k < kUR / 16; ++k)
          mma_bf16(tmem + kColDWh, desc_mn(h2t, kUH, k), desc_mn(dht, kUHeads, k), instr_desc(kUH, kUHeads) | kAmn | kBmn, keep | (k > 0));
      }
      __syncwarp();
      step_barrier();
      tc_fence_after();
      if (elect_one()) {
        // d h1 = d z2 . W2 (K = the out units of layer 2)
#pragma unroll
        for (int k = 0; k < kUH / 16; ++k) mma_bf16(tmem + kColAcc, desc_k(dz2t, kUH, k), desc_mn(w2, kUH, k), instr_desc(kUR, kUH) | kBmn, k > 0);
        mma_commit(bar_mma);
        // d W2 [out][in] += d z2^T . h1 and d b2 [out] += d z2^T . ones (K = rows)
#pragma unroll
        for (int k = 0; k < kUR / 16; ++k)
          mma_bf16(tmem + kColDW2, desc_mn(dz2t, kUH, k), desc_mn(h1t, kUH, k), instr_desc(kUH, kUH) | kAmn | kBmn, keep | (k > 0));
#pragma unroll
        for (int k = 0; k < kUR / 16; ++k)
          mma_bf16(tmem + kColDB2, desc_mn(dz2t, kUH, k), desc_mn(dht, kUHeads, k), instr_desc(kUH, kUHeads) | kAmn | kBmn, keep | (k > 0));
      }
      __syncwarp();
      if (step_any(timed_out)) timed_out = true;
    }
    if (!timed_out && my_tiles > 0) {
      tc_fence_after();
      if (elect_one()) weight_grad_1(smem_u32(sm.x[(my_tiles - 1) & 1]), my_tiles > 1 ? 1u : 0u);
      __syncwarp();
    }
  } else {
  for (int i = 0; i < my_tiles && !timed_out; ++i) {
    const long long row0 = tile_of(i) * kUR;
    const int n_valid = static_cast<int>(min(static_cast<long long>(kUR), rows.n - row0));
    const long long my_row = row < n_valid ? real_row<U>(rows, row0 + row) : -1;
    int action = 0;
    float logp_old = 0.0f, adv = 0.0f, v_old = 0.0f, ret = 0.0f;
    if (half == 0) {
      if (row < n_valid && my_row < 0) atomicExch(status, kStatusBadIndex);
      if (my_row >= 0) {  // used after the heads: the loads are in flight meanwhile
        action = rows.actions[my_row]; logp_old = rows.logp_old[my_row]; adv = rows.adv[my_row];
        v_old = rows.value_old[my_row * rows.vstride]; ret = rows.ret[my_row * rows.vstride];
      }
    }
    timed_out |= !mbar_wait(bar_mma, ph_mma); ph_mma ^= 1;
    tc_fence_after();
    uint32_t gate1[2], gate2[2];
    fwd_epilogue(b1, h1t, gate1);
    fence_async_smem(); tc_fence_before();
    step_barrier();
    timed_out |= !mbar_wait(bar_mma, ph_mma); ph_mma ^= 1;
    tc_fence_after();
    fwd_epilogue(b2, h2t, gate2);
    fence_async_smem(); tc_fence_before();
    step_barrier();
    timed_out |= !mbar_wait(bar_mma, ph_mma); ph_mma ^= 1;
    tc_fence_after();
    // ---- loss terms and the per-row derivatives with respect to the six logits and the value (thread = row)
    if (half == 0) {
      float hv[16], d[8];
      tmem_ld16(tmem + kColHead + lane_off, hv);
#pragma unroll
      for (int k = 0; k < 8; ++k) d[k] = 0.0f;
      if (my_row >= 0) {
        float l[kActions], m = -INFINITY, sum = 0.0f;
#pragma unroll
        for (int k = 0; k < kActions; ++k) { l[k] = hv[k] + bh[k]; m = fmaxf(m, l[k]); }
#pragma unroll
        for (int k = 0; k < kActions; ++k) sum += expf(l[k] - m);
        const float lse = m + logf(sum);
        float ent = 0.0f, p[kActions], lp[kActions], lpa = 0.0f;
#pragma unroll
        for (int k = 0; k < kActions; ++k) {
          lp[k] = l[k] - lse; p[k] = expf(lp[k]); ent -= p[k] * lp[k];
          if (k == action) lpa = lp[k];
        }
        const float rho = expf(lpa - logp_old);
        const float ahat = (adv - mean) * inv_std;
        const float clipped = fminf(fmaxf(rho, 1.0f - hp.clip_eps), 1.0f + hp.clip_eps);
        const float s1 = rho * ahat, s2 = clipped * ahat;
        const bool inside = rho >= 1.0f - hp.clip_eps && rho <= 1.0f + hp.clip_eps;
        const float d_logp = (inside || s1 < s2) ? -s1 * inv_n : 0.0f;  // the clipped branch is constant in rho
#pragma unroll
        for (int k = 0; k < kActions; ++k)
          d[k] = d_logp * ((k == action ? 1.0f : 0.0f) - p[k]) + hp.ent_coef * inv_n * p[k] * (lp[k] + ent);
        t_actor += fminf(s1, s2);
        t_ent += ent;
        const float v = hv[kActions] + bh[kActions];
        const float u = v - ret, uc = v_old + fminf(fmaxf(v - v_old, -hp.clip_eps), hp.clip_eps) - ret;
        const bool in_range = fabsf(v - v_old) <= hp.clip_eps;
        d[kActions] = (in_range || u * u > uc * uc) ? hp.vf_coef * u * inv_n : 0.0f;
        t_value += 0.5 * fmaxf(u * u, uc * uc);
      }
      // columns 0..6: the derivatives; column 7: one (it turns the d z^T products into column sums)
      sts_v4(dht + static_cast<uint32_t>((row >> 3) * (kUHeads * 16) + (row & 7) * 16), pack_bf16(d[0], d[1]), pack_bf16(d[2], d[3]),
             pack_bf16(d[4], d[5]), pack_bf16(d[6], 1.0f));
#pragma unroll
      for (int k = 0; k <= kActions; ++k) gbh[k] += d[k];  // the heads' bias gradients sum the unrounded derivatives
    }
    fence_async_smem(); tc_fence_before();
    step_barrier();
    timed_out |= !mbar_wait(bar_mma, ph_mma); ph_mma ^= 1;
    tc_fence_after();
    bwd_epilogue(gate2, dz2t);
    fence_async_smem(); tc_fence_before();
    step_barrier();
    timed_out |= !mbar_wait(bar_mma, ph_mma); ph_mma ^= 1;  // d h1 is there, and h2's last reader (d Wh) is done
    tc_fence_after();
    bwd_epilogue(gate1, dz1t);
    fence_async_smem(); tc_fence_before();
    if (step_any(timed_out)) timed_out = true;
  }
  if (timed_out) *reinterpret_cast<volatile int *>(&sm.abort) = 1;
#pragma unroll
  for (int k = 0; k <= kActions; ++k) {
    for (int o = 16; o > 0; o >>= 1) gbh[k] += __shfl_xor_sync(0xFFFFFFFFu, gbh[k], o);
    if (lane == 0 && half == 0) sm.red[warp][k] = gbh[k];
  }
  }
  // ---- the CTA's slice: accumulators out of tensor memory, once
  timed_out = __syncthreads_or(timed_out) != 0;  // (the last products have been issued)
  if (my_tiles > 0 && !timed_out) timed_out = !mbar_wait(bar_end, static_cast<uint32_t>(my_tiles - 1) & 1u);
  timed_out = __syncthreads_or(timed_out) != 0;
  if (!timed_out && my_tiles > 0 && warp < kUMain / 32) {
    tc_fence_after();
    float *part = partial + static_cast<size_t>(blockIdx.x) * kSlice;
    const int unit = (warp & 3) * 32 + lane;  // tensor-memory lane = out unit (d W2, d W1, d b) or hidden unit (d Wh)
    auto put16 = [&](float *dst, uint32_t col, int n) {  // n columns from accumulator column `col` on
      float v[16];
      tmem_ld16(tmem + lane_off + col, v);
#pragma unroll
      for (int c = 0; c < 16; c += 4)
        if (c < n) *reinterpret_cast<float4 *>(dst + (static_cast<size_t>(c / 4) * kUH + unit) * 4) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    };
    if (half == 0) {
      for (int c0 = 0; c0 < kUH; c0 += 16) put16(part + kSlW2 + c0 * kUH, kColDW2 + c0, 16);
    } else {
      for (int c0 = 0; c0 < kUK1; c0 += 16) put16(part + kSlW1 + c0 * kUH, kColDW1 + c0, 16);
      put16(part + kSlWh, kColDWh, 8);
      float v[16];
      tmem_ld16(tmem + kColDB2 + lane_off, v);
      part[kSlB2 + unit] = v[7];
      tmem_ld16(tmem + kColDB1 + lane_off, v);
      part[kSlB1 + unit] = v[7];
    }
    if (tid <= kActions) part[kSlBh + tid] = (sm.red[0][tid] + sm.red[1][tid]) + (sm.red[2][tid] + sm.red[3][tid]);
  }
  if (warp < kUMain / 32) {  // loss-term sums of the warp, lane 0 writes them (warps 4..7 hold zeros)
    double s[3] = {t_actor, t_ent, t_value};
#pragma unroll
    for (int k = 0; k < 3; ++k)
      for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], o);
    if (lane == 0) {
      double *tp = term_partial + (static_cast<size_t>(blockIdx.x) * 8 + warp) * 3;
      tp[0] = s[0]; tp[1] = s[1]; tp[2] = s[2];
    }
  }
  if (timed_out && tid == 0) atomicExch(status, kStatusTimeout);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

bool ppo_tc_supported(const mava_config_t &cfg, int D) {
  return cfg.net_kind == MAVA_NET_SHARED_TORSO && cfg.hidden <= kUH && cfg.hidden % 8 == 0 && D <= kUK1;
}

size_t ppo_tc_image_bytes() { return kImgBytes; }

size_t ppo_tc_slice_floats() { return kSlice; }

cudaError_t launch_ppo_net_tc(mava_rollout *h, const float *params_dev, const ParamLayout &L, const UpdRows &rows, const UpdHyper &hp,
                              const Moments &adv, void *image, float *partial, double *term_partial, int slices, float *grad, const TermSums &terms,
                              const Moments &norm) {
  const PrepImage prep{params_dev, static_cast<unsigned char *>(image), L, h->D, h->cfg.hidden};
  cudaError_t err = launch_prologue(adv, prep, kPrepBlocks, h->stream);
  if (err != cudaSuccess) return err;
  const size_t smem = sizeof(UtcSmem);
  const auto kern = rows_need_64_bits(rows, rows.n) ? ppo_net_tc_kernel<uint64_t> : ppo_net_tc_kernel<uint32_t>;
  err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (err != cudaSuccess) return err;
  err = launch_dependent(kern, slices, kUThreads, smem, h->stream, static_cast<const unsigned char *>(image), rows, hp,
                         static_cast<const double *>(adv.out), partial, term_partial, h->d_status, h->D, adv.early);
  if (err != cudaSuccess) return err;
  h->launches += 3;
  return launch_dependent(reduce_slices_kernel<SliceMap>, kReduceBlocks, kReduceThreads, 0, h->stream, static_cast<const float *>(partial), kSlice, slices, grad,
                          terms, norm, SliceMap{L, h->D, h->cfg.hidden});
}
cudaError_t launch_grad_moments_tc(mava_rollout *h, const ParamLayout &L, const Moments &norm) {
  return launch_dependent(grad_moments_kernel<SliceMap>, kMomentBlocks, 256, 0, h->stream, norm, kSlice, SliceMap{L, h->D, h->cfg.hidden});
}

}  // namespace mava

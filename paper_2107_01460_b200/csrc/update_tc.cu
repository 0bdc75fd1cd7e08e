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
//              d W1 += d z1^T . x, d b2 += d z2^T . 1, d b1 += d z1^T . 1 (the ones are a constant tile of 16 rows).
// Two tiles are in flight: tile s goes forward while tile s - 1 goes backward, so that one's epilogue runs beside the other's products.
// Both fit an SM because d z2 takes h2's place and d z1 h1's (behind the weight-gradient products that read them), and
// the heads' derivatives are kept once, eight columns wide.  Sixteen warps share every epilogue (32 rows x 32 columns each), eight
// bring the rows in, one issues the MMAs in a fixed order, one fetches what the loss needs.  What bounds it (10x10, 61 k rows a
// gradient): 6.7 k cycles per tile and SM against 8 k for one tile at a time.  Some 4.6 k of them are products: 30 of N = 128 at 65 cycles
// and 8 of N = 80 at 41 (2.3 k), and 32 of N = 16 that each stream a 4 KB A operand from shared memory and take 65 to 80, as long as one
// of N = 128 (24 where x has a spare column: 4.0 k).  Beside them the row of dependent epilogues (0.6 to 0.8 k each, half of it
// conversions and gate bits at half rate) and the waits between them.
// Rows: fewer than 40 KB can be on their way through the 28 KB of L1 that are left; with more loads in flight, or the look-up of a
// row in front of an epilogue, every other access of the SM stalls behind them.  Two passes of three minibatches over 549 k rows:
// 407 -> 376 us; sixteen minibatches of 33 k rows: 502 -> 478.
// The weight-gradient accumulators stay in tensor memory for all tiles of the CTA and are written once, into the CTA's
// own slice of the partial-gradient array; a last kernel adds the slices in a fixed order (reduce_slices_kernel: four quarters of
// them, each in slice order), so the gradient is the same bytes on every call.  Rounding points are those of the bf16-operand
// mode of the float64 oracle.
// A hidden width below 128 is padded with zero units (their activations, gates and gradients are exactly zero).
// MMAs are issued by one elected lane; tcgen05.commit tracks all MMAs issued before it, so a tile buffer may be rewritten as
// soon as a later commit has been waited for.  Every mbarrier wait is bounded.
#include <cuda_bf16.h>
#include <stddef.h>

#include "common.cuh"
#include "layout.h"
#include "tc_common.cuh"
#include "update_common.cuh"

namespace mava {
namespace {

constexpr int kUR = 128;        // rows per tile (M of the per-row products, K of the weight-gradient products)
constexpr int kUH = 128;        // hidden width, padded
constexpr int kUK1 = 80;        // input width, padded to the MMA's K step
constexpr int kUHeads = 16;     // N of the products with the heads: six logits, the value, a column of zeros; the other eight repeat or are not read
constexpr int kUHeadRows = 8;   // of which these exist in memory
constexpr int kUMain = 512;     // threads of the epilogues: a warp has 32 rows x 32 columns of a tile
constexpr int kLossWarps = 8;   // of which these also do the loss: four the actor's part, four the value's, a row per thread
constexpr int kULoaders = 8;    // warps that bring the rows in, 16 rows each
constexpr int kUThreads = kUMain + 32 * kULoaders + 128;  // and a warpgroup: one warp issues the MMAs, one fetches what the loss needs

// weight image: fp32 b1 [H], b2 [H], bh [8]; then bf16 tiles W1 [H][K1], Wh [8][H], W2 [H][H] (the heads as an N = 16 operand: what lies
// behind them gives columns that nobody reads)
constexpr uint32_t kImgB1 = 0, kImgB2 = kImgB1 + kUH * 4, kImgBh = kImgB2 + kUH * 4, kImgW1 = kImgBh + 32;
constexpr uint32_t kImgWh = kImgW1 + kUH * kUK1 * 2, kImgW2 = kImgWh + kUHeadRows * kUH * 2, kImgBytes = kImgW2 + kUH * kUH * 2;
static_assert(kImgBytes % 16 == 0 && kImgWh % 16 == 0, "bulk copies");

// tensor-memory columns: an accumulator per tile in flight, used by z1, z2, the heads, d h2 and d h1 in turn; the weight gradients
constexpr uint32_t kColAcc = 0, kColDW2 = 256, kColDW1 = 384, kColDWh = 464, kColDB2 = 480, kColDB1 = 496;
constexpr uint32_t kTmemCols = 512;

// The x tile is [feature chunk][row], 16 bytes more than the rows need from chunk to chunk: the loaders' stores (lane = two
// features) then spread over the banks.
constexpr uint32_t kXChunk = kUR * 16 + 16, kXTile = (kUK1 / 8) * kXChunk;
constexpr uint32_t kHTile = kUR * kUH * 2;
// At the end, in W2's place (its last reader is done): sums over the CTA's rows of the heads' bias gradients and of the loss terms
struct UtcSums { double term[4][3]; float bias[4][8]; };

// Products that an epilogue waits for, and epilogues that a product waits for: a barrier each, one phase per tile.
enum { kZ1, kZ2, kLogits, kDh2, kDWh, kDh1, kDW2, kProducts };
enum { kH1, kH2, kLoss, kDz2, kDz1, kEpilogues };

struct UtcSmem {  // two tiles are in flight, an even and an odd one
  alignas(128) unsigned char h1[2][kHTile];  // d z1 once d W2 has read h1
  alignas(128) unsigned char h2[2][kHTile];  // d z2 once d Wh has read h2
  alignas(128) unsigned char x[2][kXTile];
  alignas(128) unsigned char dhead[kUR * kUHeadRows * 2];  // of either tile: one's last reader is done before the other's loss
  alignas(128) unsigned char img[kImgBytes];
  // what the loss needs of a tile's rows (the old log-probs and advantages take the place of the biases, which are in registers by then)
  float value_old[kUR], ret[kUR];
  unsigned char action[kUR];  // 0xFF: no such row
  alignas(16) unsigned char ones[16 * kUHeadRows * 2];  // bf16 ones, the rows of a K step: operand of the column sums, never rewritten
  alignas(8) uint64_t bar_load[2], done[kProducts], ready[kEpilogues], x_full[2], x_empty[2], rows_full, bar_end;
  uint32_t tmem_base;
  int abort;  // a warp gave up
};
static_assert(sizeof(UtcSmem) <= 232448, "shared memory of a block");

struct PrepImage {
  const float *params;
  unsigned char *image;
  ParamLayout L;
  int D, H;
  // Element i of the image: its parameter (if there is one; every parameter has one place in the image) and where it lies.
  struct Place { size_t param; uint32_t at; bool real, wide /* fp32 instead of bf16 */; };
  __device__ Place place(int i) const;
  __device__ void put(const Place &p, float v) const {
    if (p.wide) *reinterpret_cast<float *>(image + p.at) = v;
    else *reinterpret_cast<__nv_bfloat16 *>(image + p.at) = __float2bfloat16_rn(v);
  }
  __device__ void operator()(int tid, int nth) const;
};
// One element per thread: a kernel that everything behind it waits for (as loops over the parts with 8 k threads it took 3 us more).
constexpr int kPrepW1 = kUH * kUK1, kPrepW2 = kUH * kUH, kPrepWh = kUHeadRows * kUH, kPrepTotal = kPrepW1 + kPrepW2 + kPrepWh + 2 * kUH + 8;
constexpr int kPrepBlocks = (kPrepTotal + 255) / 256;
__device__ __forceinline__ PrepImage::Place PrepImage::place(int j) const {
  if (j < kPrepW1) {
    const int n = j / kUK1, k = j - n * kUK1;
    return Place{L.W1 + static_cast<size_t>(n) * D + k, kImgW1 + canon_offset(n, k, kUK1), n < H && k < D, false};
  }
  if ((j -= kPrepW1) < kPrepW2) {
    const int n = j / kUH, k = j - n * kUH;
    return Place{L.W2 + static_cast<size_t>(n) * H + k, kImgW2 + canon_offset(n, k, kUH), n < H && k < H, false};
  }
  if ((j -= kPrepW2) < kPrepWh) {
    const int n = j / kUH, k = j - n * kUH;
    return Place{n < kActions ? L.Wa + static_cast<size_t>(n) * H + k : L.Wv + k, kImgWh + canon_offset(n, k, kUH), k < H && n <= kActions, false};
  }
  if ((j -= kPrepWh) < 2 * kUH) {
    const int n = j % kUH;
    return Place{(j < kUH ? L.b1 : L.b2) + n, (j < kUH ? kImgB1 : kImgB2) + 4 * n, n < H, true};
  }
  j -= 2 * kUH;
  return Place{j < kActions ? L.ba + j : L.bv, kImgBh + 4 * j, j <= kActions, true};
}
__device__ __forceinline__ void PrepImage::operator()(int tid, int nth) const {
  for (int i = tid; i < kPrepTotal; i += nth) {
    const Place p = place(i);
    put(p, p.real ? __ldcg(params + p.param) : 0.0f);
  }
}

// An optimiser step that leaves the next gradient its weight image and, by blocks of their own while the kernels in front still run,
// its advantages' moments.  Everything but the gradient is read before the wait: what was launched before the gradient in front is
// complete when this starts (launch_ppo_grad), the step before this one too.
__global__ void __launch_bounds__(256) step_image_kernel(AdamArgs adam, PrepImage prep, Moments next) {
  dependents_may_start();
  if (static_cast<int>(blockIdx.x) < kMomentBlocks) {
    moments_block<uint32_t>(next);  // (at most n_envs environments: no more rows than the trajectory has, below 2^32 in any memory)
    wait_for_predecessor();
    return;
  }
  const int i = (static_cast<int>(blockIdx.x) - kMomentBlocks) * 256 + static_cast<int>(threadIdx.x);
  PrepImage::Place p{0, 0, false, false};
  if (i < kPrepTotal) p = prep.place(i);
  AdamState state{0.0f, 0.0f, 0.0f};
  if (p.real) state = adam_load(adam, p.param);
  wait_for_predecessor();
  const float grad = p.real ? __ldcg(adam.grad + p.param) : 0.0f, scale = adam_scale(adam);
  if (i < kPrepTotal) prep.put(p, p.real ? adam_element(adam, state, grad, scale, p.param) : 0.0f);
}

// A canonical tile of C features read with the feature index as K: chunks (K groups) 128 bytes apart, 8-row groups C*16.  The same tile
// read with the row index as K: the 8-row groups are the K groups, the feature chunks the MN groups, so the descriptor's
// leading-dimension offset is C*16 and its stride offset 128.
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;  // operand is MN-major
// A descriptor from an address in 16-byte units: one addition to a word that is otherwise constant (14 bits hold any address of a block).
template <uint32_t LBO, uint32_t SBO>
__device__ __forceinline__ uint64_t desc16(uint32_t addr16) {
  constexpr uint32_t lo = (LBO >> 4) << 16;
  constexpr uint64_t hi = (static_cast<uint64_t>(SBO >> 4) << 32) | (1ull << 46);
  return hi | (addr16 + lo);
}

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

constexpr int kLoadRows = kUR / kULoaders;  // per loader warp, all of their loads in flight at once

__device__ __forceinline__ void prefetch_l2(const float *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void tmem_ld_row8(uint32_t taddr, float *v) {  // thread = lane
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    asm volatile("" : "+r"(r[i]));
    v[i] = __uint_as_float(r[i]);
  }
}
// Waits for the tensor-memory loads; what they brought is not touched before.
__device__ __forceinline__ void tmem_ld_wait32(uint32_t *r) {
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(r[i]));
}

template <class U>  // row numbers of the batch (real_row)
__global__ void __launch_bounds__(kUThreads, 1)
ppo_net_tc_kernel(const unsigned char *image, UpdRows rows, UpdHyper hp, const double *adv_stats,
                  float *partial, double *term_partial, int *status, int D, int H, bool rows_ready, int debug_expire) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  UtcSmem &sm = *reinterpret_cast<UtcSmem *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);  // (uniform to the compiler)
  const int wq = warp & 3, cq = (warp >> 2) & 3;  // of an epilogue warp: its rows (32, = tensor-memory lanes) and columns (32)
  const uint32_t bar_load = smem_u32(&sm.bar_load[0]), done0 = smem_u32(&sm.done[0]), ready0 = smem_u32(&sm.ready[0]), x_full0 = smem_u32(&sm.x_full[0]),
                 x_empty0 = smem_u32(&sm.x_empty[0]), rows_full = smem_u32(&sm.rows_full), bar_end = smem_u32(&sm.bar_end);
  if (tid == 0) {
    sm.abort = 0;
    for (uint32_t i = 0; i < 2; ++i) { mbar_init(bar_load + 8 * i, 1); mbar_init(x_full0 + 8 * i, kULoaders); mbar_init(x_empty0 + 8 * i, 1); }
    for (uint32_t i = 0; i < kProducts; ++i) mbar_init(done0 + 8 * i, 1);
    for (uint32_t i = 0; i < kEpilogues; ++i) mbar_init(ready0 + 8 * i, i == kLoss ? kLossWarps : kUMain / 32);
    mbar_init(rows_full, 1); mbar_init(bar_end, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid < static_cast<int>(sizeof(sm.ones) / 4)) {
    sts_u32(smem_u32(sm.ones) + 4u * static_cast<uint32_t>(tid), 0x3F803F80u);
    fence_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // What fetches rows needs neither the weights nor the moments: the first tile's come while both are on their way.
  const bool loader = warp >= kUMain / 32 && warp < kUMain / 32 + kULoaders;
  const bool fetches = loader || warp == kUMain / 32 + kULoaders + 1;
  if (!fetches || !rows_ready) wait_for_predecessor();
  if (!fetches) dependents_may_start();  // (after the wait: launch_ppo_grad)
  if (tid == 0) {  // the first layer's weights and the biases, then the rest
    constexpr uint32_t kChunk = 16384;
    mbar_expect_tx(bar_load, kImgWh);
    for (uint32_t o = 0; o < kImgWh; o += kChunk) bulk_load(smem_u32(sm.img + o), image + o, min(kChunk, kImgWh - o), bar_load);
    mbar_expect_tx(bar_load + 8, kImgBytes - kImgWh);
    for (uint32_t o = kImgWh; o < kImgBytes; o += kChunk) bulk_load(smem_u32(sm.img + o), image + o, min(kChunk, kImgBytes - o), bar_load + 8);
  }

  const uint32_t tmem = sm.tmem_base;
  const uint32_t lane_off = static_cast<uint32_t>(wq * 32) << 16;
  const uint32_t h1t = smem_u32(sm.h1[0]), h2t = smem_u32(sm.h2[0]), xt0 = smem_u32(sm.x[0]), dht = smem_u32(sm.dhead);
  const long long n_tiles = (rows.n + kUR - 1) / kUR;
  const int my_tiles = blockIdx.x < n_tiles ? static_cast<int>((n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
  auto tile_of = [&](int i) { return static_cast<long long>(blockIdx.x) + static_cast<long long>(i) * gridDim.x; };
  volatile int *abort_flag = &sm.abort;
  bool ok = true;

  if (loader) {
    // ---- the rows.  A tile's rows are in registers (as bf16) before its x tile is free, which is late: d W1 of the tile two before, the
    // last of its products, reads it.  A lane has two neighbouring columns (one 4-byte store) below 64, and two of the sixteen
    // above of every fourth row; the second load of a pair finds its sectors in L1.
    const int lw = warp - kUMain / 32, sub = lane >> 3, c2 = 64 + 2 * (lane & 7);
    const bool has0 = c2 < D, has1 = c2 + 1 < D;
    const float pad0 = c2 == D ? 1.0f : 0.0f, pad1 = c2 + 1 == D ? 1.0f : 0.0f;  // a spare column holds ones (d b1)
    auto row_of = [&](int i) {
      const long long q = tile_of(i) * kUR + kLoadRows * lw + lane;
      return row_lookup<U>(rows, q, lane < kLoadRows && i < my_tiles && q < rows.n);
    };
    RowLookup next = row_of(0);
    for (int i = 0; i < my_tiles && ok; ++i) {
      const int src = row_found(rows, next);
      next = row_of(i + 1);
      float v[kLoadRows][2], t[kLoadRows / 4][2];
#pragma unroll
      for (int r = 0; r < kLoadRows; ++r) {
        const int s = __shfl_sync(0xFFFFFFFFu, src, r);
        const float *p = rows.x + static_cast<long long>(s) * D + 2 * lane;
        v[r][0] = ldg_if_cached(p, s >= 0);  // (D > 64: these are columns of every row)
        v[r][1] = ldg_if_cached(p + 1, s >= 0);
        if ((r & 3) == 0) {
          const int s4 = __shfl_sync(0xFFFFFFFFu, src, r + sub);
          const float *p4 = rows.x + static_cast<long long>(s4) * D + c2;
          t[r / 4][0] = ldg_if_cached(p4, s4 >= 0 && has0);
          t[r / 4][1] = ldg_if_cached(p4 + 1, s4 >= 0 && has1);
        }
      }
      const int ahead = row_found(rows, next);
      if (ahead >= 0) {  // into L2 (D > 64: the row's first, middle and last lines)
        const float *p = rows.x + static_cast<long long>(ahead) * D;
        prefetch_l2(p); prefetch_l2(p + 32); prefetch_l2(p + 64); prefetch_l2(p + D - 1);
      }
      uint32_t pk[kLoadRows], pt[kLoadRows / 4];
#pragma unroll
      for (int r = 0; r < kLoadRows; ++r) pk[r] = pack_bf16(v[r][0], v[r][1]);
#pragma unroll
      for (int r = 0; r < kLoadRows / 4; ++r) pt[r] = pack_bf16(has0 ? t[r][0] : pad0, has1 ? t[r][1] : pad1);
      if (i >= 2) ok = ok && mbar_sleep_warp(x_empty0 + 8u * (i & 1), static_cast<uint32_t>((i >> 1) - 1) & 1u);
      if (!ok || *abort_flag) break;
      const uint32_t xt = xt0 + kXTile * static_cast<uint32_t>(i & 1) + 16u * static_cast<uint32_t>(kLoadRows * lw);
      const uint32_t at = xt + static_cast<uint32_t>(lane >> 2) * kXChunk + (lane & 3) * 4;
      const uint32_t at4 = xt + static_cast<uint32_t>(8 + ((lane & 7) >> 2)) * kXChunk + (lane & 3) * 4 + 16u * static_cast<uint32_t>(sub);
#pragma unroll
      for (int r = 0; r < kLoadRows; ++r) {
        sts_u32(at + 16u * r, pk[r]);
        if ((r & 3) == 0) sts_u32(at4 + 16u * r, pt[r / 4]);  // (behind column D: zeros)
      }
      fence_async_smem();
      warp_arrive(x_full0 + 8u * (i & 1), lane);
    }
  } else if (warp >= kUMain / 32 + kULoaders) {
    if (warp == kUMain / 32 + kULoaders) {
    // ---- the MMAs: tile s goes forward while tile s - 1 goes backward.  The products that only a weight gradient needs are behind
    // those that a chain waits for.  tcgen05.commit covers everything issued before it, so who has waited for a later product
    // knows that the earlier ones have read their tiles.  The order of the products is fixed, so that of every sum is.
    auto handed_over = [&](int what, int tile) {
      ok = ok && mbar_sleep_warp(ready0 + 8u * what, static_cast<uint32_t>(tile) & 1u);
      tc_fence_after();
    };
    constexpr uint32_t kFwd = instr_desc(kUR, kUH), kHead = instr_desc(kUR, kUHeads), kGrad = kAmn | kBmn;
    // operands of step k (16 features or rows), `at` = the tile's address in 16-byte units
    auto act_k = [](uint32_t at, int k) { return desc16<128, kUH * 16>(at + k * 16); };              // activations, feature as K
    auto act_mn = [](uint32_t at, int k) { return desc16<kUH * 16, 128>(at + k * 2 * kUH); };        // row as K
    auto dh_mn = [](uint32_t at, int k) { return desc16<128, 0>(at + k * 16); };                     // dhead, row as K, its columns twice
    auto ones_mn = [](uint32_t at) { return desc16<128, 0>(at); };                                   // the same rows of ones for every step
    constexpr uint32_t kX16 = kXTile / 16, kH16 = kHTile / 16;
    const uint32_t block16 = smem_u32(&sm) >> 4;
    uint32_t base = block16;
    // not a loop invariant to the compiler: it would keep every product's descriptors in registers that it does not have
    auto fresh = [&]() { asm volatile("mov.u32 %0, %1;" : "=r"(base) : "r"(block16)); };
#define AT16(member) (base + static_cast<uint32_t>(offsetof(UtcSmem, member) / 16))
#define IMG16(off) (base + static_cast<uint32_t>((offsetof(UtcSmem, img) + (off)) / 16))
    ok = mbar_sleep_warp(bar_load, 0);
    if (debug_expire && blockIdx.x == 0) ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar_end, 0, 1u << 12)) != 0;  // (nothing completes this phase before the end)
#pragma unroll 1
    for (int s = 0; s <= my_tiles && ok; ++s) {
      const bool fwd = s < my_tiles, bwd = s > 0;
      const int pf = s & 1, pb = pf ^ 1;
      const uint32_t accf = tmem + kColAcc + 128u * pf, accb = tmem + kColAcc + 128u * pb;
      const uint32_t hf = kH16 * pf, hb = kH16 * pb, xf = kX16 * pf, xb = kX16 * pb;
      const uint32_t keep = s > 1 ? 1u : 0u;  // the weight-gradient accumulators start at the CTA's first tile
      if (bwd) {
        handed_over(kLoss, s - 1);
        fresh();
        if (ok && elect_one()) {
          // d h2 = dhead . Wh: K = 16 is the eight columns of either operand twice (step 0 from one to the other half), so dhead
          // is kept at half its size
          mma_bf16(accb, desc16<0, 128>(AT16(dhead)), desc16<0, 128>(IMG16(kImgWh)), kFwd | kBmn, 0);
          mma_commit(done0 + 8 * kDh2);
          // d Wh^T [unit][head column] += h2^T . dhead (K = rows)
#pragma unroll
          for (int k = 0; k < kUR / 16; ++k)
            mma_bf16(tmem + kColDWh, act_mn(AT16(h2) + hb, k), dh_mn(AT16(dhead), k), instr_desc(kUH, kUHeads) | kGrad, keep | (k > 0));
          mma_commit(done0 + 8 * kDWh);  // (d z2 takes h2's place)
        }
        __syncwarp();
      }
      if (fwd) {
        ok = ok && mbar_sleep_warp(x_full0 + 8u * pf, static_cast<uint32_t>(s >> 1) & 1u);
        tc_fence_after();
        fresh();
        if (ok && elect_one()) {  // z1
#pragma unroll
          for (int k = 0; k < kUK1 / 16; ++k)
            mma_bf16(accf, desc16<kXChunk, 128>(AT16(x) + xf + k * (2 * kXChunk / 16)), desc16<128, kUK1 * 16>(IMG16(kImgW1) + k * 16), kFwd, k > 0);
          mma_commit(done0 + 8 * kZ1);
        }
        __syncwarp();
        if (s == 0) ok = ok && mbar_sleep_warp(bar_load + 8, 0);
      }
      if (bwd) {
        handed_over(kDz2, s - 1);
        fresh();
        if (ok && elect_one()) {
          // d h1 = d z2 . W2 (K = the out units of layer 2)
#pragma unroll
          for (int k = 0; k < kUH / 16; ++k) mma_bf16(accb, act_k(AT16(h2) + hb, k), act_mn(IMG16(kImgW2), k), kFwd | kBmn, k > 0);
          mma_commit(done0 + 8 * kDh1);
          // d W2 [out][in] += d z2^T . h1 (K = rows)
#pragma unroll
          for (int k = 0; k < kUR / 16; ++k)
            mma_bf16(tmem + kColDW2, act_mn(AT16(h2) + hb, k), act_mn(AT16(h1) + hb, k), kFwd | kGrad, keep | (k > 0));
          mma_commit(done0 + 8 * kDW2);  // (d z1 takes h1's place)
        }
        __syncwarp();
      }
      if (fwd) {
        handed_over(kH1, s);
        fresh();
        if (ok && elect_one()) {  // z2
#pragma unroll
          for (int k = 0; k < kUH / 16; ++k) mma_bf16(accf, act_k(AT16(h1) + hf, k), act_k(IMG16(kImgW2), k), kFwd, k > 0);
          mma_commit(done0 + 8 * kZ2);
        }
        __syncwarp();
      }
      if (bwd) {
        fresh();
        if (ok && elect_one()) {  // d b2 [out] += d z2^T . ones
#pragma unroll
          for (int k = 0; k < kUR / 16; ++k)
            mma_bf16(tmem + kColDB2, act_mn(AT16(h2) + hb, k), ones_mn(AT16(ones)), instr_desc(kUH, kUHeads) | kGrad, keep | (k > 0));
        }
        __syncwarp();
        handed_over(kDz1, s - 1);
        fresh();
        if (ok && elect_one()) {  // d W1 [out][in] += d z1^T . x
#pragma unroll
          for (int k = 0; k < kUR / 16; ++k)
            mma_bf16(tmem + kColDW1, act_mn(AT16(h1) + hb, k), desc16<128, kXChunk>(AT16(x) + xb + k * 16), instr_desc(kUH, kUK1) | kGrad, keep | (k > 0));
          mma_commit(x_empty0 + 8u * pb);
        }
        __syncwarp();
      }
      if (fwd) {
        handed_over(kH2, s);
        fresh();
        if (ok && elect_one()) {  // heads
#pragma unroll
          for (int k = 0; k < kUH / 16; ++k) mma_bf16(accf, act_k(AT16(h2) + hf, k), act_k(IMG16(kImgWh), k), kHead, k > 0);
          mma_commit(done0 + 8 * kLogits);
        }
        __syncwarp();
      }
      if (bwd) {
        fresh();
        if (D == kUK1 && ok && elect_one()) {  // d b1 [out] += d z1^T . ones (otherwise a column of d W1)
#pragma unroll
          for (int k = 0; k < kUR / 16; ++k)
            mma_bf16(tmem + kColDB1, act_mn(AT16(h1) + hb, k), ones_mn(AT16(ones)), instr_desc(kUH, kUHeads) | kGrad, keep | (k > 0));
        }
        __syncwarp();
      }
    }
#undef AT16
#undef IMG16
    if (elect_one()) mma_commit(bar_end);  // covers every MMA issued, after a time-out too
    __syncwarp();
    } else if (warp == kUMain / 32 + kULoaders + 1) {
      // ---- what the loss needs of the rows, four rows per lane.  The place for it is free once the loss of the tile before, or the first
      // tile's first epilogue (it has the biases), is done.
      float *logp_old = reinterpret_cast<float *>(sm.img + kImgB1), *adv = reinterpret_cast<float *>(sm.img + kImgB2);
      auto row_of = [&](int i, int k) {
        const long long q = tile_of(i) * kUR + 32 * k + lane;
        return row_lookup<U>(rows, q, i < my_tiles && q < rows.n);
      };
      RowLookup next[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) next[k] = row_of(0, k);
#pragma unroll 1
      for (int i = 0; i < my_tiles && ok; ++i) {
        float v[4][5];
        bool real[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int src = row_found(rows, next[k]);
          real[k] = src >= 0;
          v[k][0] = ldg_if(rows.logp_old + src, real[k]); v[k][1] = ldg_if(rows.adv + src, real[k]);
          v[k][2] = ldg_if(rows.value_old + static_cast<long long>(src) * rows.vstride, real[k]);
          v[k][3] = ldg_if(rows.ret + static_cast<long long>(src) * rows.vstride, real[k]);
          v[k][4] = ldg_if(reinterpret_cast<const float *>(rows.actions) + src, real[k]);
          if (!real[k] && tile_of(i) * kUR + 32 * k + lane < rows.n) atomicExch(status, kStatusBadIndex);
          next[k] = row_of(i + 1, k);
        }
        ok = i == 0 ? mbar_sleep_warp(ready0 + 8 * kH1, 0) : mbar_sleep_warp(ready0 + 8 * kLoss, static_cast<uint32_t>(i - 1) & 1u);
        if (!ok) break;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int r = 32 * k + lane, a = __float_as_int(v[k][4]);
          logp_old[r] = v[k][0]; adv[r] = v[k][1]; sm.value_old[r] = v[k][2]; sm.ret[r] = v[k][3];
          sm.action[r] = static_cast<unsigned char>(real[k] ? (a >= 0 && a < kActions ? a : 0xFE) : 0xFF);
        }
        warp_arrive(rows_full, lane);
      }
    }
  } else {
    // ---- the epilogues, every warp its part of either tile's: while the products of one are under way, the other's turn
    const uint32_t acc0 = tmem + kColAcc + lane_off;
    // where stmatrix4 puts the matrices (row group, chunk), (+1, chunk), (row group, +1), (+1, +1) of this warp's rows and columns
    const uint32_t my_at = static_cast<uint32_t>((wq * 4 + ((lane >> 3) & 1)) * (kUH * 16) + (cq * 4 + (lane >> 4)) * 128 + (lane & 7) * 16);
    const float mean = static_cast<float>(__ldcg(adv_stats));
    const float inv_std = 1.0f / (static_cast<float>(__ldcg(adv_stats + 1)) + 1e-8f);
    const float inv_n = 1.0f / static_cast<float>(rows.n);
    const bool is_actor = cq == 0, is_value = cq == 1;  // this warp's part of the loss
    double t0 = 0.0, t1 = 0.0;  // surrogate and entropy, or value
    float gbh[kActions];        // gradient of the heads' biases, this thread's rows (value: [0])
#pragma unroll
    for (int k = 0; k < kActions; ++k) gbh[k] = 0.0f;
    auto product = [&](int what, int tile) { ok = ok && mbar_sleep_warp(done0 + 8u * what, static_cast<uint32_t>(tile) & 1u); tc_fence_after(); };
    auto hand_over = [&](int what) { fence_async_smem(); tc_fence_before(); warp_arrive(ready0 + 8u * what, lane); };
    // this warp's 32 x 32 accumulators of tile parity p
    auto load_acc = [&](int p, uint32_t (&r)[32]) {
      const uint32_t at = acc0 + 128u * p + 32u * cq;
      tmem_ld_16x32_nowait(at, r);
      tmem_ld_16x32_nowait(at + (16u << 16), r + 16);
      tmem_ld_wait32(r);
    };
    auto store = [&](uint32_t tile, const uint32_t *pk) {
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int j = 0; j < 4; j += 2)
          stmatrix4(tile + my_at + static_cast<uint32_t>(c * 2 * kUH * 16 + j * 128), pk + 8 * c + 2 * j);
    };
    // hidden-layer epilogue: + bias -> ReLU -> bf16 -> `tile`; one gate bit per unit out (pair i: bits 15 - i and 31 - i).  Two
    // columns per instruction throughout.
    auto fwd_epilogue = [&](int p, const float2 *bias, uint32_t tile) {
      uint32_t r[32], pk[16], gate[2] = {0, 0};
      load_acc(p, r);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float2 b = bias[(i & 7) >> 1];
        add2(r[2 * i], r[2 * i + 1], b.x, b.y);
        pk[i] = relu_pack_bf16(r[2 * i], r[2 * i + 1]);
        gate[i & 1] |= positive_mask(pk[i]) & (0x80008000u >> i);
      }
      store(tile, pk);
      return gate[0] | gate[1];
    };
    // backward epilogue: d h (accumulator) gated by the layer's ReLU, as bf16 pairs
    auto bwd_epilogue = [&](int p, uint32_t gate, uint32_t *pk) {
      uint32_t r[32];
      load_acc(p, r);
#pragma unroll
      for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])) & sign_mask(gate << i);
    };
    ok = mbar_sleep_warp(bar_load, 0);
    float2 b1[4], b2[4];
    {
      const float *src = reinterpret_cast<const float *>(sm.img) + 32 * cq + 2 * (lane & 3);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        b1[j] = *reinterpret_cast<const float2 *>(src + kImgB1 / 4 + 8 * j);
        b2[j] = *reinterpret_cast<const float2 *>(src + kImgB2 / 4 + 8 * j);
      }
    }
    const float *bh = reinterpret_cast<const float *>(sm.img + kImgBh);
    uint32_t gate1 = 0, gate2 = 0;
#pragma unroll 1
    for (int s = 0; s <= my_tiles && ok; ++s) {
      const bool fwd = s < my_tiles, bwd = s > 0;
      const int pf = s & 1, pb = pf ^ 1;
      if (bwd) {  // d z2
        uint32_t pk[16];
        product(kDh2, s - 1);
        bwd_epilogue(pb, gate2, pk);
        product(kDWh, s - 1);
        store(h2t + kHTile * pb, pk);
        hand_over(kDz2);
      }
      const uint32_t gate1_b = gate1;
      if (fwd) {
        product(kZ1, s);
        gate1 = fwd_epilogue(pf, b1, h1t + kHTile * pf);
        hand_over(kH1);
      }
      if (bwd) {  // d z1
        uint32_t pk[16];
        product(kDh1, s - 1);
        bwd_epilogue(pb, gate1_b, pk);
        product(kDW2, s - 1);
        store(h1t + kHTile * pb, pk);
        hand_over(kDz1);
      }
      if (fwd) {
        product(kZ2, s);
        gate2 = fwd_epilogue(pf, b2, h2t + kHTile * pf);
        hand_over(kH2);
      }
      if (fwd && (is_actor || is_value)) ok = ok && mbar_sleep_warp(rows_full, static_cast<uint32_t>(s) & 1u);
      const int row = 32 * wq + lane, action = sm.action[row];
      const bool real = action != 0xFF;
      // loss terms and the per-row derivatives with respect to the six logits and the value.  dhead: columns 0..6 the derivatives at
      // half their size; column 7: zero
      if (fwd && is_actor) {
        product(kLogits, s);
        const float in0 = reinterpret_cast<const float *>(sm.img + kImgB1)[row], in1 = reinterpret_cast<const float *>(sm.img + kImgB2)[row];
        float l[8], p[kActions], d[kActions], m = -INFINITY, sum = 0.0f;
        tmem_ld_row8(acc0 + 128u * pf, l);
#pragma unroll
        for (int k = 0; k < kActions; ++k) { l[k] += bh[k]; m = fmaxf(m, l[k]); }
#pragma unroll
        for (int k = 0; k < kActions; ++k) sum += expf(l[k] - m);
        const float lse = m + logf(sum);
        float ent = 0.0f, lpa = 0.0f;
#pragma unroll
        for (int k = 0; k < kActions; ++k) {
          l[k] -= lse; p[k] = expf(l[k]); ent -= p[k] * l[k];
          if (k == action) lpa = l[k];
        }
        const float rho = expf(lpa - in0);
        const float ahat = (in1 - mean) * inv_std;
        const float clipped = fminf(fmaxf(rho, 1.0f - hp.clip_eps), 1.0f + hp.clip_eps);
        const float s1 = rho * ahat, s2 = clipped * ahat;
        const bool inside = rho >= 1.0f - hp.clip_eps && rho <= 1.0f + hp.clip_eps;
        const float d_logp = (inside || s1 < s2) ? -s1 * inv_n : 0.0f;  // the clipped branch is constant in rho
#pragma unroll
        for (int k = 0; k < kActions; ++k) {
          d[k] = d_logp * ((k == action ? 1.0f : 0.0f) - p[k]) + hp.ent_coef * inv_n * p[k] * (l[k] + ent);
          if (!real) d[k] = 0.0f;
        }
        const uint32_t at = dht + 16u * static_cast<uint32_t>(row);
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at), "r"(pack_bf16(0.5f * d[0], 0.5f * d[1])), "r"(pack_bf16(0.5f * d[2], 0.5f * d[3])) : "memory");
        sts_u32(at + 8u, pack_bf16(0.5f * d[4], 0.5f * d[5]));
        hand_over(kLoss);
#pragma unroll
        for (int k = 0; k < kActions; ++k) gbh[k] += d[k];  // (unrounded)
        if (real) { t0 += fminf(s1, s2); t1 += ent; }
      }
      if (fwd && is_value) {
        product(kLogits, s);
        const float in0 = sm.value_old[row], in1 = sm.ret[row];
        float l[8], d = 0.0f;
        tmem_ld_row8(acc0 + 128u * pf, l);
        if (real) {
          const float v = l[kActions] + bh[kActions], u = v - in1, uc = in0 + fminf(fmaxf(v - in0, -hp.clip_eps), hp.clip_eps) - in1;
          const bool in_range = fabsf(v - in0) <= hp.clip_eps;
          d = (in_range || u * u > uc * uc) ? hp.vf_coef * u * inv_n : 0.0f;
          t0 += 0.5 * fmaxf(u * u, uc * uc);
        }
        sts_u32(dht + 16u * static_cast<uint32_t>(row) + 12u, pack_bf16(0.5f * d, 0.0f));
        hand_over(kLoss);
        gbh[0] += d;
      }
    }
    if (is_actor || is_value) {
      UtcSums &sums = *reinterpret_cast<UtcSums *>(sm.img + kImgW2);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < kActions; ++k) gbh[k] += __shfl_xor_sync(0xFFFFFFFFu, gbh[k], o);
        t0 += __shfl_xor_sync(0xFFFFFFFFu, t0, o); t1 += __shfl_xor_sync(0xFFFFFFFFu, t1, o);
      }
      if (lane == 0 && is_actor) {
#pragma unroll
        for (int k = 0; k < kActions; ++k) sums.bias[wq][k] = gbh[k];
        sums.term[wq][0] = t0; sums.term[wq][1] = t1;
      }
      if (lane == 0 && is_value) { sums.bias[wq][kActions] = gbh[0]; sums.term[wq][2] = t0; }
    }
  }
  // ---- the CTA's slice: accumulators out of tensor memory, once (what belongs to real units)
  if (!ok) *abort_flag = 1;
  ok = __syncthreads_and(ok) != 0;  // (the last products have been issued)
  if (!ok) { mbar_wait(bar_load, 0); mbar_wait(bar_load + 8, 0); }  // who gave up may not have waited for the whole image: the copies land first
  ok &= mbar_wait(bar_end, 0);
  ok = __syncthreads_and(ok) != 0;
  const UtcSums &sums = *reinterpret_cast<const UtcSums *>(sm.img + kImgW2);
  if (ok && my_tiles > 0 && warp < kUMain / 32) {
    tc_fence_after();
    float *part = partial + static_cast<size_t>(blockIdx.x) * kSlice;
    const int unit = 32 * wq + lane;  // tensor-memory lane = out unit (d W2, d W1, d b) or hidden unit (d Wh)
    auto put = [&](float *dst, const uint32_t *v, int n, float scale) {  // n columns
      if (unit < H)
#pragma unroll
        for (int c = 0; c < n; c += 4)
          *reinterpret_cast<float4 *>(dst + (static_cast<size_t>(c / 4) * kUH + unit) * 4) =
              make_float4(scale * __uint_as_float(v[c]), scale * __uint_as_float(v[c + 1]), scale * __uint_as_float(v[c + 2]), scale * __uint_as_float(v[c + 3]));
    };
    uint32_t v[32];
    const uint32_t from = tmem + lane_off;
    if (cq < 3) {  // 32 columns of d W2 (0, 32, 96 ..) and those of d W1 from 0, 32, 64 on
      if (cq < 2 || H > 96) {
        const int c0 = cq < 2 ? 32 * cq : 96;
        if (c0 < H) {
          tmem_ld32_nowait(from + kColDW2 + c0, v);
          tmem_ld_wait32(v);
          put(part + kSlW2 + c0 * kUH, v, 32, 1.0f);
        }
      }
      tmem_ld32_nowait(from + kColDW1 + (cq < 2 ? 32 * cq : 48), v);
      tmem_ld_wait32(v);
      if (cq < 2) put(part + kSlW1 + 32 * cq * kUH, v, 32, 1.0f);
      else put(part + kSlW1 + 64 * kUH, v + 16, 16, 1.0f);
    } else {
      if (64 < H) {
        tmem_ld32_nowait(from + kColDW2 + 64, v);
        tmem_ld_wait32(v);
        put(part + kSlW2 + 64 * kUH, v, 32, 1.0f);
      }
      float w[16];
      tmem_ld16(from + kColDWh, w);
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = __float_as_uint(w[c]);
      put(part + kSlWh, v, 8, 2.0f);  // (dhead at half its size)
      tmem_ld16(from + kColDB2, w);
      if (unit < H) part[kSlB2 + unit] = w[0];
      uint32_t db1;
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(db1) : "r"(from + (D == kUK1 ? kColDB1 : kColDW1 + static_cast<uint32_t>(D))) : "memory");
      tmem_ld_wait();
      asm volatile("" : "+r"(db1));
      if (unit < H) part[kSlB1 + unit] = __uint_as_float(db1);
    }
    if (tid <= kActions) part[kSlBh + tid] = (sums.bias[0][tid] + sums.bias[1][tid]) + (sums.bias[2][tid] + sums.bias[3][tid]);
  }
  if (tid < 12) term_partial[static_cast<size_t>(blockIdx.x) * 12 + tid] = (&sums.term[0][0])[tid];
  if (!ok && tid == 0) atomicExch(status, kStatusTimeout);
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
                              const Moments &adv, bool prepared, void *image, float *partial, double *term_partial, int slices, float *grad,
                              const TermSums &terms, double *squares) {
  cudaError_t err = cudaSuccess;
  if (!prepared) {
    err = launch_prologue(adv, PrepImage{params_dev, static_cast<unsigned char *>(image), L, h->D, h->cfg.hidden}, kPrepBlocks, h->stream);
    if (err != cudaSuccess) return err;
    h->launches += 1;
  }
  const int expire = (h->expire_next & MAVA_EXPIRE_UPDATE) ? 1 : 0;
  h->expire_next &= ~MAVA_EXPIRE_UPDATE;
  const size_t smem = sizeof(UtcSmem);
  const auto kern = rows_need_64_bits(rows, rows.n) ? ppo_net_tc_kernel<uint64_t> : ppo_net_tc_kernel<uint32_t>;
  err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (err != cudaSuccess) return err;
  err = launch_dependent(kern, slices, kUThreads, smem, h->stream, static_cast<const unsigned char *>(image), rows, hp,
                         static_cast<const double *>(adv.out), partial, term_partial, h->d_status, h->D, h->cfg.hidden, prepared, expire);
  if (err != cudaSuccess) return err;
  h->launches += 2;
  return launch_dependent(reduce_slices_kernel<SliceMap>, kReduceBlocks, kReduceThreads, 0, h->stream, static_cast<const float *>(partial), kSlice, slices, grad,
                          terms, squares, SliceMap{L, h->D, h->cfg.hidden});
}
cudaError_t launch_grad_squares_tc(mava_rollout *h, const ParamLayout &L, const float *grad, double *squares) {
  return launch_dependent(grad_squares_kernel<SliceMap>, kMomentBlocks, kGradLanes, 0, h->stream, grad, squares, kSlice, SliceMap{L, h->D, h->cfg.hidden});
}
cudaError_t launch_step_tc(mava_rollout *h, const AdamArgs &adam, const ParamLayout &L, const Moments &next, void *image) {
  h->launches += 1;
  return launch_dependent(step_image_kernel, kMomentBlocks + kPrepBlocks, 256, 0, h->stream, adam, PrepImage{adam.params, static_cast<unsigned char *>(image), L, h->D, h->cfg.hidden}, next);
}

}  // namespace mava

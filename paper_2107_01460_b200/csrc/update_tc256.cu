// Update block on the tensor cores for hidden width 256 (sm_100a, tcgen05): the actor / shared-torso net and the
// centralised critic of the two largest shapes.  The weight gradient of the second layer alone (256 x 256 fp32) fills all
// 512 columns of an SM's tensor memory, and the weights (184 KB in bf16) leave no room for bf16 activation tiles in shared
// memory, so no SM can do a tile's row pass and its weight gradients.  One cooperative kernel therefore gives every SM one
// of three roles for the whole batch, and tiles travel between them through a ring of slots (three per row SM; about what L2
// holds beside the observations: most of what passes through is read from L2, and most of it is written back as well):
//   row SMs      per 128-row tile: forward and backward through the layers with the activations in tensor memory as the A
//                operand of the next product, the loss and its per-row derivatives in fp32; every bf16 matrix that a weight
//                gradient needs (x, h1, h2, d z2, d z1, the heads' derivatives) is stored to the tile's slot in the canonical
//                core-matrix layout [row][feature];
//   W2 SMs       stream the slots with bulk copies and read them with the row index as K (MN-major operands, see
//                update_tc.cu): d W2 += d z2^T . h1 (two 128 x 256 accumulators = all of tensor memory); d b2 by column sums;
//   W1 SMs       d W1 += d z1^T . x (up to two input slabs each) and d Wh^T += h2^T . dhead; d b1 is the product with a
//                column of ones that rides in x.
// Each weight SM adds to its own partial sums (every kFlushTiles tiles), and a last kernel adds those in a fixed order: same bytes on
// every call.
// Hand-over of a slot: the row SM's stores, then a release of the slot's counter; a weight SM acquires it, copies the tile
// into its shared-memory ring and releases the slot's "read" counter.  A tile's consumer is fixed by the tile's number, so
// the order of every sum is fixed too.  The launch is cooperative because the roles wait for one another.
// Rounding points are those of the bf16-operand mode of the float64 oracle.  Every wait is bounded.
//
// What bounds it (8 agents on 20x20): row SMs by themselves take 16.1 k cycles a tile, 12.4 k without the stores to the ring:
// eight epilogue warps for two groups' seven passes over half an accumulator each, the products (5.2 k) beside them.  The
// stores, 287 KB a tile at the 30 bytes per cycle that an SM's path into L2 takes, are 9.8 k.  A W2 SM by itself takes 3.1 k
// cycles a tile for its shared-memory reads.  Side by side they compete for L2: of the 4.75 GB that 4096 environments x 64
// steps send through the ring 3.8 GB are written back to HBM.
#include <cuda_bf16.h>

#include "common.cuh"
#include "layout.h"
#include "tc_common.cuh"
#include "update_common.cuh"

namespace mava {
namespace {

constexpr int kR = 128;       // rows per tile
constexpr int kH = 256;       // hidden width
constexpr int kK1 = 96;       // input width of a slab, padded (D = 81, 85); column D is ones (its product with d z1 is d b1)
constexpr int kHeads = 16;
constexpr int kThreads = 512;
// Registers of a row SM: the block starts with 128 per thread; 2 x 128 x 176 + 128 x 88 + 128 x 72 = 512 x 128.
constexpr int kGroupRegs = 176, kLoaderRegs = 88, kIssueRegs = 72;

// Image in shared memory: W1 (one input slab) | W2 | Wh | b1 | b2 | bh.  In global memory the image holds all slabs of W1
// first (kImgW2 bytes each), then the rest in the same order.
constexpr uint32_t kImgW1 = 0, kImgW2 = kImgW1 + kH * kK1 * 2, kImgWh = kImgW2 + kH * kH * 2;
constexpr uint32_t kImgB1 = kImgWh + kHeads * kH * 2, kImgB2 = kImgB1 + kH * 4, kImgBh = kImgB2 + kH * 4;
constexpr uint32_t kImgBytes = kImgBh + 32;
static_assert(kImgBytes % 16 == 0, "bulk copies");

// A slot of the ring: one x tile [128][96] per input slab; h1, h2, d z2, d z1 [128][256]; dhead [128][16].  An input slab is
// one agent's observation: the actor / shared-torso net has one, the centralised critic (input = the agents' observations
// side by side) one per agent.
constexpr uint32_t kXLbo = kALbo, kXSbo = (kK1 / 8) * kALbo;  // x tile: feature chunks 144 bytes apart (the converter's
                                                               // 2-byte stores then spread over the banks), row groups 1728
constexpr uint32_t kStXBytes = (kR / 8) * kXSbo;
constexpr uint32_t kActBytes = kR * kH * 2;
constexpr uint32_t kStDhBytes = kR * kHeads * 2;
constexpr uint32_t kSlotH1 = 0, kSlotH2 = kActBytes, kSlotDz2 = 2 * kActBytes, kSlotDz1 = 3 * kActBytes, kSlotDh = 4 * kActBytes,
                   kSlotX = kSlotDh + kStDhBytes;
__host__ __device__ constexpr size_t slot_bytes(int slabs) { return kSlotX + static_cast<size_t>(slabs) * kStXBytes; }

// tensor memory of a row SM: the accumulator as two column halves that the two thread groups use in turn; each group's
// hidden activations (bf16, two per column)
constexpr uint32_t kColAcc = 0, kColHid = 256, kTmemCols = 512;

struct RowSmem {
  alignas(128) unsigned char img[(kImgBytes + 127) / 128 * 128];
  alignas(128) unsigned char x[kStXBytes];
  alignas(128) unsigned char dhead[2][kStDhBytes];
  int rmap[kR];  // trajectory rows of the tile that is being fetched
  float red[8][8];
  alignas(8) uint64_t bar_load, x_full, x_empty, w1_full;
  uint64_t acc_free[2], acc_full[2][2], hid_ready[2][2], dh_ready[2], tile_done[2];
  uint32_t tmem_base;
};

// A weight SM's ring: items of 32 rows.  After kFlushTiles tiles the accumulators are added to the SM's partial sums in memory
// and start again at zero: a longer chain of fp32 additions inside the tensor core costs precision (16.8 million rows in one
// chain per SM: gradient off by 1e-3 relative; in chains of 48 tiles: 1e-5).
constexpr int kFlushTiles = 48;
constexpr int kItemRows = 32, kItemsPerTile = kR / kItemRows;
constexpr uint32_t kItemAct = kItemRows * kH * 2;                    // 16 KB: an item's rows of a [128][256] tile
constexpr uint32_t kXPart = (kItemRows / 8) * kXSbo, kDhPart = kItemRows * kHeads * 2;
constexpr uint32_t kRingBytes = 208 * 1024;
constexpr int kMaxStages = 6;
constexpr int kConsumerWarps = 8;
struct WgtSmem {
  alignas(128) unsigned char ring[kRingBytes];
  alignas(8) uint64_t full[kMaxStages], empty[kMaxStages], done, drained;
  uint32_t tmem_base;
};
constexpr size_t kSmemBytes = sizeof(RowSmem) > sizeof(WgtSmem) ? sizeof(RowSmem) : sizeof(WgtSmem);
static_assert(kSmemBytes <= 232448, "shared memory of a block");

// Which net the kernels work on: offsets of its layers in the flat parameter (= gradient) array and its input shape.
struct Net256 {
  size_t W1, b1, W2, b2, Wa, ba, Wv, bv;
  int D;          // width of one input slab (an agent's observation)
  int slabs;      // 1, or the number of agents for the centralised critic
  int w1_ld;      // input width of the first layer = slabs * D
  int has_actor, has_value;
};

// How a launch is cut up.
struct Split {
  int n_tiles, n_slots;
  int n_row, n_w2, n_w1;   // SMs per role; n_w1 per group of slabs
  int groups, per_group;   // groups of input slabs, slabs per group (the last may have fewer)
};
// Partial sums, matrices as [column / 4][unit][4] so that the lanes of a warp (= units) write whole lines.
// W2 SM: W2 [256 columns], b2 [256].  W1 SM: [per_group] x [96 columns] (column D of slab 0: b1), Wh [8 columns].
constexpr size_t kPartW2 = static_cast<size_t>(kH) * kH + kH;
__host__ __device__ constexpr size_t part_w1(int per_group) { return static_cast<size_t>(per_group) * kH * kK1 + kH * 8; }

struct Upd256Args {
  const unsigned char *image;
  UpdRows rows;
  UpdHyper hp;
  const double *adv_stats;
  unsigned char *ring;
  uint32_t *full, *x_full, *read;  // per slot: uses written (row groups / x tile), reads so far
  float *part_w2, *part_w1, *part_head;
  double *term_partial;            // [n_row][8 warps][3]
  int *status;
  Split sp;
  Net256 net;
};

// The weight image, and the ring's counters back to zero.
struct Prep256 {
  const float *params;
  unsigned char *image;
  Net256 net;
  uint32_t *counters;
  int n_counters;
  __device__ void operator()(int tid, int nth) const;
};
__device__ __forceinline__ void Prep256::operator()(int tid, int nth) const {
  const int D = net.D;
  for (int i = tid; i < n_counters; i += nth) counters[i] = 0;
  for (int i = tid; i < net.slabs * kH * kK1; i += nth) {
    const int a = i / (kH * kK1), r = i - a * (kH * kK1), n = r / kK1, k = r - n * kK1;
    reinterpret_cast<__nv_bfloat16 *>(image + static_cast<size_t>(a) * kImgW2)[canon_offset(n, k, kK1) / 2] =
        __float2bfloat16_rn(k < D ? __ldcg(params + net.W1 + static_cast<size_t>(n) * net.w1_ld + a * D + k) : 0.0f);
  }
  unsigned char *rest = image + static_cast<size_t>(net.slabs) * kImgW2 - kImgW2;  // so that rest + kImgX is where X lies
  auto bf = [&](uint32_t off) { return reinterpret_cast<__nv_bfloat16 *>(rest + off); };
  for (int i = tid; i < kH * kH; i += nth) {
    const int n = i / kH, k = i - n * kH;
    bf(kImgW2)[canon_offset(n, k, kH) / 2] = __float2bfloat16_rn(__ldcg(params + net.W2 + static_cast<size_t>(n) * kH + k));
  }
  for (int i = tid; i < kHeads * kH; i += nth) {
    const int n = i / kH, k = i - n * kH;
    float v = 0.0f;
    if (n < kActions && net.has_actor) v = __ldcg(params + net.Wa + static_cast<size_t>(n) * kH + k);
    else if (n == kActions && net.has_value) v = __ldcg(params + net.Wv + k);
    bf(kImgWh)[canon_offset(n, k, kH) / 2] = __float2bfloat16_rn(v);
  }
  float *b1 = reinterpret_cast<float *>(rest + kImgB1), *b2 = reinterpret_cast<float *>(rest + kImgB2), *bh = reinterpret_cast<float *>(rest + kImgBh);
  for (int i = tid; i < kH; i += nth) { b1[i] = __ldcg(params + net.b1 + i); b2[i] = __ldcg(params + net.b2 + i); }
  if (tid < 8) bh[tid] = (tid < kActions && net.has_actor) ? __ldcg(params + net.ba + tid) : ((tid == kActions && net.has_value) ? __ldcg(params + net.bv) : 0.0f);
}

__device__ __forceinline__ uint64_t desc_k(uint32_t tile, int C, int k) { return smem_desc(tile + k * 256, 128, C * 16); }
__device__ __forceinline__ uint64_t desc_mn(uint32_t tile, int C, int k) { return smem_desc(tile + k * 2 * C * 16, C * 16, 128); }
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;
// The descriptor `bytes` further on: the address field counts 16-byte units and cannot carry out of its 14 bits here, so one
// addition replaces the field arithmetic (and the issuing thread needs no register per descriptor).
__device__ __forceinline__ uint64_t desc_at(uint64_t base, uint32_t bytes) { return base + (bytes >> 4); }

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void stg_v4(void *p, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v) { asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void red_release(uint32_t *p) { asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory"); }
__device__ __forceinline__ void fence_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
// Bounded wait until *p has reached `value`.
__device__ __forceinline__ bool wait_count(const uint32_t *p, uint32_t value) {
#pragma unroll 1
  for (uint32_t i = 0; i < kSpinLimit; ++i)
    if (static_cast<int32_t>(ld_acquire(p) - value) >= 0) return true;
  return false;
}
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t *r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// ---- epilogues of a row SM --------------------------------------------------------------------------------------------
// A thread owns a row; one call handles a half (128 columns) of the accumulator, 32 columns at a time with the next load in
// flight.  What a layer hands on goes back to tensor memory (A operand of the next product) and to the slot.
enum class Epi { kHidden1, kHidden2, kGrad2, kGrad1 };

// 32 accumulator columns -> 16 packed pairs, also stored to the slot; gates: kHidden1 collects one bit per unit (pair i:
// bits 15 - i and 31 - i) that kGrad1 applies; kGrad2 takes its gate from the activations still in tensor memory (`act`).
template <Epi E>
__device__ __forceinline__ void epi_batch(uint32_t *v, const uint32_t *act, uint32_t bias, uint32_t &gate, uint32_t *pk, unsigned char *dst) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if constexpr (E == Epi::kHidden1 || E == Epi::kHidden2) {
      const float4 ba = lds_float4(bias + 32u * q), bb = lds_float4(bias + 32u * q + 16u);
      add2(v[8 * q], v[8 * q + 1], ba.x, ba.y); add2(v[8 * q + 2], v[8 * q + 3], ba.z, ba.w);
      add2(v[8 * q + 4], v[8 * q + 5], bb.x, bb.y); add2(v[8 * q + 6], v[8 * q + 7], bb.z, bb.w);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * q + e;
      if constexpr (E == Epi::kHidden1 || E == Epi::kHidden2) {
        pk[i] = relu_pack_bf16(v[2 * i], v[2 * i + 1]);
        if constexpr (E == Epi::kHidden1) gate |= positive_mask(pk[i]) & (0x80008000u >> i);
      } else {
        const uint32_t p = pack_bf16(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
        if constexpr (E == Epi::kGrad2) pk[i] = p & positive_mask(act[i]);
        else pk[i] = p & sign_mask(gate << i);
      }
    }
    stg_v4(dst + q * 128, pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
  }
}
// DEFER: the products of the other column half may still be reading the hidden columns, so what goes there waits (in
// registers) for `other_full` to complete.  Returns whether the waits were in time.
template <Epi E, bool DEFER>
__device__ __forceinline__ bool epilogue_half(uint32_t acc, uint32_t hid, uint32_t bias, uint32_t *gate, unsigned char *dst, uint32_t acc_free,
                                              uint32_t hid_ready, int lane, uint32_t other_full = 0, uint32_t other_ph = 0) {
  uint32_t ra[32], rb[32], ha[16], hb[16], pk[DEFER ? 4 : 1][16];
  bool ok = true;
  tmem_ld32_nowait(acc, ra);
  if constexpr (E == Epi::kGrad2) tmem_ld16_nowait(hid, ha);
#pragma unroll
  for (int c = 0; c < 4; c += 2) {
    tmem_ld_wait();
    tmem_ld32_nowait(acc + 32u * (c + 1), rb);
    if constexpr (E == Epi::kGrad2) tmem_ld16_nowait(hid + 16u * (c + 1), hb);
    epi_batch<E>(ra, ha, bias + 128u * c, gate[c], pk[DEFER ? c : 0], dst + c * 512);
    if constexpr (E != Epi::kGrad1 && !DEFER) tmem_st16(hid + 16u * c, pk[0]);
    tmem_ld_wait();
    if (c == 0) {
      tmem_ld32_nowait(acc + 64u, ra);
      if constexpr (E == Epi::kGrad2) tmem_ld16_nowait(hid + 32u, ha);
    } else {  // the accumulator half has been read
      tc_fence_before();
      warp_arrive(acc_free, lane);
    }
    epi_batch<E>(rb, hb, bias + 128u * (c + 1), gate[c + 1], pk[DEFER ? c + 1 : 0], dst + (c + 1) * 512);
    if constexpr (E != Epi::kGrad1 && !DEFER) tmem_st16(hid + 16u * (c + 1), pk[0]);
  }
  if constexpr (DEFER) {
    ok = mbar_wait(other_full, other_ph);
    tc_fence_after();
#pragma unroll
    for (int c = 0; c < 4; ++c) tmem_st16(hid + 16u * c, pk[DEFER ? c : 0]);
  }
  if constexpr (E != Epi::kGrad1) {
    tmem_st_wait();
    tc_fence_before();
    warp_arrive(hid_ready, lane);
  }
  return ok;
}

// ---- row SM -----------------------------------------------------------------------------------------------------------
// Warps 0..7: two groups of 128 threads (thread = row), each with its own tile (even / odd tiles of the SM) and hidden
// columns.  Warps 8..11: the next tile's rows from the obs array, as bf16, into the x tile.  Warp 12: all MMAs, in a fixed
// order, one group half a tile behind the other (one group's epilogue runs beside the other's products, and tiles are
// finished one by one: with both groups in step they came in pairs and the ring of slots ran dry).  Warp 13: hands finished
// tiles over.
template <class U>  // row numbers of the batch (real_row)
__device__ __forceinline__ bool row_role(const Upd256Args &a, RowSmem &sm, uint32_t tmem) {
  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  const Split &sp = a.sp;
  const Net256 &net = a.net;
  const int D = net.D, slabs = net.slabs;
  const int my_tiles = (sp.n_tiles - static_cast<int>(blockIdx.x) + sp.n_row - 1) / sp.n_row;
  const size_t slot_size = slot_bytes(slabs);
  const uint32_t w1 = smem_u32(sm.img + kImgW1), w2 = smem_u32(sm.img + kImgW2), wh = smem_u32(sm.img + kImgWh), xt = smem_u32(sm.x);
  auto tile_of = [&](int s) { return static_cast<int>(blockIdx.x) + s * sp.n_row; };
  bool ok = true;

  if (warp < 8) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGroupRegs));
    const int g = warp >> 2, row = tid & 127;
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t acc = tmem + kColAcc + lane_off, hid = tmem + kColHid + 128u * g + lane_off;
    const uint32_t full0 = smem_u32(&sm.acc_full[g][0]), full1 = smem_u32(&sm.acc_full[g][1]), free0 = smem_u32(&sm.acc_free[0]),
                   free1 = smem_u32(&sm.acc_free[1]), ready0 = smem_u32(&sm.hid_ready[g][0]), ready1 = smem_u32(&sm.hid_ready[g][1]);
    const uint32_t dht = smem_u32(sm.dhead[g]) + static_cast<uint32_t>((row >> 3) * (kHeads * 16) + (row & 7) * 16);
    const uint32_t b1 = smem_u32(sm.img + kImgB1), b2 = smem_u32(sm.img + kImgB2);
    const float *bh = reinterpret_cast<const float *>(sm.img + kImgBh);
    const float mean = static_cast<float>(a.adv_stats[0]);
    const float inv_std = 1.0f / (static_cast<float>(a.adv_stats[1]) + 1e-8f);
    const float inv_n = 1.0f / static_cast<float>(a.rows.n);
    const UpdHyper hp = a.hp;
    const bool has_actor = net.has_actor, has_value = net.has_value;
    const size_t row_off = static_cast<size_t>((row >> 3) * 4096 + (row & 7) * 16);  // 8-row groups, a row's 16-byte pieces 128 apart
    double t_actor = 0.0, t_ent = 0.0, t_value = 0.0;
    float gbh[kActions + 1];
#pragma unroll
    for (int k = 0; k <= kActions; ++k) gbh[k] = 0.0f;
    uint32_t ph0 = 0, ph1 = 0;
    for (int s = g; s < my_tiles && ok; s += 2) {
      const int lt = tile_of(s);
      const long long row0 = static_cast<long long>(lt) * kR;
      unsigned char *slot = a.ring + static_cast<size_t>(lt % sp.n_slots) * slot_size;
      const long long my_row = row0 + row < a.rows.n ? real_row<U>(a.rows, row0 + row) : -1;
      int action = 0;
      float logp_old = 0.0f, adv = 0.0f, v_old = 0.0f, ret = 0.0f;
      if (row0 + row < a.rows.n && my_row < 0) atomicExch(a.status, kStatusBadIndex);
      if (my_row >= 0) {  // used after the heads: the loads are in flight meanwhile
        if (has_actor) { action = a.rows.actions[my_row]; logp_old = a.rows.logp_old[my_row]; adv = a.rows.adv[my_row]; }
        if (has_value) { v_old = a.rows.value_old[my_row * a.rows.vstride]; ret = a.rows.ret[my_row * a.rows.vstride]; }
      }
      uint32_t gate[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) gate[k] = 0;
      unsigned char *dst = slot + row_off;
      // (the x tile is only handed to the MMAs once the slot is free to be written)
      ok = mbar_wait(full0, ph0); ph0 ^= 1;
      if (!__all_sync(0xFFFFFFFFu, ok)) { ok = false; break; }
      tc_fence_after();
      epilogue_half<Epi::kHidden1, false>(acc, hid, b1, gate, dst + kSlotH1, free0, ready0, lane);
      ok = mbar_wait(full1, ph1); ph1 ^= 1;
      tc_fence_after();
      epilogue_half<Epi::kHidden1, false>(acc + 128u, hid + 64u, b1 + 512u, gate + 4, dst + kSlotH1 + 2048, free1, ready1, lane);
      ok = ok && mbar_wait(full0, ph0); ph0 ^= 1;
      tc_fence_after();
      ok &= epilogue_half<Epi::kHidden2, true>(acc, hid, b2, gate, dst + kSlotH2, free0, ready0, lane, full1, ph1);
      ph1 ^= 1;
      epilogue_half<Epi::kHidden2, false>(acc + 128u, hid + 64u, b2 + 512u, gate, dst + kSlotH2 + 2048, free1, ready1, lane);
      ok = ok && mbar_wait(full0, ph0); ph0 ^= 1;
      tc_fence_after();
      float hv[16], d[8];
      tmem_ld16(acc, hv);
      tc_fence_before();
      warp_arrive(free0, lane);
#pragma unroll
      for (int k = 0; k < 8; ++k) d[k] = 0.0f;
      if (my_row >= 0 && has_actor) {
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
      }
      if (my_row >= 0 && has_value) {
        const float v = hv[kActions] + bh[kActions];
        const float u = v - ret, uc = v_old + fminf(fmaxf(v - v_old, -hp.clip_eps), hp.clip_eps) - ret;
        const bool in_range = fabsf(v - v_old) <= hp.clip_eps;
        d[kActions] = (in_range || u * u > uc * uc) ? hp.vf_coef * u * inv_n : 0.0f;
        t_value += 0.5 * fmaxf(u * u, uc * uc);
      }
      const uint32_t q0 = pack_bf16(d[0], d[1]), q1 = pack_bf16(d[2], d[3]), q2 = pack_bf16(d[4], d[5]), q3 = pack_bf16(d[6], 0.0f);
      sts_v4(dht, q0, q1, q2, q3);
      fence_async_smem();
      warp_arrive(smem_u32(&sm.dh_ready[g]), lane);
      unsigned char *dh = slot + kSlotDh + (row >> 3) * (kHeads * 16) + (row & 7) * 16;
      stg_v4(dh, q0, q1, q2, q3);
      stg_v4(dh + 128, 0u, 0u, 0u, 0u);
#pragma unroll
      for (int k = 0; k <= kActions; ++k) gbh[k] += d[k];  // the heads' bias gradients sum the unrounded derivatives
      ok = ok && mbar_wait(full0, ph0); ph0 ^= 1;
      tc_fence_after();
      epilogue_half<Epi::kGrad2, false>(acc, hid, 0, gate, dst + kSlotDz2, free0, ready0, lane);
      ok = ok && mbar_wait(full1, ph1); ph1 ^= 1;
      tc_fence_after();
      epilogue_half<Epi::kGrad2, false>(acc + 128u, hid + 64u, 0, gate, dst + kSlotDz2 + 2048, free1, ready1, lane);
      ok = ok && mbar_wait(full0, ph0); ph0 ^= 1;
      tc_fence_after();
      epilogue_half<Epi::kGrad1, false>(acc, hid, 0, gate, dst + kSlotDz1, free0, 0, lane);
      ok = ok && mbar_wait(full1, ph1); ph1 ^= 1;
      tc_fence_after();
      epilogue_half<Epi::kGrad1, false>(acc + 128u, hid + 64u, 0, gate + 4, dst + kSlotDz1 + 2048, free1, 0, lane);
      warp_arrive(smem_u32(&sm.tile_done[g]), lane);
      ok = __all_sync(0xFFFFFFFFu, ok);
    }
    // sums over the SM's rows: the heads' bias gradients, the loss terms
#pragma unroll
    for (int k = 0; k <= kActions; ++k)
      for (int o = 16; o > 0; o >>= 1) gbh[k] += __shfl_xor_sync(0xFFFFFFFFu, gbh[k], o);
    double t[3] = {t_actor, t_ent, t_value};
#pragma unroll
    for (int k = 0; k < 3; ++k)
      for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xFFFFFFFFu, t[k], o);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k <= kActions; ++k) sm.red[warp][k] = gbh[k];
      double *tp = a.term_partial + (static_cast<size_t>(blockIdx.x) * 8 + warp) * 3;
      tp[0] = t[0]; tp[1] = t[1]; tp[2] = t[2];
    }
  } else if (warp < 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kLoaderRegs));
    // ---- the rows: warp w of four the rows 32 w .., sixteen at a time, consecutive lanes consecutive features
    const int lw = warp - 8;
    const bool third = lane + 64 < D;
    const uint32_t my_col = xt + a_offset<kK1>(32 * lw, lane), rmap = smem_u32(&sm.rmap[32 * lw]);
    const bool lead = tid == 256;
    const uint32_t x_full = smem_u32(&sm.x_full), x_empty = smem_u32(&sm.x_empty), w1_full = smem_u32(&sm.w1_full);
    const uint32_t reads = static_cast<uint32_t>(1 + sp.groups);  // reads of a slot per use
    int n = 0, prev_slot = -1;
    uint32_t prev_use = 0;
    for (int s = 0; s < my_tiles && ok; ++s) {
      const int lt = tile_of(s), use = lt / sp.n_slots, slot_no = lt - use * sp.n_slots;
      const long long q = static_cast<long long>(lt) * kR + 32 * lw + lane;
      __syncwarp();
      sm.rmap[32 * lw + lane] = static_cast<int>(q < a.rows.n ? real_row<U>(a.rows, q) : -1);
      __syncwarp();
      unsigned char *slot = a.ring + static_cast<size_t>(slot_no) * slot_size;
      for (int sl = 0; sl < slabs && ok; ++sl, ++n) {
#pragma unroll 1
        for (int b = 0; b < 32; b += 16) {
          float v[16][3];
#pragma unroll
          for (int r = 0; r < 16; ++r) {
            const int src = lds_s32(rmap + 4u * static_cast<uint32_t>(b + r));
            const float *p = a.rows.x + static_cast<long long>(src) * net.w1_ld + sl * D + lane;
            v[r][0] = ldg_if(p, src >= 0);  // (D > 64: the first two are columns of every row)
            v[r][1] = ldg_if(p + 32, src >= 0);
            v[r][2] = ldg_if(p + 64, src >= 0 && third);
          }
          if (b == 0) {  // the x tile is free: the previous slab's products and its copy to the slot have read it
            if (n > 0) ok = mbar_wait(x_empty, static_cast<uint32_t>(n - 1) & 1u);
            if (lead) {
              bulk_store_wait_all();
              if (sl == 0) {
                if (prev_slot >= 0) { fence_async_all(); st_release(a.x_full + prev_slot, prev_use + 1u); }
                if (use > 0) ok = ok && wait_count(a.read + slot_no, reads * static_cast<uint32_t>(use));
              }
              if (slabs > 1 && ok) {
                mbar_expect_tx(w1_full, kImgW2);
                for (uint32_t o = 0; o < kImgW2; o += 16384) bulk_load(w1 + o, a.image + static_cast<size_t>(sl) * kImgW2 + o, 16384, w1_full);
              }
            }
            ok = group_any(2, !ok) == false;
            if (!ok) break;
          }
#pragma unroll
          for (int r = 0; r < 16; ++r) {  // (a chunk of eight features is 144 bytes on: 32 features are 576)
            const uint32_t at = my_col + static_cast<uint32_t>(b / 8) * kXSbo + (r >> 3) * kXSbo + (r & 7) * 16;
            sts_u16(at, bf16_bits(v[r][0]));
            sts_u16(at + 576u, bf16_bits(v[r][1]));
            if (third) sts_u16(at + 1152u, bf16_bits(v[r][2]));
          }
        }
        if (!ok) break;
        fence_async_smem();
        group_sync(2);
        if (lead) {
          bulk_store(slot + kSlotX + static_cast<size_t>(sl) * kStXBytes, xt, kStXBytes);
          mbar_arrive(x_full);
        }
      }
      prev_slot = slot_no; prev_use = static_cast<uint32_t>(use);
    }
    if (lead) {
      bulk_store_wait_all();
      if (ok && prev_slot >= 0) { fence_async_all(); st_release(a.x_full + prev_slot, prev_use + 1u); }
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
    if (warp == 12) {  // the whole warp walks through the waits, one lane issues (elect_one)
      uint32_t uses[2] = {0, 0};  // of each accumulator half
      uint32_t hid_ph[2] = {0, 0}, dh_ph[2] = {0, 0};
      uint32_t n = 0;
      auto take = [&](int h) {  // the half's previous epilogue has read it
        ok = ok && mbar_wait_warp(smem_u32(&sm.acc_free[h]), (uses[h] & 1u) ^ 1u);
        ++uses[h];
        tc_fence_after();
      };
      auto hidden = [&](int g, int h) { ok = ok && mbar_wait_warp(smem_u32(&sm.hid_ready[g][h]), hid_ph[g]); tc_fence_after(); };
      constexpr uint32_t idesc = instr_desc(kR, 128);
      uint64_t d_x = smem_desc(xt, kXLbo, kXSbo), d_w1 = desc_k(w1, kK1, 0), d_w2 = desc_k(w2, kH, 0), d_w2t = desc_mn(w2, kH, 0),
               d_wh = desc_k(wh, kH, 0), d_wht = desc_mn(wh, kH, 0);
      // not loop invariants to the compiler: it would keep every product's descriptors in registers that it does not have
      auto fresh = [&]() { asm volatile("" : "+l"(d_x), "+l"(d_w1), "+l"(d_w2), "+l"(d_w2t), "+l"(d_wh), "+l"(d_wht)); };
      // tile s (group s & 1) goes forward while tile s - 1 (the other group) goes backward: the groups stay half a tile apart
#pragma unroll 1
      for (int s = 0; s <= my_tiles && ok; ++s) {
        const bool fwd = s < my_tiles, bwd = s > 0;
        const int g = s & 1, o = g ^ 1;
        const uint32_t hd = tmem + kColHid + 128u * g, ho = tmem + kColHid + 128u * o;
        fresh();
        if (fwd) {  // z1 = sum over slabs of x_a . W1_a^T
#pragma unroll 1
          for (int sl = 0; sl < slabs && ok; ++sl, ++n) {
            ok = mbar_wait_warp(smem_u32(&sm.x_full), n & 1u);
            if (slabs > 1) ok = ok && mbar_wait_warp(smem_u32(&sm.w1_full), n & 1u);
            tc_fence_after();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (sl == 0) take(h);
              if (elect_one()) {
#pragma unroll
                for (int k = 0; k < kK1 / 16; ++k)
                  mma_bf16(tmem + kColAcc + 128u * h, desc_at(d_x, k * 2 * kXLbo), desc_at(d_w1, h * 16 * (kK1 * 16) + k * 256), idesc, (sl > 0) | (k > 0));
                if (sl == slabs - 1) mma_commit(smem_u32(&sm.acc_full[g][h]));
                if (h == 1) mma_commit(smem_u32(&sm.x_empty));
              }
              __syncwarp();
            }
          }
        }
        if (bwd && ok) {  // d h2 = dhead . Wh
          ok = mbar_wait_warp(smem_u32(&sm.dh_ready[o]), dh_ph[o]);
          dh_ph[o] ^= 1;
          tc_fence_after();
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            take(h);
            if (elect_one()) {
              mma_bf16(tmem + kColAcc + 128u * h, desc_k(smem_u32(sm.dhead[o]), kHeads, 0), desc_at(d_wht, h * 16 * 128), idesc | kBmn, 0);
              mma_commit(smem_u32(&sm.acc_full[o][h]));
            }
            __syncwarp();
          }
        }
        fresh();
        if (fwd && ok) {  // z2 = h1 . W2^T; the first half of the K steps needs only the first half of h1
          hidden(g, 0);
          take(0);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 8; ++k) mma_bf16_ts(tmem + kColAcc, hd + k * 8, desc_at(d_w2, k * 256), idesc, k > 0);
          }
          __syncwarp();
          hidden(g, 1);
          if (elect_one()) {
#pragma unroll
            for (int k = 8; k < 16; ++k) mma_bf16_ts(tmem + kColAcc, hd + k * 8, desc_at(d_w2, k * 256), idesc, 1);
            mma_commit(smem_u32(&sm.acc_full[g][0]));
          }
          __syncwarp();
          take(1);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 16; ++k) mma_bf16_ts(tmem + kColAcc + 128u, hd + k * 8, desc_at(d_w2, 16 * (kH * 16) + k * 256), idesc, k > 0);
            mma_commit(smem_u32(&sm.acc_full[g][1]));
          }
          __syncwarp();
          hid_ph[g] ^= 1;
        }
        fresh();
        if (bwd && ok) {  // d h1 = d z2 . W2
          hidden(o, 0);
          take(0);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 8; ++k) mma_bf16_ts(tmem + kColAcc, ho + k * 8, desc_at(d_w2t, k * 2 * kH * 16), idesc | kBmn, k > 0);
          }
          __syncwarp();
          hidden(o, 1);
          if (elect_one()) {
#pragma unroll
            for (int k = 8; k < 16; ++k) mma_bf16_ts(tmem + kColAcc, ho + k * 8, desc_at(d_w2t, k * 2 * kH * 16), idesc | kBmn, 1);
            mma_commit(smem_u32(&sm.acc_full[o][0]));
          }
          __syncwarp();
          take(1);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 16; ++k) mma_bf16_ts(tmem + kColAcc + 128u, ho + k * 8, desc_at(d_w2t, 16 * 128 + k * 2 * kH * 16), idesc | kBmn, k > 0);
            mma_commit(smem_u32(&sm.acc_full[o][1]));
          }
          __syncwarp();
          hid_ph[o] ^= 1;
        }
        fresh();
        if (fwd && ok) {  // heads
          hidden(g, 0);
          hidden(g, 1);
          take(0);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 16; ++k) mma_bf16_ts(tmem + kColAcc, hd + k * 8, desc_at(d_wh, k * 256), instr_desc(kR, kHeads), k > 0);
            mma_commit(smem_u32(&sm.acc_full[g][0]));
          }
          __syncwarp();
          hid_ph[g] ^= 1;
        }
      }
    }
    if (warp == 13 && lane == 0) {
      for (int s = 0; s < my_tiles && ok; ++s) {
        ok = mbar_wait(smem_u32(&sm.tile_done[s & 1]), static_cast<uint32_t>(s >> 1) & 1u);
        if (!ok) break;
        const int lt = tile_of(s), use = lt / sp.n_slots;
        __threadfence();    // the groups' stores, observed through the barrier, before the counter
        fence_async_all();  // the reader's copies go through the async proxy
        st_release(a.full + (lt - use * sp.n_slots), static_cast<uint32_t>(use) + 1u);
      }
    }
  }
  return ok;
}

// ---- weight SMs -------------------------------------------------------------------------------------------------------
// A work item is 32 rows of a tile.  Warp 8: copies, two items' worth of stages ahead; warp 9: MMAs; warps 0..7 (W2 SMs):
// the column sums of d z2.
// NS: input slabs of this W1 SM (0: a W2 SM); HEADS: it also does d Wh.  Compile-time, so that the operands of copies and MMAs
// stay in uniform registers (with run-time loops around them a W1 tile took 3.5 k cycles to issue).
template <int NS, bool HEADS>
__device__ __forceinline__ bool weight_role(const Upd256Args &a, WgtSmem &sm, uint32_t tmem, int rank, int peers, int slab0) {
  constexpr bool W2 = NS == 0, heads_too = HEADS;
  constexpr int n_slabs = NS;
  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  const Split &sp = a.sp;
  const Net256 &net = a.net;
  const size_t slot_size = slot_bytes(net.slabs);
  // stage: W2: d z2, h1; W1: d z1, x of up to two slabs, and with slab 0 h2 and dhead
  constexpr uint32_t o_b = kItemAct, o_x = kItemAct, o_h2 = o_x + n_slabs * kXPart, o_dh = o_h2 + kItemAct;
  constexpr uint32_t stage_bytes = W2 ? 2 * kItemAct : (heads_too ? o_dh + kDhPart : o_h2);
  constexpr int kFit = static_cast<int>(kRingBytes / stage_bytes), S = kFit < kMaxStages ? kFit : kMaxStages;
  const uint32_t ring = smem_u32(sm.ring), full0 = smem_u32(&sm.full[0]), empty0 = smem_u32(&sm.empty[0]), done_bar = smem_u32(&sm.done);
  const int my_tiles = (sp.n_tiles - rank + peers - 1) / peers, n_items = kItemsPerTile * my_tiles;
  bool ok = true;
  float db0 = 0.0f, db1 = 0.0f;

  if (warp == kConsumerWarps) {
    int issued = 0, s = 0;
    uint32_t round = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      const int lt = rank + i * peers, use = lt / sp.n_slots, slot_no = lt - use * sp.n_slots;
      ok = wait_count(a.full + slot_no, static_cast<uint32_t>(use) + 1u);
      if (!W2) ok = ok && wait_count(a.x_full + slot_no, static_cast<uint32_t>(use) + 1u);
      ok = __all_sync(0xFFFFFFFFu, ok);
      fence_async_all();
      const unsigned char *slot = a.ring + static_cast<size_t>(slot_no) * slot_size;
#pragma unroll 1
      for (int q = 0; q < kItemsPerTile && ok; ++q) {
        if (round > 0) ok = mbar_wait_warp(empty0 + 8u * s, (round - 1u) & 1u);
        if (!ok) break;
        const uint32_t dst = ring + static_cast<uint32_t>(s) * stage_bytes, bar = full0 + 8u * s;
        if (elect_one()) {
          mbar_expect_tx(bar, stage_bytes);
          bulk_load(dst, slot + (W2 ? kSlotDz2 : kSlotDz1) + static_cast<size_t>(q) * kItemAct, kItemAct, bar);
          if constexpr (W2) {
            bulk_load(dst + o_b, slot + kSlotH1 + static_cast<size_t>(q) * kItemAct, kItemAct, bar);
          } else {
#pragma unroll
            for (int x = 0; x < n_slabs; ++x)
              bulk_load(dst + o_x + x * kXPart, slot + kSlotX + static_cast<size_t>(slab0 + x) * kStXBytes + static_cast<size_t>(q) * kXPart, kXPart, bar);
            if constexpr (heads_too) {
              bulk_load(dst + o_h2, slot + kSlotH2 + static_cast<size_t>(q) * kItemAct, kItemAct, bar);
              bulk_load(dst + o_dh, slot + kSlotDh + static_cast<size_t>(q) * kDhPart, kDhPart, bar);
            }
          }
        }
        __syncwarp();
        ++issued;
        if (++s == S) { s = 0; ++round; }
      }
    }
    if (!ok)  // let the copies still in flight land before the block goes away
      for (int u = issued > S ? issued - S : 0; u < issued; ++u) mbar_wait(full0 + 8u * (u % S), (u / S) & 1);
  } else if (warp == kConsumerWarps + 1) {
    int s = 0;
    uint32_t round = 0, keep = 0, flushes = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      if (i > 0 && i % kFlushTiles == 0) {
        if (elect_one()) mma_commit(done_bar);  // covers every MMA issued above
        __syncwarp();
        ok = mbar_wait_warp(smem_u32(&sm.drained), flushes & 1u);
        if (!ok) break;
        tc_fence_after();
        ++flushes;
        keep = 0;
      }
      for (int q = 0; q < kItemsPerTile; ++q) {
        ok = mbar_wait_warp(full0 + 8u * s, round & 1u);
        if (!ok) break;
        tc_fence_after();
        const uint32_t base = ring + static_cast<uint32_t>(s) * stage_bytes;
        if (elect_one()) {
          if (W2) {
#pragma unroll
            for (int k = 0; k < kItemRows / 16; ++k)
#pragma unroll
              for (int h = 0; h < 2; ++h)
                mma_bf16(tmem + 256u * h, desc_mn(base + h * 2048, kH, k), desc_mn(base + o_b, kH, k), instr_desc(128, 256) | kAmn | kBmn, keep | (k > 0));
          } else {
#pragma unroll
            for (int k = 0; k < kItemRows / 16; ++k)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int x = 0; x < n_slabs; ++x)
                  mma_bf16(tmem + static_cast<uint32_t>((2 * x + h) * kK1), desc_mn(base + h * 2048, kH, k),
                           smem_desc(base + o_x + x * kXPart + k * 2 * kXSbo, kXSbo, kXLbo), instr_desc(128, kK1) | kAmn | kBmn, keep | (k > 0));
                if (heads_too)
                  mma_bf16(tmem + static_cast<uint32_t>(4 * kK1 + 32 * h), desc_mn(base + o_h2 + h * 2048, kH, k), desc_mn(base + o_dh, kHeads, k),
                           instr_desc(128, kHeads) | kAmn | kBmn, keep | (k > 0));
              }
          }
          mma_commit(empty0 + 8u * s);
        }
        __syncwarp();
        keep = 1;
        if (++s == S) { s = 0; ++round; }
      }
      if (ok && lane == 0) red_release(a.read + (rank + i * peers) % sp.n_slots);  // the tile's copies have all landed
    }
    if (ok && elect_one()) mma_commit(done_bar);
    __syncwarp();
  } else if (warp < kConsumerWarps) {
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int h = warp >> 2, unit = h * 128 + (warp & 3) * 32 + lane;  // out-unit half; tensor-memory lane = unit inside the half
    float *part = W2 ? a.part_w2 + static_cast<size_t>(rank) * kPartW2
                     : a.part_w1 + (static_cast<size_t>(slab0 / sp.per_group) * sp.n_w1 + rank) * part_w1(sp.per_group);
    uint32_t flushes = 0;
    // `n` (a multiple of 8) accumulator columns from `col` on, to (first time) or onto the partial sums at `dst`
    auto put = [&](float *dst, uint32_t col, int n) {
      for (int c0 = 0; c0 < n; c0 += 8) {
        uint32_t v[8];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                     : "r"(tmem + lane_off + col + c0)
                     : "memory");
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float *to = dst + (static_cast<size_t>(c0 / 4 + q) * kH + unit) * 4;
          if (flushes == 0) stg_v4(to, v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          else
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(to), "f"(__uint_as_float(v[4 * q])), "f"(__uint_as_float(v[4 * q + 1])),
                         "f"(__uint_as_float(v[4 * q + 2])), "f"(__uint_as_float(v[4 * q + 3]))
                         : "memory");
        }
      }
    };
    auto flush = [&]() {
      const bool in_time = mbar_wait_warp(done_bar, flushes & 1u);
      if (!in_time) return false;
      tc_fence_after();
      if (W2) {
        put(part, static_cast<uint32_t>(h * 256), kH);
      } else {
        for (int x = 0; x < n_slabs; ++x) put(part + static_cast<size_t>(x) * kH * kK1, static_cast<uint32_t>((2 * x + h) * kK1), kK1);
        if (heads_too) put(part + static_cast<size_t>(sp.per_group) * kH * kK1, static_cast<uint32_t>(4 * kK1 + 32 * h), 8);
      }
      ++flushes;
      tc_fence_before();
      warp_arrive(smem_u32(&sm.drained), lane);
      return true;
    };
    if (W2) {
      // column sums of d z2.  Thread (w, l): units 2p, 2p + 1 with p = 32 (w & 3) + l, over the item's rows 16 (w >> 2) .. + 15,
      // by 4-byte loads.  A warp's 32 unit pairs are eight 16-byte pieces 128 bytes apart, i.e. on the same four banks: each
      // piece's four lanes therefore start at a different row of the 8-row group (row offset 16 bytes = four banks) and a load
      // touches all 32 banks once.  The two row halves are added at the end, in a fixed order: the same bytes on every call.
      const int p = (warp & 3) * 32 + lane, rot = lane >> 2;
      const uint32_t my_col = static_cast<uint32_t>((p >> 2) * 128 + (p & 3) * 4) + static_cast<uint32_t>(warp >> 2) * 2 * 4096;
      float t0 = 0.0f, t1 = 0.0f;  // since the last flush
      int s = 0;
      uint32_t round = 0;
      for (int u = 0; u < n_items && ok; ++u) {
        if (u > 0 && u % (kFlushTiles * kItemsPerTile) == 0) {
          db0 += t0; db1 += t1; t0 = t1 = 0.0f;
          ok = flush();
          if (!ok) break;
        }
        ok = mbar_wait_warp(full0 + 8u * s, round & 1u);
        if (!ok) break;
        const uint32_t base = ring + static_cast<uint32_t>(s) * stage_bytes;
#pragma unroll
        for (int rg = 0; rg < 2; ++rg)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t w = lds_u32(base + my_col + static_cast<uint32_t>(rg * 4096) + static_cast<uint32_t>(((j + rot) & 7) * 16));
            t0 += __uint_as_float(w << 16);
            t1 += __uint_as_float(w & 0xFFFF0000u);
          }
        // the stage's next writer is a bulk copy (async proxy); these were generic-proxy reads
        fence_async_smem();
        warp_arrive(empty0 + 8u * s, lane);
        if (++s == S) { s = 0; ++round; }
      }
      db0 += t0; db1 += t1;
    } else {
      for (int i = kFlushTiles; i < my_tiles && ok; i += kFlushTiles) ok = flush();
    }
    if (ok) ok = flush();
  }
  ok = __syncthreads_and(ok) != 0;
  if (W2) {  // the two row halves of the bias sums meet in the ring, which is idle: every copy and every MMA has completed
    float *xch = reinterpret_cast<float *>(sm.ring);
    const int p = (warp & 3) * 32 + lane;
    if (ok && warp >= 4 && warp < kConsumerWarps) { xch[2 * p] = db0; xch[2 * p + 1] = db1; }
    __syncthreads();
    if (ok && warp < 4) {
      float *to = a.part_w2 + static_cast<size_t>(rank) * kPartW2 + kH * kH + 2 * tid;
      to[0] = db0 + xch[2 * p];
      to[1] = db1 + xch[2 * p + 1];
    }
  }
  return ok;
}

template <class U>
__global__ void __launch_bounds__(kThreads, 1) ppo_update256_kernel(const __grid_constant__ Upd256Args a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int bid = static_cast<int>(blockIdx.x);
  const Split &sp = a.sp;
  const bool row_sm = bid < sp.n_row, w2_sm = !row_sm && bid < sp.n_row + sp.n_w2;
  RowSmem &rs = *reinterpret_cast<RowSmem *>(smem_raw);
  WgtSmem &ws = *reinterpret_cast<WgtSmem *>(smem_raw);
  uint32_t *tmem_slot = row_sm ? &rs.tmem_base : &ws.tmem_base;
  if (tid == 0) {
    if (row_sm) {
      mbar_init(smem_u32(&rs.bar_load), 1); mbar_init(smem_u32(&rs.x_full), 1); mbar_init(smem_u32(&rs.x_empty), 1); mbar_init(smem_u32(&rs.w1_full), 1);
      for (int i = 0; i < 2; ++i) {
        mbar_init(smem_u32(&rs.acc_free[i]), 4);  // the four warps of the group that read the half
        mbar_init(smem_u32(&rs.dh_ready[i]), 4);
        mbar_init(smem_u32(&rs.tile_done[i]), 4);
        for (int h = 0; h < 2; ++h) { mbar_init(smem_u32(&rs.acc_full[i][h]), 1); mbar_init(smem_u32(&rs.hid_ready[i][h]), 4); }
      }
    } else {
      for (int s = 0; s < kMaxStages; ++s) {
        mbar_init(smem_u32(&ws.full[s]), 1);
        mbar_init(smem_u32(&ws.empty[s]), w2_sm ? 1 + kConsumerWarps : 1);
      }
      mbar_init(smem_u32(&ws.done), 1);
      mbar_init(smem_u32(&ws.drained), kConsumerWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (row_sm) {  // the x tile: zeros, and the column of ones behind the features; the dhead tiles' upper columns: zeros
    for (int i = tid; i < static_cast<int>(sizeof(rs.x) / 16); i += kThreads) sts_zero16(smem_u32(rs.x) + 16u * i);
    for (int i = tid; i < static_cast<int>(sizeof(rs.dhead) / 16); i += kThreads) sts_zero16(smem_u32(rs.dhead) + 16u * i);
    __syncthreads();
    if (tid < kR) sts_u16(smem_u32(rs.x) + a_offset<kK1>(tid, a.net.D), 0x3F80);
    fence_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;
  if (row_sm) {
    if (tid == 0) {  // everything but W1 stays for the whole run; with one slab W1 does too
      constexpr uint32_t kChunk = 16384;
      const uint32_t first = a.net.slabs == 1 ? 0u : kImgW2;
      const unsigned char *rest = a.image + static_cast<size_t>(a.net.slabs) * kImgW2 - kImgW2;
      mbar_expect_tx(smem_u32(&rs.bar_load), kImgBytes - first);
      for (uint32_t o = first; o < kImgBytes; o += kChunk)
        bulk_load(smem_u32(rs.img + o), (o < kImgW2 ? a.image : rest) + o, min(kChunk, kImgBytes - o), smem_u32(&rs.bar_load));
    }
    ok = mbar_wait(smem_u32(&rs.bar_load), 0);
    ok = __syncthreads_and(ok) != 0;
    if (ok) ok = row_role<U>(a, rs, tmem);
    ok = __syncthreads_and(ok) != 0;
    if (tid <= kActions) {
      float s = 0.0f;
      for (int w = 0; w < 8; ++w) s += rs.red[w][tid];
      a.part_head[static_cast<size_t>(bid) * 8 + tid] = ok ? s : 0.0f;
    }
  } else if (w2_sm) {
    ok = weight_role<0, false>(a, ws, tmem, bid - sp.n_row, sp.n_w2, 0);
  } else {
    const int i = bid - sp.n_row - sp.n_w2, group = i / sp.n_w1, slab0 = group * sp.per_group;
    const int rank = i - group * sp.n_w1, ns = min(sp.per_group, a.net.slabs - slab0);
    if (group == 0) ok = ns == 1 ? weight_role<1, true>(a, ws, tmem, rank, sp.n_w1, 0) : weight_role<2, true>(a, ws, tmem, rank, sp.n_w1, 0);
    else ok = ns == 1 ? weight_role<1, false>(a, ws, tmem, rank, sp.n_w1, slab0) : weight_role<2, false>(a, ws, tmem, rank, sp.n_w1, slab0);
  }
  if (!ok && tid == 0) atomicExch(a.status, kStatusTimeout);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// The net's gradient from the roles' partial sums, each in rank order.  Thread i reads element i of the partial sums (whole
// lines) and finds where it belongs.
__global__ void reduce256_kernel(float *__restrict__ grad, Net256 net, Split sp, const float *__restrict__ part_w2, const float *__restrict__ part_w1p,
                                 const float *__restrict__ part_head, TermSums terms) {
  if (blockIdx.x == 0) loss_terms(terms);
  const int n_w2 = static_cast<int>(kPartW2), per_w1 = static_cast<int>(part_w1(sp.per_group)), n_w1 = sp.groups * per_w1, total = n_w2 + n_w1 + kActions + 1;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const float *src;
    size_t stride, out;
    int n;
    if (i < n_w2) {
      src = part_w2 + i; stride = kPartW2; n = sp.n_w2;
      const int c = (i / (4 * kH)) * 4 + (i & 3), unit = (i >> 2) % kH;
      out = i < kH * kH ? net.W2 + static_cast<size_t>(unit) * kH + c : net.b2 + (i - kH * kH);
    } else if (i < n_w2 + n_w1) {
      const int group = (i - n_w2) / per_w1, j = i - n_w2 - group * per_w1, x = j / (kH * kK1);
      const int e = x < sp.per_group ? j - x * (kH * kK1) : j - sp.per_group * (kH * kK1);
      const int c = (e / (4 * kH)) * 4 + (e & 3), unit = (e >> 2) % kH, slab = group * sp.per_group + x;
      stride = per_w1; n = sp.n_w1;
      src = part_w1p + static_cast<size_t>(group) * sp.n_w1 * stride + j;
      if (x == sp.per_group) {
        if (group > 0 || c > kActions || (c < kActions ? !net.has_actor : !net.has_value)) continue;
        out = c < kActions ? net.Wa + static_cast<size_t>(c) * kH + unit : net.Wv + unit;
      } else {
        if (slab >= net.slabs || c > net.D || (c == net.D && slab > 0)) continue;
        out = c == net.D ? net.b1 + unit : net.W1 + static_cast<size_t>(unit) * net.w1_ld + static_cast<size_t>(slab) * net.D + c;
      }
    } else {
      const int k = i - n_w2 - n_w1;
      if (k < kActions ? !net.has_actor : !net.has_value) continue;
      src = part_head + k; stride = 8; n = sp.n_row;
      out = k < kActions ? net.ba + k : net.bv;
    }
    float s = 0.0f;
#pragma unroll 8
    for (int c = 0; c < n; ++c) s += src[c * stride];
    grad[out] = s;
  }
}

// SMs per role, in proportion to weights that come from timing splits of 148 SMs (the roles slow one another through L2, so the
// cycles that each takes by itself, see above, are no guide).  One gradient, us:
//   one slab (8 agents, 4096 environments x 64 steps; the rule gives 102 row, 22 W2, 24 W1 SMs: 1850)
//     W2 SMs 16 / 19 / 22 / 25 / 28 with 24 W1: 2171 / 1912 / 1850 / 1803 / 1917;  W1 18 / 21 / 27 / 30 with 22 W2: 2112 / 1863 / 1807 / 2000
//   four slabs (actor and critic of 4 agents, 4096 x 64; the rule gives the critic 100, 12 and 2 x 18: 1470)
//     W2 SMs 6 / 9 / 15 / 18: 1714 / 1500 / 1465 / 1484;  W1 12 / 15 / 21 / 24 per pair of slabs: 1557 / 1472 / 1473 / 1510
// Too few of a role costs much, a few more than the rule gives little either way (full batches, under the power cap: within 5 %).
Split make_split(long long tiles, int sms, int slabs) {
  Split s{};
  s.n_tiles = static_cast<int>(tiles);
  s.per_group = slabs == 1 ? 1 : 2;
  s.groups = (slabs + s.per_group - 1) / s.per_group;
  const double row = 10.5 + 3.0 * (slabs - 1), w2 = 2.3, w1 = 2.5 + 0.9 * (s.per_group - 1);
  const double all = row + w2 + w1 * s.groups;
  s.n_w2 = static_cast<int>(sms * w2 / all + 0.5);
  s.n_w1 = static_cast<int>(sms * w1 / all + 0.5);
  auto within = [&](int v) { return static_cast<int>(v < 1 ? 1 : (v > tiles ? tiles : v)); };
  s.n_w2 = within(s.n_w2);
  s.n_w1 = within(s.n_w1);
  s.n_row = within(sms - s.n_w2 - s.groups * s.n_w1);
  s.n_slots = static_cast<int>(tiles < 3LL * s.n_row ? tiles : 3LL * s.n_row);
  return s;
}

size_t round256(size_t n) { return (n + 255) / 256 * 256; }
struct Scratch256 { size_t image, counters, terms, part_head, part_w2, part_w1, bytes; };
Scratch256 scratch_layout(const Split &s, int slabs) {
  Scratch256 L{};
  size_t off = 0;
  auto take = [&](size_t n) { const size_t at = off; off += round256(n); return at; };
  L.image = take(static_cast<size_t>(slabs - 1) * kImgW2 + kImgBytes);
  L.counters = take(sizeof(uint32_t) * 3 * s.n_slots);
  L.terms = take(sizeof(double) * 3 * 8 * s.n_row);
  L.part_head = take(sizeof(float) * 8 * s.n_row);
  L.part_w2 = take(sizeof(float) * kPartW2 * s.n_w2);
  L.part_w1 = take(sizeof(float) * part_w1(s.per_group) * s.n_w1 * s.groups);
  L.bytes = off;
  return L;
}

}  // namespace

bool ppo_tc256_supported(const mava_config_t &cfg, int D) { return cfg.hidden == kH && D + 1 <= kK1 && D > 64; }

Tc256Need ppo_tc256_need(long long n_rows, int sms, int slabs) {
  const Split s = make_split((n_rows + kR - 1) / kR, sms, slabs);
  return Tc256Need{scratch_layout(s, slabs).bytes, static_cast<size_t>(s.n_slots) * slot_bytes(slabs)};
}

cudaError_t launch_ppo_net_tc256(mava_rollout *h, const float *params_dev, const Tc256Net &desc, const UpdRows &rows, const UpdHyper &hp,
                                 const Moments &adv, const double *adv_stats, void *scratch, void *ring, int sms, float *grad, TermSums &terms) {
  Upd256Args a{};
  Net256 &net = a.net;
  net.W1 = desc.W1; net.b1 = desc.b1; net.W2 = desc.W2; net.b2 = desc.b2; net.Wa = desc.Wa; net.ba = desc.ba; net.Wv = desc.Wv; net.bv = desc.bv;
  net.D = h->D; net.slabs = desc.slabs; net.w1_ld = desc.slabs * h->D; net.has_actor = desc.has_actor ? 1 : 0; net.has_value = desc.has_value ? 1 : 0;
  a.sp = make_split((rows.n + kR - 1) / kR, sms, desc.slabs);
  const Scratch256 L = scratch_layout(a.sp, desc.slabs);
  unsigned char *base = static_cast<unsigned char *>(scratch);
  a.image = base + L.image;
  a.rows = rows; a.hp = hp; a.adv_stats = adv_stats;
  a.ring = static_cast<unsigned char *>(ring);
  a.full = reinterpret_cast<uint32_t *>(base + L.counters); a.x_full = a.full + a.sp.n_slots; a.read = a.x_full + a.sp.n_slots;
  a.part_w2 = reinterpret_cast<float *>(base + L.part_w2); a.part_w1 = reinterpret_cast<float *>(base + L.part_w1);
  a.part_head = reinterpret_cast<float *>(base + L.part_head);
  a.term_partial = reinterpret_cast<double *>(base + L.terms);
  a.status = h->d_status;
  if (desc.has_actor) { terms.actor = a.term_partial; terms.n_actor_part = 8 * a.sp.n_row; }
  if (desc.has_value) { terms.value = a.term_partial; terms.n_value_part = 8 * a.sp.n_row; }
  cudaError_t err = launch_prologue(adv, Prep256{params_dev, base + L.image, net, a.full, 3 * a.sp.n_slots}, 64, h->stream);
  if (err != cudaSuccess) return err;
  const auto kern = rows_need_64_bits(rows, rows.n) ? ppo_update256_kernel<uint64_t> : ppo_update256_kernel<uint32_t>;
  err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemBytes));
  if (err != cudaSuccess) return err;
  void *args[] = {&a};
  const int grid = a.sp.n_row + a.sp.n_w2 + a.sp.groups * a.sp.n_w1;
  err = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kern), dim3(grid), dim3(kThreads), args, kSmemBytes, h->stream);
  if (err != cudaSuccess) return err;
  reduce256_kernel<<<2 * sms, 256, 0, h->stream>>>(grad, net, a.sp, a.part_w2, a.part_w1, a.part_head, desc.has_value ? terms : TermSums{});
  h->launches += 3;
  return cudaGetLastError();
}

}  // namespace mava

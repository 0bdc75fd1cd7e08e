// Rollout with the recurrent policy on the tensor cores (sm_100a, tcgen05; H = 64): the fused loop of rollout_tc.cu
// with a gated recurrent unit between the embedding and the heads.  One persistent CTA per SM: eight epilogue warps (32 rows x 32
// units each; those of the first half also keep the environments in registers, env.cuh, thread = row = tensor-memory lane) and a
// helper warp for every 32 rows.  Per step:
//   1. the bf16 observation rows into the A tile;
//   2. MMAs: embedding pre-activation x . W1^T, and straight away the hidden part of the three gates from the carried
//      hidden tile (h . Whr^T, h . Whz^T into the r|z accumulator, h . Whn^T into its own); an event for the helper, which draws the
//      step's uniform, stores the last step's outputs and writes the fp32 observation rows;
//   3. epilogue: e = relu(. + b1) as a bf16 tile; MMAs: the input part e . Wir^T, e . Wiz^T on top of the r|z
//      accumulator, e . Win^T into its own;
//   4. gate epilogue in fp32: r, z, n, h' = (1 - z) n + z h; h' rounded to bf16 replaces the row of the hidden tile (the carried state
//      is that bf16 number, as in the oracle's bf16-operand mode);
//   5. heads MMA on the new hidden tile; sampler; warp-level transition; a finished episode zeroes its agents' rows
//      of the hidden tile.
// What bounds it (10x10, 5001 environments: one tile of 102 rows per SM, 101 steps): the step's chain, of which the gate epilogue is
// 3.1 k cycles at the least: six special-function operations a unit, 16 a cycle and SM.  (Sharing reciprocals, 4.25 a unit, takes the
// collection to 493 us but rounds differently, and once in a while that moves an action.)  The epilogues read 16x256b fragments, so
// a thread has the same eight units of four rows: biases and carried state stay in registers.  With stores, draws, fp32 rows
// and biases on the chain a step took 9.8 k cycles; 592 -> 544 us.
// The bootstrap step (t == T) writes h' into the embedding tile instead, so the carried state is not advanced.
// The hidden vectors live in a per-handle fp32 array between runs.  Every mbarrier wait is bounded.
#include <cuda_bf16.h>

#include "common.cuh"
#include "env.cuh"
#include "launch.cuh"
#include "layout.h"
#include "tc_common.cuh"

namespace mava {
namespace {

constexpr int kRH = 64;    // hidden width
constexpr int kRecMain = 256, kRecThreads = kRecMain + kTileRows;  // epilogues (a warp has 32 rows x 32 units); a helper warp per 32 rows
constexpr int kRK1 = 80;   // input width, padded (D = 79, 80)

// weight image
constexpr uint32_t kW1 = 0, kWih = kW1 + kRH * kRK1 * 2, kWhh = kWih + 3 * kRH * kRH * 2, kWh = kWhh + 3 * kRH * kRH * 2;
constexpr uint32_t kB1 = kWh + kHeadRows * kRH * 2, kBrz = kB1 + kRH * 4, kBin = kBrz + 2 * kRH * 4, kBhn = kBin + kRH * 4, kBh = kBhn + kRH * 4;
constexpr uint32_t kRecImage = kBh + 32;
static_assert(kRecImage % 16 == 0, "bulk copy");

constexpr uint32_t kColE = 0, kColRZ = 64, kColIn = 192, kColHn = 256, kRecTmem = 512;  // the heads reuse kColE

// An event's record (words): entities, step / cap, then the outputs of the step before.  48 bytes: the 16-byte accesses of eight
// consecutive rows meet no bank conflict.
constexpr int kEvFrac = 6, kEvValue = 7, kEvLogp = 8, kEvReward = 9, kEvAction = 10 /* | done << 8 */, kEvPitch = 12;

template <int N>
struct RecTcSmem {
  static constexpr int D = kObsFixed + N;
  alignas(128) unsigned char img[(kRecImage + 127) / 128 * 128];
  alignas(128) unsigned char a[(kTileRows / 8) * (kRK1 / 8) * kALbo];  // bf16 observations (padded core-matrix pitch)
  alignas(128) unsigned char emb[kTileRows * kRH * 2];                 // bf16 embedding; the bootstrap step's h'
  alignas(128) unsigned char hid[kTileRows * kRH * 2];                 // bf16 hidden vectors, carried
  alignas(128) float stage[kTileRows * D];                             // fp32 observation block in the global layout
  alignas(16) uint32_t event[kTileRows * kEvPitch];
  float uniform[kTileRows];                                            // of the step's draw
  unsigned char over[kTileRows];                                       // the row's episode ended with the last step
  alignas(8) uint64_t load_bar, emb_bar, gate_bar, head_bar, ev_full[4], ev_empty[4];
  int quit[4];  // set before the last event of a warp that gave up
  uint32_t tmem_base;
};

__global__ void prep_rec_tc_kernel(const float *params, unsigned char *image, ParamLayout L, int D) {
  wait_for_predecessor();
  auto bf = [&](uint32_t off) { return reinterpret_cast<__nv_bfloat16 *>(image + off); };
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  for (int i = tid; i < kRH * kRK1; i += nth) {
    const int n = i / kRK1, k = i - n * kRK1;
    bf(kW1)[canon_offset(n, k, kRK1) / 2] = __float2bfloat16_rn(k < D ? __ldcg(params + L.W1 + static_cast<size_t>(n) * D + k) : 0.0f);
  }
  for (int i = tid; i < 3 * kRH * kRH; i += nth) {
    const int n = i / kRH, k = i - n * kRH;
    bf(kWih)[canon_offset(n, k, kRH) / 2] = __float2bfloat16_rn(__ldcg(params + L.Wih + i));
    bf(kWhh)[canon_offset(n, k, kRH) / 2] = __float2bfloat16_rn(__ldcg(params + L.Whh + i));
  }
  for (int i = tid; i < kHeadRows * kRH; i += nth) {
    const int n = i / kRH, k = i - n * kRH;
    float v = 0.0f;
    if (n < kActions) v = __ldcg(params + L.Wa + static_cast<size_t>(n) * kRH + k);
    else if (n == kActions) v = __ldcg(params + L.Wv + k);
    bf(kWh)[canon_offset(n, k, kRH) / 2] = __float2bfloat16_rn(v);
  }
  float *b1 = reinterpret_cast<float *>(image + kB1), *brz = reinterpret_cast<float *>(image + kBrz),
        *bin = reinterpret_cast<float *>(image + kBin), *bhn = reinterpret_cast<float *>(image + kBhn), *bh = reinterpret_cast<float *>(image + kBh);
  for (int i = tid; i < kRH; i += nth) {
    b1[i] = __ldcg(params + L.b1 + i);
    brz[i] = __ldcg(params + L.bih + i) + __ldcg(params + L.bhh + i);                      // r: both parts' biases
    brz[kRH + i] = __ldcg(params + L.bih + kRH + i) + __ldcg(params + L.bhh + kRH + i);    // z
    bin[i] = __ldcg(params + L.bih + 2 * kRH + i);
    bhn[i] = __ldcg(params + L.bhh + 2 * kRH + i);
  }
  if (tid < 8) bh[tid] = tid < kActions ? __ldcg(params + L.ba + tid) : (tid == kActions ? __ldcg(params + L.bv) : 0.0f);
}

__device__ __forceinline__ uint64_t rdesc(uint32_t tile, int C, int k) { return smem_desc(tile + k * 256, 128, C * 16); }
// Branch-free forms (ex2.approx and rcp.approx: a few 1e-7, far below the bf16 step the result is rounded to), so
// that the compiler can interleave the units of a row.  The arguments are clamped to where the functions have long saturated in
// binary32, which keeps the exponential finite.
__device__ __forceinline__ float sigm(float v) { return __fdividef(1.0f, 1.0f + __expf(-fminf(fmaxf(v, -30.0f), 30.0f))); }
__device__ __forceinline__ float tanh_fast(float v) { return 1.0f - __fdividef(2.0f, 1.0f + __expf(2.0f * fminf(fmaxf(v, -15.0f), 15.0f))); }
__device__ __forceinline__ uint4 lds_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ void loaded16(uint32_t *r) {  // (after the wait: what the loads brought is not touched before)
#pragma unroll
  for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));
}
// The counterpart of stmatrix4.
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t *r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

template <int N, int F>
__global__ void __launch_bounds__(kRecThreads, 1)
rollout_rec_tc_kernel(RolloutArgs a, const unsigned char *image, float *hidden, int ept, int n_tiles) {
  constexpr int D = kObsFixed + N, K1 = kRK1, H = kRH;
  constexpr int EPW = 32 / N, RPW = EPW * N;
  static_assert(N + F <= kEvFrac, "an event's record");
  static_assert((RPW * D) % 4 == 0, "a warp's fp32 rows are whole 16-byte pieces");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  RecTcSmem<N> &sm = *reinterpret_cast<RecTcSmem<N> *>(smem_raw);
  const int tid = threadIdx.x, row = tid & (kTileRows - 1), warp = row >> 5, lane = tid & 31;  // (warp: of the row)
  const int role = __shfl_sync(0xFFFFFFFFu, tid >> 7, 0);  // 0, 1: epilogue halves (0 keeps the environments too); 2: helpers
  const bool first_warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0) == 0;  // (uniform to the compiler: this warp issues the MMAs)
  const uint32_t load_bar = smem_u32(&sm.load_bar), emb_bar = smem_u32(&sm.emb_bar), gate_bar = smem_u32(&sm.gate_bar), head_bar = smem_u32(&sm.head_bar);
  const uint32_t ev_full = smem_u32(&sm.ev_full[warp]), ev_empty = smem_u32(&sm.ev_empty[warp]);
  if (tid == 0) {
    mbar_init(load_bar, 1); mbar_init(emb_bar, 1); mbar_init(gate_bar, 1); mbar_init(head_bar, 1);
    for (int i = 0; i < 4; ++i) { sm.quit[i] = 0; mbar_init(smem_u32(&sm.ev_full[i]), 1); mbar_init(smem_u32(&sm.ev_empty[i]), 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (first_warp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)), "r"(kRecTmem) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const uint32_t a_addr = smem_u32(sm.a), emb_addr = smem_u32(sm.emb), hid_addr = smem_u32(sm.hid), stage_addr = smem_u32(sm.stage);
  for (int i = tid; i < static_cast<int>(sizeof(sm.a) / 16); i += kRecThreads) sts_zero16(a_addr + 16u * i);
  dependents_may_start();
  wait_for_predecessor();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0) {
    mbar_expect_tx(load_bar, kRecImage);
    for (uint32_t o = 0; o < kRecImage; o += 16384) bulk_load(smem_u32(sm.img + o), image + o, min(16384u, kRecImage - o), load_bar);
  }
  bool timed_out = !mbar_wait(load_bar, 0);
  timed_out = __syncthreads_or(timed_out) != 0;

  const uint32_t tmem = sm.tmem_base;
  const size_t M = static_cast<size_t>(a.env.n_envs) * N;
  const int le = warp * EPW + lane / N, ag = lane % N, crow = le * N + ag;
  const uint32_t event_addr = smem_u32(sm.event) + static_cast<uint32_t>(row * kEvPitch * 4);
  uint32_t ev_phase = 0;  // of the next event

  if (role == 2) {
    // ---- helper warp: event k of a tile has the state that step k acts on and the outputs of step k - 1.  It draws the step's uniform,
    // stores the outputs and writes the fp32 observation rows, which leave as a bulk copy of its own.
    const uint32_t chunk = stage_addr + static_cast<uint32_t>(warp * RPW * D * 4);
    constexpr int kChunk16 = RPW * D / 4;
    bool bulk_pending = false, stop = timed_out;  // (bulk_pending: lane 0)
    for (int it = 0; !stop; ++it) {
      const int tile = it * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);
      if (tile >= n_tiles) break;
      const int e0 = tile * ept, n_env = min(ept, a.env.n_envs - e0);
      const bool active = lane < RPW && le < n_env;
      const int n_mine = max(0, min(RPW, n_env * N - warp * RPW));  // rows of this warp
      const uint32_t env_id = static_cast<uint32_t>(a.env.first_env + e0 + le);
      for (int k = 0; k <= a.T + 1; ++k) {
        stop = !mbar_wait_warp(ev_full, ev_phase);
        ev_phase ^= 1;
        if (stop) timed_out = true;
        if (stop || *reinterpret_cast<volatile int *>(&sm.quit[warp])) { stop = true; break; }
        uint32_t rec[kEvPitch];
#pragma unroll
        for (int q = 0; q < kEvPitch; q += 4) {
          const uint4 v = lds_v4(event_addr + 4u * q);
          rec[q] = v.x; rec[q + 1] = v.y; rec[q + 2] = v.z; rec[q + 3] = v.w;
        }
        if (active && k < a.T)
          sts_f32(smem_u32(&sm.uniform[row]), action_uniform(a.env, a.t_global0 + static_cast<uint32_t>(k), env_id, static_cast<uint32_t>(ag)));
        __syncwarp();
        if (lane == 0) mbar_arrive(ev_empty);
        if (k >= 1 && active) {
          const size_t at = static_cast<size_t>(k - 1) * M + static_cast<size_t>(e0) * N + crow;
          a.buf.values[at] = __uint_as_float(rec[kEvValue]);
          if (k - 1 < a.T) {  // (the bootstrap step has a value only)
            a.buf.actions[at] = static_cast<int32_t>(rec[kEvAction] & 0xFFu);
            a.buf.logp[at] = __uint_as_float(rec[kEvLogp]);
            a.buf.rewards[at] = __uint_as_float(rec[kEvReward]);
            if (ag == 0) a.buf.dones[static_cast<size_t>(k - 1) * a.env.n_envs + e0 + le] = static_cast<uint8_t>(rec[kEvAction] >> 8);
          }
        }
        if (k < a.T && n_mine > 0) {
          if (bulk_pending) { bulk_store_wait_read(); bulk_pending = false; }
          __syncwarp();
          for (int i = lane; i < kChunk16; i += 32) sts_zero16(chunk + 16u * i);
          __syncwarp();
          if (active) {
            EnvRegs<N, F> env;
#pragma unroll
            for (int q = 0; q < N + F; ++q) env.ent[q] = rec[q];
            write_row_f32<N, F, 0>(env, a.env, ag, __uint_as_float(rec[kEvFrac]), chunk + 4u * static_cast<uint32_t>(lane * D));
          }
          fence_async_smem();
          __syncwarp();
          float *obs_dst = a.buf.obs + (static_cast<size_t>(k) * M + static_cast<size_t>(e0) * N + warp * RPW) * D;
          const int count = n_mine * D;
          if (whole_pieces16(obs_dst, count)) {
            if (lane == 0) { bulk_store(obs_dst, chunk, static_cast<uint32_t>(count) * 4u); bulk_pending = true; }
          } else {
            for (int i = lane; i < count; i += 32) obs_dst[i] = lds_f32(chunk + 4u * i);
          }
        }
      }
    }
  } else {
  const int half = role;
  auto rows_sync = [] { asm volatile("bar.sync 2, %0;" ::"n"(kTileRows) : "memory"); };  // the warps that keep the environments
  auto main_any = [](bool pred) {  // all epilogue warps; whether one of them has given up
    uint32_t out;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}"
                 : "=r"(out) : "r"(static_cast<uint32_t>(pred)), "n"(kRecMain) : "memory");
    return out != 0;
  };
  const uint32_t lane_off = static_cast<uint32_t>(warp * 32) << 16;
  const uint32_t w1 = smem_u32(sm.img + kW1), wih = smem_u32(sm.img + kWih), whh = smem_u32(sm.img + kWhh), wh = smem_u32(sm.img + kWh);
  const float *bhd = reinterpret_cast<const float *>(sm.img + kBh);
  const uint32_t my_hid = hid_addr + static_cast<uint32_t>((row >> 3) * (H * 16) + (row & 7) * 16);  // chunk c of this row: + 128 c
  // the matrices of this warp's rows and units (stmatrix4): row group 2 c + {0, 1}, chunk j + {0, 1} at + c * 2 * H * 16 + j * 128
  const uint32_t my_at = static_cast<uint32_t>((warp * 4 + ((lane >> 3) & 1)) * (H * 16) + (half * 4 + (lane >> 4)) * 128 + (lane & 7) * 16);
  const int u0 = 32 * half, first_row = warp * 32 + (lane >> 2);  // this thread's units: u0 + 8 j + 2 (lane % 4) + {0, 1}; rows: + 8 k, k = 0..3
  float2 b1[4], br[4], bz[4], bi[4], bh[4];
  {
    const float *src = reinterpret_cast<const float *>(sm.img) + u0 + 2 * (lane & 3);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      b1[j] = *reinterpret_cast<const float2 *>(src + kB1 / 4 + 8 * j);
      br[j] = *reinterpret_cast<const float2 *>(src + kBrz / 4 + 8 * j);
      bz[j] = *reinterpret_cast<const float2 *>(src + kBrz / 4 + H + 8 * j);
      bi[j] = *reinterpret_cast<const float2 *>(src + kBin / 4 + 8 * j);
      bh[j] = *reinterpret_cast<const float2 *>(src + kBhn / 4 + 8 * j);
    }
  }
  uint32_t phase = 0;  // of the three products' barriers: one phase per step

  for (int it = 0; !timed_out; ++it) {
    const int tile = it * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);
    if (tile >= n_tiles) break;
    const int e0 = tile * ept;
    const int n_env = min(ept, a.env.n_envs - e0);
    const bool mine = lane < RPW && le < n_env;   // the row exists
    const bool active = mine && half == 0;        // and this thread keeps its environment
    const int base = active ? lane - ag : lane;
    const uint32_t env_id = static_cast<uint32_t>(a.env.first_env + e0 + le);
    EnvRegs<N, F> env;
    if (active) {
      load_env(env, a.state[e0 + le]);
    } else {
#pragma unroll
      for (int k = 0; k < N + F; ++k) env.ent[k] = 0;
      env.step = 0; env.episode = 0; env.total = 1;
    }
    {  // this row's hidden vector into the hidden tile (a carried state is a bf16 number: the conversion is exact)
      const float *src = hidden + (static_cast<size_t>(e0) * N + crow) * H;
#pragma unroll
      for (int q = 0; q < H / 16; ++q) {
        const int c = half * (H / 16) + q;
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) pk[e] = mine ? pack_bf16(src[8 * c + 2 * e], src[8 * c + 2 * e + 1]) : 0u;
        sts_v4(my_hid + 128u * c, pk[0], pk[1], pk[2], pk[3]);
      }
    }
    if (half == 0) sm.over[row] = 0;
    fence_async_smem();
    timed_out = main_any(timed_out);
    if (timed_out) break;
    uint32_t hk[2][8];  // this thread's part of the hidden tile: kept from step to step
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      ldmatrix4(hid_addr + my_at + static_cast<uint32_t>(c * 2 * H * 16), hk[c]);
      ldmatrix4(hid_addr + my_at + static_cast<uint32_t>(c * 2 * H * 16 + 256), hk[c] + 4);
    }
    float pend_value = 0.0f, pend_logp = 0.0f, pend_reward = 0.0f;
    int pend_action = 0;
    bool pend_done = false;
    auto publish = [&](float frac) {  // the next event for this warp's helper (whole warp)
      if (active) {
        uint32_t w[kEvPitch];
#pragma unroll
        for (int q = 0; q < kEvFrac; ++q) w[q] = q < N + F ? env.ent[q < N + F ? q : 0] : 0u;
        w[kEvFrac] = __float_as_uint(frac); w[kEvValue] = __float_as_uint(pend_value); w[kEvLogp] = __float_as_uint(pend_logp);
        w[kEvReward] = __float_as_uint(pend_reward); w[kEvAction] = static_cast<uint32_t>(pend_action) | (pend_done ? 0x100u : 0u);
        w[11] = 0u;
#pragma unroll
        for (int q = 0; q < kEvPitch; q += 4) sts_v4(event_addr + 4u * q, w[q], w[q + 1], w[q + 2], w[q + 3]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(ev_full);
    };
    auto await_helper = [&]() {  // it has taken the last event over (and drawn its step's uniform)
      timed_out |= !mbar_wait_warp(ev_empty, ev_phase);
      ev_phase ^= 1;
    };
    for (int t = 0; t <= a.T; ++t) {
      const bool last = t == a.T;
      const size_t row0 = static_cast<size_t>(t) * M + static_cast<size_t>(e0) * N;
      if (half == 0) {
        // 1. the bf16 observation rows
        float frac = 0.0f;
        if (active) {
          frac = step_fraction(env.step, a.env.cap);
          write_row_bf16<N, F, K1, false, 0, kALbo>(env, a.env, ag, frac, a_addr + a_offset<K1>(row, 0));
        }
        fence_async_smem();
        tc_fence_before();
        rows_sync();
        // 2. embedding pre-activation; hidden part of the gates (every warp has read these accumulators before the last step's heads)
        if (first_warp) {
          if (elect_one()) {
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < K1 / 16; ++k)
              mma_bf16(tmem + kColE, smem_desc(a_addr + k * 2 * kALbo, kALbo, (K1 / 8) * kALbo), rdesc(w1, K1, k), instr_desc(kTileRows, H), k > 0);
            mma_commit(emb_bar);
#pragma unroll
            for (int k = 0; k < H / 16; ++k) {
              mma_bf16(tmem + kColRZ, rdesc(hid_addr, H, k), rdesc(whh, H, k), instr_desc(kTileRows, 2 * H), k > 0);
              mma_bf16(tmem + kColHn, rdesc(hid_addr, H, k), rdesc(whh + 2 * H * H * 2, H, k), instr_desc(kTileRows, H), k > 0);
            }
          }
          __syncwarp();
        }
        publish(frac);
      }
      timed_out |= !mbar_wait_warp(emb_bar, phase);
      tc_fence_after();
      // 3. e = relu(. + b1) as a bf16 tile
      {
        uint32_t r[2][16];
        tmem_ld_16x32_nowait(tmem + kColE + lane_off + static_cast<uint32_t>(u0), r[0]);
        tmem_ld_16x32_nowait(tmem + kColE + lane_off + (16u << 16) + static_cast<uint32_t>(u0), r[1]);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t pk[8];
          loaded16(r[c]);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            pk[i] = relu_pack_bf16(__float_as_uint(__uint_as_float(r[c][2 * i]) + b1[i / 2].x), __float_as_uint(__uint_as_float(r[c][2 * i + 1]) + b1[i / 2].y));
          stmatrix4(emb_addr + my_at + static_cast<uint32_t>(c * 2 * H * 16), pk);
          stmatrix4(emb_addr + my_at + static_cast<uint32_t>(c * 2 * H * 16 + 256), pk + 4);
        }
      }
      fence_async_smem();
      tc_fence_before();
      if (main_any(timed_out)) { timed_out = true; break; }
      if (first_warp) {
        if (elect_one()) {
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < H / 16; ++k) {
            mma_bf16(tmem + kColRZ, rdesc(emb_addr, H, k), rdesc(wih, H, k), instr_desc(kTileRows, 2 * H), 1);
            mma_bf16(tmem + kColIn, rdesc(emb_addr, H, k), rdesc(wih + 2 * H * H * 2, H, k), instr_desc(kTileRows, H), k > 0);
          }
          mma_commit(gate_bar);
        }
        __syncwarp();
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)  // a finished episode leaves no memory behind (its rows of the tile are zero already)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          if (sm.over[first_row + 16 * c + 8 * k]) hk[c][k] = hk[c][2 + k] = hk[c][4 + k] = hk[c][6 + k] = 0u;
      timed_out |= !mbar_wait_warp(gate_bar, phase);
      tc_fence_after();
      // 4. gates (fp32) and the new hidden vector
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const uint32_t at = tmem + lane_off + (static_cast<uint32_t>(16 * c) << 16) + static_cast<uint32_t>(u0);
        uint32_t gr[16], gz[16], gi[16], gh[16], pk[8];
        tmem_ld_16x32_nowait(at + kColRZ, gr);
        tmem_ld_16x32_nowait(at + kColRZ + H, gz);
        tmem_ld_16x32_nowait(at + kColIn, gi);
        tmem_ld_16x32_nowait(at + kColHn, gh);
        tmem_ld_wait();
        loaded16(gr); loaded16(gz); loaded16(gi); loaded16(gh);
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // two neighbouring units of a row
          const int j = i / 2;
          float hn[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int x = 2 * i + e;
            const float hprev = __uint_as_float(e == 0 ? (hk[c][i] << 16) : (hk[c][i] & 0xFFFF0000u));
            const float r = sigm(__uint_as_float(gr[x]) + (e ? br[j].y : br[j].x));
            const float z = sigm(__uint_as_float(gz[x]) + (e ? bz[j].y : bz[j].x));
            const float n = tanh_fast(__uint_as_float(gi[x]) + (e ? bi[j].y : bi[j].x) + r * (__uint_as_float(gh[x]) + (e ? bh[j].y : bh[j].x)));
            hn[e] = (1.0f - z) * n + z * hprev;
          }
          pk[i] = pack_bf16(hn[0], hn[1]);
        }
        const uint32_t dst = (last ? emb_addr : hid_addr) + my_at + static_cast<uint32_t>(c * 2 * H * 16);
        stmatrix4(dst, pk);
        stmatrix4(dst + 256u, pk + 4);
        if (!last) {
#pragma unroll
          for (int i = 0; i < 8; ++i) hk[c][i] = pk[i];
        }
      }
      fence_async_smem();
      tc_fence_before();
      if (main_any(timed_out)) { timed_out = true; break; }
      const uint32_t this_phase = phase;
      phase ^= 1;
      if (half == 1) continue;
      // 5. heads on the new hidden vectors
      if (first_warp) {
        if (elect_one()) {
          tc_fence_after();
          const uint32_t src = last ? emb_addr : hid_addr;
#pragma unroll
          for (int k = 0; k < H / 16; ++k) mma_bf16(tmem + kColE, rdesc(src, H, k), rdesc(wh, H, k), instr_desc(kTileRows, kHeadRows), k > 0);
          mma_commit(head_bar);
        }
        __syncwarp();
      }
      await_helper();
      const float u = sm.uniform[row];
      timed_out |= !mbar_wait_warp(head_bar, this_phase);
      tc_fence_after();
      int action = 0;
      float hv[16];
      tmem_ld16(tmem + kColE + lane_off, hv);
#pragma unroll
      for (int k = 0; k <= kActions; ++k) hv[k] += bhd[k];
      if (active) {
        pend_value = hv[kActions];
        if (!last) {
          float m, sum;
          action = draw_action(hv, u, m, sum);
          if (a.forced) {
            action = a.forced[row0 + crow];
            if (action < 0 || action >= kActions) action = 0;
          }
          float la = hv[0];
#pragma unroll
          for (int k = 1; k < kActions; ++k) la = (action == k) ? hv[k] : la;
          pend_action = action;
          pend_logp = la - m - __logf(sum);
          if (a.write_logits) {
#pragma unroll
            for (int k = 0; k < kActions; ++k) a.buf.logits[(row0 + crow) * kActions + k] = hv[k];
          }
        }
      }
      tc_fence_before();
      if (last) break;
      bool done;
      step_env_warp<N, F>(env, a.env, env_id, ag, base, active, action, pend_reward, done);
      pend_done = done;
      sm.over[row] = active && done ? 1 : 0;
      if (active && done) {  // a finished episode leaves no memory behind
#pragma unroll
        for (int c = 0; c < H / 8; ++c) sts_zero16(my_hid + 128u * c);
      }
    }
    timed_out = main_any(timed_out);
    if (half == 0) {  // the last event: outputs only, or the word that there is none
      if (timed_out) *reinterpret_cast<volatile int *>(&sm.quit[warp]) = 1;
      publish(0.0f);
      if (!timed_out) await_helper();
    }
    if (!timed_out && mine) {
      float *dst = hidden + (static_cast<size_t>(e0) * N + crow) * H;
#pragma unroll
      for (int q = 0; q < H / 16; ++q) {
        const int c = half * (H / 16) + q;
        const uint4 hp = lds_v4(my_hid + 128u * c);
        const uint32_t hw[4] = {hp.x, hp.y, hp.z, hp.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          dst[8 * c + 2 * e] = __uint_as_float(hw[e] << 16);
          dst[8 * c + 2 * e + 1] = __uint_as_float(hw[e] & 0xFFFF0000u);
        }
      }
      if (active && ag == 0) store_env(env, a.state[e0 + le]);
    }
    timed_out = main_any(timed_out);  // the hidden tile is rewritten by the next tile's rows
  }
  }
  if (timed_out && lane == 0) atomicExch(a.status, kStatusTimeout);
  bulk_store_wait_all();
  tc_fence_before();
  __syncthreads();
  if (first_warp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kRecTmem) : "memory");
  }
}

template <int N, int F>
cudaError_t launch_rec_tc_variant(mava_rollout *h, const RolloutArgs &args) {
  constexpr int D = kObsFixed + N, EPT_MAX = 4 * (32 / N);
  auto kern = rollout_rec_tc_kernel<N, F>;
  const size_t smem = sizeof(RecTcSmem<N>);
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (err != cudaSuccess) return err;
  int sms = 0;
  err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
  if (err != cudaSuccess) return err;
  int ept = (h->cfg.n_envs + sms - 1) / sms;
  if (ept > EPT_MAX) ept = EPT_MAX;
  if (ept < 1) ept = 1;
  for (int e = ept; e <= EPT_MAX; ++e)  // tiles that start on 16-byte boundaries: the rows of each helper warp then leave as a bulk copy
    if ((e * N * D) % 4 == 0) { ept = e; break; }
  const int n_tiles = (h->cfg.n_envs + ept - 1) / ept;
  h->launches += 1;
  return launch_dependent(kern, n_tiles < sms ? n_tiles : sms, kRecThreads, smem, h->stream, args, static_cast<const unsigned char *>(h->d_wtc), h->d_hidden,
                          ept, n_tiles);
}

}  // namespace

size_t rec_tc_weight_bytes(const mava_config_t &) { return kRecImage; }

cudaError_t launch_rollout_rec_tc(mava_rollout *h, const float *params_dev, const RolloutArgs &args) {
  if (h->cfg.hidden != kRH || h->D > kRK1) return cudaErrorNotSupported;
  // 48 blocks: one element of each gate matrix per thread
  cudaError_t err = launch_dependent(prep_rec_tc_kernel, 48, 256, 0, h->stream, params_dev, static_cast<unsigned char *>(h->d_wtc),
                                     param_layout(h->cfg, h->D, 1), h->D);
  h->launches += 1;
  if (err != cudaSuccess) return err;
  switch (h->variant) {
    case 5: return launch_rec_tc_variant<2, 2>(h, args);
    case 6: return launch_rec_tc_variant<3, 3>(h, args);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace mava

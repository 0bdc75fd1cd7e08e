// Small-batch form of the bf16 tensor-core rollout (H = 128), included by rollout_tc.cu.
//
// When one SM gets at most RB = 16 or 32 agent rows, a 128-row tile would spend its MMAs and
// epilogues on empty rows while the per-step chain (three dependent MMA round trips) is all that
// counts.  Here the operands change places: the weights are the M = 128 operand (one hidden unit
// per tensor-memory lane), the tile's rows are the N = RB operand, so an epilogue handles RB instead of 128 columns per
// thread.  The weights stay in tensor memory for the whole run: an MMA of N = 16 whose A operand comes from there issues in
// 13 cycles, from shared memory it takes 40 to 75 (streaming the 4 KB of A), and a step has 23 of them.
// The products and their order of accumulation (bias tile first, then K in ascending steps) are
// those of the 128-row kernel, and so are the results.
//   thread j < 128: hidden unit j in the epilogues (tensor-memory lane j);
//   threads 0 .. RB-1 (warp 0): also agent row j of the tile: sampler, transition, the bf16 observation row (env.cuh);
//   warp 3: issues the MMAs;
//   warp 4: everything that the step's chain does not wait for: the outputs of the step before, the fp32 observation rows
//   and their bulk copy, the uniforms of the step after next.  Warp 0 hands it a record per row and step (an event) through
//   two buffers; event k is published while step k's first layer runs.
// Same weight image as the 128-row kernel.
// What bounds it is the chain of a step: observation row, three MMA round trips of 0.4 to 0.5 k cycles with their epilogues, sampler,
// transition.  With the weights in shared memory and the fp32 rows, stores and draws spread over warps 0 to 3 a step took 4.0 k
// cycles (8x8-2p-2f, 1024 environments, T = 128: collection 280 us, evaluation block 180 us); as it stands 235 and 135 to 145 us.
// Warehouse, 10x10, 740 and 1480 environments x 64 steps: 172 and 174 us in the 128-row form, 131 and 147 here.
#pragma once

template <int N, int H, int RB>
struct SmallShape {
  using S = TcShape<N, H>;
  static_assert(H == kTileRows, "the hidden width is the M of the MMA");
  static_assert(RB == 16 || RB == 32, "rows per tile: one tensor-memory load of 16 or 32 columns");
  static constexpr int D = S::D, K1 = S::K1;
  static constexpr int EPT_MAX = RB / N;     // environments per tile
  static constexpr int ROWS = EPT_MAX * N;   // agent rows per tile, all in warp 0
  // B operands (rows x K, K-major, core matrices 144 bytes apart as in a_offset)
  static constexpr uint32_t X_BYTES = (RB / 8) * (K1 / 8) * kALbo;
  static constexpr uint32_t HT_BYTES = (RB / 8) * (H / 8) * kALbo;
  static constexpr uint32_t STAGE_BYTES = (ROWS * D * 4 + 15) / 16 * 16;
  // tensor-memory columns: accumulators, then the A operands (two bf16 per column)
  static constexpr int ACC_COL = 0, HEAD_COL = 32, W1_COL = 64, B1_COL = W1_COL + K1 / 2, W2_COL = B1_COL + 8, B2_COL = W2_COL + H / 2,
                       WH_COL = B2_COL + 8, TMEM_COLS = 256;
  static_assert(WH_COL + H / 2 <= TMEM_COLS, "tensor memory");
  static constexpr int THREADS = kGroupThreads + 32;
};

// What warp 0 tells warp 4 about a row (words): the environment's entities, step / cap, then the outputs of the step before.
constexpr int kEvFrac = 8, kEvAction = 9, kEvLogp = 10, kEvValue = 11, kEvReward = 12, kEvDone = 13, kEvLogit = 14, kEvPitch = 20;

template <int N, int F, int H, int RB>
struct SmallSmem {
  using S = TcShape<N, H>;
  using Q = SmallShape<N, H, RB>;
  alignas(128) unsigned char weights[S::IMAGE_BYTES];
  alignas(128) unsigned char x[Q::X_BYTES];         // bf16 observations, N operand of layer 1
  alignas(128) unsigned char ht[Q::HT_BYTES];       // bf16 hidden activations, N operand of layer 2 and of the heads
  alignas(128) unsigned char stage[Q::STAGE_BYTES]; // fp32 observation block in the global layout
  alignas(16) float logit[RB * 8];                  // heads' outputs, transposed for the row threads
  alignas(16) uint32_t event[2][RB * kEvPitch];
  float uniform[4][RB];                             // uniforms of the action draws, by step mod 4
  alignas(8) uint64_t mma_bar, load_bar, ev_full[2], ev_empty[2];
  uint32_t tmem_base;
  int abort;
};

// Accumulator columns 0 .. RB-1 of this thread's lane.
template <int RB>
__device__ __forceinline__ void small_tmem_ld(uint32_t taddr, float *v) {
  if constexpr (RB == 16) {
    tmem_ld16(taddr, v);
  } else {
    uint32_t r[32];
    tmem_ld32_nowait(taddr, r);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
  }
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t *r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]),
               "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// Row `unit` of an operand image (K columns, canonical layout) into this thread's lane of tensor memory; rows from `rows` on are zero.
template <int K>
__device__ __forceinline__ void operand_to_tmem(uint32_t image, uint32_t taddr, int unit, int rows = kTileRows) {
  static_assert(K % 16 == 0, "K steps of 16");
#pragma unroll
  for (int c = 0; c < K / 8; c += 2) {
    uint32_t r[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t *w = r + 4 * q;
      if (unit < rows)
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(image + canon_offset(unit, 8 * (c + q), K)));
      else
        w[0] = w[1] = w[2] = w[3] = 0u;
    }
    __syncwarp();
    tmem_st8(taddr + static_cast<uint32_t>(4 * c), r);
  }
}

// Hidden unit `unit` of all rows: ReLU, bf16, into column `unit` of the hidden-activation operand.
template <int H, int RB>
__device__ __forceinline__ void small_epilogue(uint32_t acc_taddr, uint32_t ht_addr, int unit) {
  float v[RB];
  small_tmem_ld<RB>(acc_taddr, v);
#pragma unroll
  for (int n = 0; n < RB; n += 2) {
    const uint32_t p = relu_pack_bf16(__float_as_uint(v[n]), __float_as_uint(v[n + 1]));
    sts_u16(ht_addr + a_offset<H>(n, unit), static_cast<uint16_t>(p & 0xFFFFu));
    sts_u16(ht_addr + a_offset<H>(n + 1, unit), static_cast<uint16_t>(p >> 16));
  }
}

// One dense layer, weights as the M operand: accumulator[unit][row] = bias[unit] + sum_k W[unit][k] x[row][k].
template <int K, int RB, bool BIAS_TILE>
__device__ __forceinline__ void small_issue_layer(uint32_t d_tmem, uint32_t w_tmem, uint32_t x_addr, uint32_t bias_tmem, uint32_t ones_addr, uint32_t bar) {
  constexpr uint32_t idesc = instr_desc(kTileRows, RB);
  if (elect_one()) {
    tc_fence_after();
    if (BIAS_TILE) mma_bf16_ts(d_tmem, bias_tmem, smem_desc(ones_addr, 128, 256), idesc, 0);
#pragma unroll
    for (int k = 0; k < K / 16; ++k)
      mma_bf16_ts(d_tmem, w_tmem + k * 8, smem_desc(x_addr + k * 2 * kALbo, kALbo, (K / 8) * kALbo), idesc, (BIAS_TILE || k > 0) ? 1u : 0u);
    mma_commit(bar);
  }
  __syncwarp();
}

constexpr int kSmallIssuer = 3, kSmallHelper = 4;  // warps

template <int N, int F, int H, int RB, bool EVAL, int ENV>
__global__ void __launch_bounds__(SmallShape<N, H, RB>::THREADS, 1)
rollout_tc_small_kernel(RolloutArgs a, const unsigned char *image, int ept) {
  using S = TcShape<N, H>;
  using Q = SmallShape<N, H, RB>;
  constexpr int D = S::D, K1 = S::K1;
  constexpr bool ev = EVAL;     // evaluation block: nothing of the trajectory is stored
  static_assert(N + F <= kEvFrac, "an event's record");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  SmallSmem<N, F, H, RB> &sm = *reinterpret_cast<SmallSmem<N, F, H, RB> *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31;
  const int wg = __shfl_sync(0xFFFFFFFFu, tid / 32, 0);  // warp (uniform to the compiler)

  // ---- one-time set-up: barriers, tensor memory, weights -------------------------------------
  if (tid == 0) {
    sm.abort = 0;
    mbar_init(smem_u32(&sm.load_bar), 1);
    mbar_init(smem_u32(&sm.mma_bar), 1);
    for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&sm.ev_full[i]), 1); mbar_init(smem_u32(&sm.ev_empty[i]), 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wg == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "r"(Q::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const uint32_t w_addr = smem_u32(sm.weights);
  const uint32_t x_addr = smem_u32(sm.x), ht_addr = smem_u32(sm.ht), stage_addr = smem_u32(sm.stage);
  const uint32_t logit_addr = smem_u32(sm.logit), uni_addr = smem_u32(sm.uniform[0]);
  const uint32_t ev_full0 = smem_u32(&sm.ev_full[0]), ev_empty0 = smem_u32(&sm.ev_empty[0]);
  for (int i = tid; i < static_cast<int>(Q::X_BYTES / 16); i += Q::THREADS) sts_zero16(x_addr + 16u * i);
  for (int i = tid; i < static_cast<int>(Q::HT_BYTES / 16); i += Q::THREADS) sts_zero16(ht_addr + 16u * i);
  dependents_may_start();
  wait_for_predecessor();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  bool timed_out = false;
  if (tid == 0) {
    const uint32_t lbar = smem_u32(&sm.load_bar);
    mbar_expect_tx(lbar, S::IMAGE_BYTES);
    constexpr uint32_t kChunk = 16384;
    for (uint32_t off = 0; off < S::IMAGE_BYTES; off += kChunk) {
      const uint32_t n = S::IMAGE_BYTES - off < kChunk ? S::IMAGE_BYTES - off : kChunk;
      bulk_load(smem_u32(sm.weights + off), image + off, n, lbar);
    }
  }

  // ---- this CTA's tile
  const int e0 = static_cast<int>(blockIdx.x) * ept;
  const int n_env = min(ept, a.env.n_envs - e0);
  const int n_rows = n_env * N;
  const size_t M = static_cast<size_t>(a.env.n_envs) * N;
  const int le = lane / N, ag = lane % N;  // warps 0 and 4: local environment and agent of this lane (its row is `lane`)
  const bool row_lane = lane < Q::ROWS && le < n_env;
  const uint32_t env_id = static_cast<uint32_t>(a.env.first_env + e0 + le);
  const int n_steps = ev ? a.T : a.T + 1;  // with the bootstrap step
  auto draw = [&](int t) {                 // the uniform of step t's action
    if (row_lane && t < a.T) sts_f32(uni_addr + 4u * static_cast<uint32_t>((t & 3) * RB + lane), action_uniform(a.env, a.t_global0 + static_cast<uint32_t>(t), env_id, static_cast<uint32_t>(ag)));
  };
  if (wg == kSmallHelper) { draw(0); draw(1); }

  timed_out = !mbar_wait(smem_u32(&sm.load_bar), 0);
  timed_out = __syncthreads_or(timed_out) != 0;
  const uint32_t tmem_base = sm.tmem_base;
  const uint32_t lane_off = static_cast<uint32_t>(wg * 32) << 16;
  const uint32_t acc_col = tmem_base + Q::ACC_COL, head_col = tmem_base + Q::HEAD_COL;
  if (wg < 4) {  // the weights into tensor memory: thread j unit j
    operand_to_tmem<K1>(w_addr + S::W1_OFF, tmem_base + lane_off + Q::W1_COL, tid);
    if (!S::FOLD1) operand_to_tmem<16>(w_addr + S::B1_OFF, tmem_base + lane_off + Q::B1_COL, tid);
    operand_to_tmem<H>(w_addr + S::W2_OFF, tmem_base + lane_off + Q::W2_COL, tid);
    operand_to_tmem<16>(w_addr + S::B2_OFF, tmem_base + lane_off + Q::B2_COL, tid);
    operand_to_tmem<H>(w_addr + S::WH_OFF, tmem_base + lane_off + Q::WH_COL, tid, kHeadRows);
    tmem_st_wait();
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t bar = smem_u32(&sm.mma_bar);

  if (timed_out) {
    // nothing was started
  } else if (wg == kSmallHelper) {
    // ---- warp 4, lane = row
    bool bulk_pending = false;  // lane 0
    for (int k = 0; k <= n_steps && !timed_out; ++k) {
      timed_out = !mbar_wait_warp(ev_full0 + 8u * (k & 1), static_cast<uint32_t>(k >> 1) & 1u);
      if (timed_out || *reinterpret_cast<volatile int *>(&sm.abort)) break;
      const uint32_t *rec = sm.event[k & 1] + lane * kEvPitch;
      if (!ev) {
        if (k >= 1 && row_lane) {  // outputs of step k - 1 (the bootstrap step has a value only)
          const size_t at = static_cast<size_t>(k - 1) * M + static_cast<size_t>(e0) * N + lane;
          a.buf.values[at] = __uint_as_float(rec[kEvValue]);
          if (k - 1 < a.T) {
            a.buf.actions[at] = static_cast<int32_t>(rec[kEvAction]);
            a.buf.logp[at] = __uint_as_float(rec[kEvLogp]);
            a.buf.rewards[at] = __uint_as_float(rec[kEvReward]);
            if (ag == 0) a.buf.dones[static_cast<size_t>(k - 1) * a.env.n_envs + e0 + le] = static_cast<uint8_t>(rec[kEvDone]);
            if (a.write_logits) {
#pragma unroll
              for (int q = 0; q < kActions; ++q) a.buf.logits[at * kActions + q] = __uint_as_float(rec[kEvLogit + q]);
            }
          }
        }
        if (k < a.T) {  // the fp32 observation rows of step k
          if (bulk_pending) { bulk_store_wait_read(); bulk_pending = false; }
          __syncwarp();
          for (int i = lane; i < static_cast<int>(Q::STAGE_BYTES / 16); i += 32) sts_zero16(stage_addr + 16u * i);
          __syncwarp();
          if (row_lane) {
            EnvRegs<N, F> env;
#pragma unroll
            for (int q = 0; q < N + F; ++q) env.ent[q] = rec[q];
            write_row_f32<N, F, ENV>(env, a.env, ag, __uint_as_float(rec[kEvFrac]), stage_addr + 4u * static_cast<uint32_t>(lane * D));
          }
          fence_async_smem();
          __syncwarp();
          const size_t row0 = static_cast<size_t>(k) * M + static_cast<size_t>(e0) * N;
          float *obs_dst = a.buf.obs + row0 * D;
          const int count = n_rows * D;
          if (whole_pieces16(obs_dst, count)) {
            if (lane == 0) {
              bulk_store(obs_dst, stage_addr, static_cast<uint32_t>(count) * 4u);
              bulk_pending = true;
            }
          } else {
            const float *stage = reinterpret_cast<const float *>(sm.stage);
            for (int i = lane; i < count; i += 32) obs_dst[i] = stage[i];
          }
        }
      }
      draw(k + 2);
      __syncwarp();
      if (lane == 0) mbar_arrive(ev_empty0 + 8u * (k & 1));
    }
  } else {
    // ---- warps 0..3
    const float *head_bias = reinterpret_cast<const float *>(sm.weights + S::BH_OFF);
    const bool issuer = wg == kSmallIssuer, active = wg == 0 && row_lane;
    const int base = active ? lane - ag : lane;
    uint32_t phase = 0;
    EnvRegs<N, F> env;
    if (active) {
      load_env(env, a.state[e0 + le]);
    } else {
#pragma unroll
      for (int k = 0; k < N + F; ++k) env.ent[k] = 0;
      env.step = 0; env.episode = 0; env.total = 1;
    }
    float out_value = 0.0f, out_logp = 0.0f, out_reward = 0.0f, out_logit[kActions];
    int out_action = 0;
    bool out_done = false;
#pragma unroll
    for (int k = 0; k < kActions; ++k) out_logit[k] = 0.0f;
    // Event k for warp 4: the state that step k acts on and the outputs of the step before (whole warp 0).
    auto publish = [&](int k, float frac) {
      if (k >= 2) timed_out |= !mbar_wait_warp(ev_empty0 + 8u * (k & 1), static_cast<uint32_t>((k >> 1) - 1) & 1u);
      if (!ev && active) {
        uint32_t *rec = sm.event[k & 1] + lane * kEvPitch;
        uint32_t w[16];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = q < N + F ? env.ent[q < N + F ? q : 0] : 0u;
        w[kEvFrac] = __float_as_uint(frac); w[kEvAction] = static_cast<uint32_t>(out_action); w[kEvLogp] = __float_as_uint(out_logp);
        w[kEvValue] = __float_as_uint(out_value); w[kEvReward] = __float_as_uint(out_reward); w[kEvDone] = out_done ? 1u : 0u;
        w[14] = __float_as_uint(out_logit[0]); w[15] = __float_as_uint(out_logit[1]);
#pragma unroll
        for (int q = 0; q < 16; q += 4) *reinterpret_cast<uint4 *>(rec + q) = make_uint4(w[q], w[q + 1], w[q + 2], w[q + 3]);
        if (a.write_logits)
          *reinterpret_cast<uint4 *>(rec + 16) = make_uint4(__float_as_uint(out_logit[2]), __float_as_uint(out_logit[3]), __float_as_uint(out_logit[4]), __float_as_uint(out_logit[5]));
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(ev_full0 + 8u * (k & 1));
    };
    EvalSums sums;                // lanes with ag == 0: their environment
    float frac = step_fraction(env.step, a.env.cap);
    int t = 0;
    for (; t < n_steps; ++t) {
      const bool last = !ev && (t == a.T);
      // 1. the bf16 observation rows
      if (active) write_row_bf16<N, F, K1, S::FOLD1, ENV, kALbo>(env, a.env, ag, frac, x_addr + a_offset<K1>(lane, 0));
      fence_async_smem();
      tc_fence_before();
      if (group_any(0, timed_out)) { timed_out = true; break; }  // a wait of the previous step ran out
      // 2. layer 1; meanwhile warp 4 gets its event, and the step count's next value becomes a fraction
      if (issuer)
        small_issue_layer<K1, RB, !S::FOLD1>(acc_col, tmem_base + Q::W1_COL, x_addr, tmem_base + Q::B1_COL, w_addr + S::ONES_OFF, bar);
      float next_frac = 0.0f;
      if (wg == 0) {
        publish(t, frac);
        next_frac = step_fraction(env.step + 1, a.env.cap);
      }
      timed_out |= !mbar_wait(bar, phase);
      phase ^= 1;
      tc_fence_after();
      small_epilogue<H, RB>(acc_col + lane_off, ht_addr, tid);
      fence_async_smem();
      tc_fence_before();
      group_sync(0);
      // 3. layer 2
      if (issuer) small_issue_layer<H, RB, true>(acc_col, tmem_base + Q::W2_COL, ht_addr, tmem_base + Q::B2_COL, w_addr + S::ONES_OFF, bar);
      timed_out |= !mbar_wait(bar, phase);
      phase ^= 1;
      tc_fence_after();
      small_epilogue<H, RB>(acc_col + lane_off, ht_addr, tid);
      fence_async_smem();
      tc_fence_before();
      group_sync(0);
      // 4. heads: lanes 0..5 the logits, lane 6 the value, one column per row
      if (issuer) small_issue_layer<H, RB, false>(head_col, tmem_base + Q::WH_COL, ht_addr, 0u, 0u, bar);
      timed_out |= !mbar_wait(bar, phase);
      phase ^= 1;
      tc_fence_after();
      int action = 0;
      if (wg == 0) {
        float hl[RB];
        small_tmem_ld<RB>(head_col, hl);
        if (lane < 8) {
          const float b = head_bias[lane];  // the heads' biases stay fp32; entry 7 is zero
#pragma unroll
          for (int n = 0; n < RB; ++n) sts_f32(logit_addr + 4u * static_cast<uint32_t>(n * 8 + lane), hl[n] + b);
        }
        __syncwarp();
        if (active) {
          float hv[kActions + 1];
#pragma unroll
          for (int k = 0; k <= kActions; ++k) hv[k] = lds_f32(logit_addr + 4u * static_cast<uint32_t>(lane * 8 + k));
          out_value = hv[kActions];
          if (!last) {
            const float u = lds_f32(uni_addr + 4u * static_cast<uint32_t>((t & 3) * RB + lane));
            float m, sum;
            action = draw_action(hv, u, m, sum);
            const size_t row = static_cast<size_t>(t) * M + static_cast<size_t>(e0) * N + lane;
            if (a.forced) {
              action = a.forced[row];
              if (action < 0 || action >= kActions) action = 0;
            }
            if (ev) {
              if (a.greedy) action = greedy_action(hv);
              if (a.ev_actions) a.ev_actions[row] = action;
            }
            float la = hv[0];
#pragma unroll
            for (int k = 1; k < kActions; ++k) la = (action == k) ? hv[k] : la;
            out_action = action;
            out_logp = la - m - __logf(sum);
#pragma unroll
            for (int k = 0; k < kActions; ++k) out_logit[k] = hv[k];
          }
        }
        // 5. transition and auto-reset, inside warp 0
        if (!last) {
          if constexpr (ENV == 0) step_env_warp<N, F>(env, a.env, env_id, ag, base, active, action, out_reward, out_done);
          else wh_step_env_warp<N, F>(env, a.env, env_id, ag, base, active, action, out_reward, out_done);
          if (ev) sums.step(out_reward, out_done);
          frac = env.step == 0 ? 0.0f : next_frac;  // (a new episode starts at step 0)
        }
      }
      tc_fence_before();
    }
    timed_out = group_any(0, timed_out);
    if (wg == 0) {  // the last event: outputs only, or the word that there is none
      if (timed_out) *reinterpret_cast<volatile int *>(&sm.abort) = 1;
      publish(t, 0.0f);
    }
    if (!timed_out && active && ag == 0) {
      store_env(env, a.state[e0 + le]);
      if (ev) { a.ev_count[e0 + le] = sums.count; a.ev_ret[e0 + le] = sums.ret; a.ev_len[e0 + le] = sums.len; }
    }
  }
  if (timed_out) atomicExch(a.status, kStatusTimeout);
  bulk_store_wait_all();
  tc_fence_before();
  __syncthreads();
  if (wg == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(Q::TMEM_COLS) : "memory");
  }
}

template <int N, int F, int H, int RB, int ENV>
cudaError_t launch_tc_small(mava_rollout *h, const RolloutArgs &args, int sms) {
  using Q = SmallShape<N, H, RB>;
  auto kern = args.eval ? rollout_tc_small_kernel<N, F, H, RB, true, ENV> : rollout_tc_small_kernel<N, F, H, RB, false, ENV>;
  const size_t smem = sizeof(SmallSmem<N, F, H, RB>);
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (err != cudaSuccess) return err;
  int ept = (h->cfg.n_envs + sms - 1) / sms;  // the caller made sure this fits a tile
  if (ept > Q::EPT_MAX) ept = Q::EPT_MAX;
  if (ept < 1) ept = 1;
  // A tile's observation block leaves as one bulk copy when it is a whole number of 16-byte pieces
  // (every tile then also starts on such a boundary): take the next such size if the tile has room.
  for (int e = ept; e <= Q::EPT_MAX; ++e)
    if ((e * N * Q::D) % 4 == 0) { ept = e; break; }
  const int n_tiles = (h->cfg.n_envs + ept - 1) / ept;
  h->launches += 1;
  return launch_dependent(kern, n_tiles, Q::THREADS, smem, h->stream, args, static_cast<const unsigned char *>(h->d_wtc), ept);  // (n_tiles <= sms)
}

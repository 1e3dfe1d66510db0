// attn_pipe_kernel: fused attention in which every Q tile of 256 rows is worked on by one CTA from its first key to its last
// (nothing to merge between CTAs), as two sub-tiles of 128 rows with a softmax warpgroup each, one thread per row, 128 keys a
// step: causal and not at d = 128, not causal at d = 64.  (Short tiles at d = 64 and tiles of 128 rows: narrow_kernel.cuh.)
//
// What bounds the step at d = 128 is a chain: scores in tensor memory -> softmax warps (load, maximum, exponentials, P back) -> P V
// -> Q K^T of the next step, which overwrites P's columns (S0, S1, O0 and O1 fill tensor memory).  A clock record of attn_fwd_kernel
// and of attempts on the way here showed where it loses time, and this kernel differs in that:
//   * An MMA warp for each sub-tile.  Issue of a matrix instruction blocks until those in front of it have started, so one warp that
//     serves both sub-tiles leaves the tensor pipe idle during each of its waits (some 100 cycles, five a step).  The two take
//     turns, P V and Q K^T of a step at a time: left alone, they drift into step with each other, and their products then
//     delay one another (128 heads x 4096, d = 128, us: one MMA warp 982, two that do not take turns 971, that do 946).
//   * Waits without a vote.  A wait that is over passes with one test; one that expires raises the CTA's abort flag, and a warp looks
//     at its own flag once a step (wait_on).
//   * K of the next step and V of this one are counted on one barrier: one wait a step instead of two.
//   * The exponentials of a 32-score chunk carry the sums of the chunk before, the last chunk's sums come after P has been handed
//     over; the decision whether the reference moves is one comparison with a threshold that the step before has prepared.
//     (Exponentials of the first chunk ahead of the maximum, on the old reference, were 2 % faster on flat scores and slower
//     wherever references move; the code that mends them costs moves in every step.)
//   * At d = 128 one pair of eight takes the polynomial instead of two (a pair costs eight issue slots more than on the exponential
//     unit; none: 0-1 % slower).  Causal, where the kernel before took none in the common step, it is the quintic, which is as exact as
//     the unit (128 x 4096 in loops: cubic 547, quintic 549, none 551 us).  At d = 64 there is no chain: P has columns of its own, the
//     next scores are produced under this step's exponentials, both warpgroups work all the time, and three pairs of eight are
//     fastest (2: 867, 3: 829, 4: 887 us at 148 x 4096); one of them is a cubic and two are quartics, whose errors together are 0.7 times
//     those of two cubics (three cubics: 824, as it is 855, three quartics 865; 148 x 1024 55.6 / 57.1 / 57.3).
// As before it: the epilogue of a tile runs under the next one (the correction warpgroup normalises and stores it), a sub-tile runs
// only its own steps, tiles come from the hardware's queue of CTAs not yet started (clusterlaunchcontrol.try_cancel), causal ones
// longest first within groups of heads whose K and V stay in L2.
// Measured (us, the kernels before / this one, calls back to back): d = 128 causal 128 x 4096 549 / 516, 600 x 512 87.5 / 76.4, 213 shapes in
// whole tiles 0.84 times on the geometric mean; not causal 148 x 4096 1080 / 1053, 148 x 2048 with variance 3 303 / 294, 95 shapes
// in waves of whole tiles 0.91 times; d = 64 (tiles that are not long, pipe_tiles in attn_api.cu) 148 x 1024 58.9 / 57.1, 128 x 2000 195 / 178, 442
// shapes 0.959 times.  Long calls run into the power limit (990 W) and keep less: in loops of 0.8 s 4 x 32 x 4096, d = 128, takes 983 /
// 967, causal 580 / 543.
#pragma once

#include "attn_kernels.cuh"

namespace attn {

struct PipeParams {
  int Lq, Lk;              // query rows and keys per head
  int q_tiles;             // Q tiles per head = ceil(Lq / 256)
  int n_steps;             // key steps per head = ceil(Lk / 128)
  int heads;               // B * H
  int group_heads;         // causal: heads whose tiles are dealt out together, longest first
  int stages;              // ring depth (even: a K tile and its V tile side by side)
  float scale_log2;        // log2(e) / sqrt(d)
  unsigned int* status;    // as in FwdParams
};

template <int D>
struct PipeSmem {
  static constexpr int kSubBytes = kSub * D * 2;
  static constexpr int kQBytes = 2 * kSubBytes;
  static constexpr int kStageBytes = 128 * D * 2;
  static constexpr int kOutBytes = 8 * 4096;                     // two [32 rows][64 columns] bf16 chunks per correction warp
  static constexpr int kMiscBytes = 3072;
  __host__ __device__ static constexpr int total(int stages) { return kQBytes + stages * kStageBytes + kOutBytes + kMiscBytes; }
};

struct PipeMisc {
  float alpha[2][kSub];                    // [sub-tile][row] rescale factor
  float inv[2][kSub];                      // [sub-tile][row] 1 / denominator of a finished tile
  uint4 sched[2];                          // answers of try_cancel (16 bytes each)
  uint64_t sched_full[2], sched_empty[2];
  uint64_t q_full[2], q_empty[2];          // per sub-tile
  uint64_t kv_full[kMaxStages];            // of a V stage: V_j and K_{j+1}; of a K stage: a tile's K_0
  uint64_t kv_empty[kMaxStages];
  uint64_t turn[2];                        // d = 128: the sub-tile's MMA warp may issue its step
  // per sub-tile: scores ready, first part of P ready and accumulator rescaled, all of P ready, accumulator complete (d = 128: at a
  // tile's end; d = 64: every step), rescale factors ready, a tile's denominators ready, d = 64: scores are in registers
  uint64_t s_full[2], p_full[2], p_half[2], o_full[2], alpha_full[2], fin_full[2], s_free[2];
  AbortCell abort;
  uint32_t tmem_slot;
};
static_assert(sizeof(PipeMisc) <= PipeSmem<128>::kMiscBytes, "misc region too large");
constexpr int kPipeSchedReaders = 15;      // warps that read a tile's index: 8 softmax, 4 correction, 2 MMA, TMA

// A tile: its head, first row and the key steps of its two sub-tiles (n1 is n0, n0 + 1 or 0; n: the larger).
struct PipeWork {
  int bh, q_row0, n, n0, n1;
  __device__ __forceinline__ int steps(int i) const { return i ? n1 : n0; }
};
template <bool CAUSAL>
__device__ __forceinline__ PipeWork pipe_work(int index, const PipeParams& p) {
  PipeWork w;
  int q;
  if constexpr (CAUSAL) {
    const int per_group = p.group_heads * p.q_tiles;
    const int group = index / per_group, r = index - group * per_group;
    const int first = group * p.group_heads;
    const int n = p.heads - first < p.group_heads ? p.heads - first : p.group_heads;
    q = p.q_tiles - 1 - r / n;
    w.bh = first + r % n;
  } else {
    w.bh = index / p.q_tiles;
    q = index - w.bh * p.q_tiles;
  }
  w.q_row0 = q * 2 * kSub;
  // (causal: a sub-tile's last key step is the one that holds its own rows)
  w.n0 = CAUSAL ? 2 * q + 1 : p.n_steps;
  w.n1 = w.q_row0 + kSub >= p.Lq ? 0 : CAUSAL ? 2 * q + 2 : p.n_steps;
  w.n = w.n1 > w.n0 ? w.n1 : w.n0;
  return w;
}

template <int D, bool CAUSAL>
__global__ void __launch_bounds__(512, 1)
attn_pipe_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o, const PipeParams p) {
  using SM = PipeSmem<D>;
  constexpr int TKV = 128, KCH = D / 64, O_COL0 = 2 * TKV;
  constexpr bool kSplit = D == 64;                      // P has columns of its own (else it overwrites the front of its scores)
  constexpr int P_COL0 = O_COL0 + 2 * D;
  constexpr int kPoly = D == 64 ? kMixThree : CAUSAL ? kMixUnit : kMixOne;
  constexpr int kFirstK = D == 64 ? 6 : 4;              // 16-key steps of P V that the first hand-over of P allows

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t ring_smem = smem_base + SM::kQBytes;
  const uint32_t out_smem = ring_smem + p.stages * SM::kStageBytes;
  PipeMisc* const misc = reinterpret_cast<PipeMisc*>(smem_raw + SM::kQBytes + p.stages * SM::kStageBytes + SM::kOutBytes);
  volatile int* abort_flag = &misc->abort.flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    abort_cell_init(&misc->abort, p.status);
    if (smem_base & 1023u) note_timeout(wait_info(kRoleLoad, 0, 0xFFFF), &misc->abort.flag);   // swizzled tiles need 1024-byte alignment
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&misc->kv_full[s]), 1);
      mbar_init(smem_u32(&misc->kv_empty[s]), 2);              // both sub-tiles
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&misc->sched_full[i]), 1);
      mbar_init(smem_u32(&misc->sched_empty[i]), kPipeSchedReaders);
      mbar_init(smem_u32(&misc->q_full[i]), 1);
      mbar_init(smem_u32(&misc->q_empty[i]), 1);
      mbar_init(smem_u32(&misc->turn[i]), 1);
      mbar_init(smem_u32(&misc->s_full[i]), 1);
      mbar_init(smem_u32(&misc->p_full[i]), 2 * kSub);         // softmax rows + correction rows
      mbar_init(smem_u32(&misc->p_half[i]), kSub);
      mbar_init(smem_u32(&misc->o_full[i]), 1);
      mbar_init(smem_u32(&misc->alpha_full[i]), kSub);
      mbar_init(smem_u32(&misc->fin_full[i]), kSub);
      mbar_init(smem_u32(&misc->s_free[i]), kSub);
    }
    fence_mbar_init();
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
    prefetch_tmap(&tm_o);
  }
  if (warp == 15) {
    tmem_alloc(smem_u32(&misc->tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_wait();
  const uint32_t tmem_base = misc->tmem_slot;
  const bool run = *const_cast<volatile int*>(&misc->abort.flag) == 0;

  // Index of this CTA's tile number `s` (s >= 1; tile 0 is blockIdx.x), -1 after the last, -2 if a wait expired.  Every
  // role's warp calls it once per s, with all lanes.
  auto next_tile = [&](int s, uint32_t role) __attribute__((always_inline)) -> int {
    const int slot = s & 1;
    if (!wait_quiet_warp(smem_u32(&misc->sched_full[slot]), ((s - 1) >> 1) & 1, abort_flag, wait_info(role, kBarSync, s))) return -2;
    const int x = clc_answer(smem_u32(&misc->sched[slot]));
    fence_proxy_async_smem();                         // the answer has been read: the next one may be written there
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&misc->sched_empty[slot]));
    return x;
  };

  // Registers: 512 x 128 at launch, then 256 x 200, 128 x 64 and 128 x 40.
  if (warp < 8) {
    // ===================================================== softmax warpgroup of one sub-tile
    setmaxnreg_inc<200>();
    const int i = warp >> 2;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_tmem = lane_base + i * TKV;
    const uint32_t p_tmem = kSplit ? lane_base + P_COL0 + i * (TKV / 2) : s_tmem;
    const uint32_t bar_s = smem_u32(&misc->s_full[i]);
    const uint32_t bar_p = smem_u32(&misc->p_full[i]);
    const uint32_t bar_h = smem_u32(&misc->p_half[i]);
    const uint32_t bar_a = smem_u32(&misc->alpha_full[i]);
    const float scale = p.scale_log2;
    const ExpConsts ek = make_exp_consts(scale);
    const int kv_tail = CAUSAL ? 0 : p.Lk & (TKV - 1);
    bool ok = run, dead = false;
    uint32_t g = 0, done = 0;                          // steps of this sub-tile over all tiles; finished tiles
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const PipeWork w = pipe_work<CAUSAL>(tile, p);
      const int n = w.steps(i);
      if (n > 0) {
        // `lim`: how far the row maximum may lie above the reference m_run before that moves (see below; first step: it always does)
        float m_run = -INFINITY, delta = 0.f, lim = 0.f;
        for (int left = n - 1; left >= 0; --left, ++g) {
          wait_on(bar_s, g & 1, abort_flag, wait_info(kRoleSoftmax, kBarSFull, g), dead);
          tc_fence_after();
          uint32_t s[TKV], pk[16], pk2[16];
          auto chunk = [&](int c) -> uint32_t(&)[32] { return *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]); };
          // Only the last step may need a mask: the causal diagonal, which starts at the sub-tile's first row and ends, in a
          // ragged last key tile, before the padding for every row of the sequence; else a ragged last key tile.  Keys past the end
          // or after the query's position get score -inf, never zero.  (Every row has a key it may attend to.)
          const bool masked = left == 0 && (CAUSAL || kv_tail != 0);
          const int last_key = CAUSAL ? row : kv_tail - 1;
          auto mask = [&](int from) __attribute__((always_inline)) {
#pragma unroll
            for (int k = 0; k < TKV / 2; ++k)
              if (from + k > last_key) s[from + k] = 0xFF800000u;
          };
          // load the row in two halves: the maximum of the first half is taken while the second is in flight
#pragma unroll
          for (int c = 0; c < 2; ++c) tmem_ld32_nowait(s_tmem + c * 32, chunk(c));
#pragma unroll
          for (int c = 0; c < 2; ++c) tmem_ld_fence(chunk(c));
#pragma unroll
          for (int c = 2; c < 4; ++c) tmem_ld32_nowait(s_tmem + c * 32, chunk(c));
          if (masked) mask(0);
          const float mx_a = max_nan(max_nan(chain_max<0, 16>(s), chain_max<16, 32>(s)), max_nan(chain_max<32, 48>(s), chain_max<48, 64>(s)));
#pragma unroll
          for (int c = 2; c < 4; ++c) tmem_ld_fence(chunk(c));
          if constexpr (kSplit) {
            tc_fence_before();
            mbar_arrive(smem_u32(&misc->s_free[i]));   // the scores are in registers: the buffer may be overwritten
          }
          if (masked) mask(TKV / 2);
          const float mx_b = max_nan(max_nan(chain_max<64, 80>(s), chain_max<80, 96>(s)), max_nan(chain_max<96, 112>(s), chain_max<112, 128>(s)));
          // Lazy rescale, as in attn_fwd_kernel: the reference moves to the row maximum if that lies above it by more than
          // kRescaleThreshold, or by anything that gives the new maximum's key more than 1 / kDominanceFactor of the denominator.
          const float m_cand = max_nan(mx_a, mx_b) * scale;
          const float gap = m_cand - m_run;
          const bool move = !(gap <= lim);             // (a NaN moves it)
          m_run = move ? m_cand : m_run;
          const uint64_t neg_m2 = pack_f32x2(-m_run, -m_run);
          const float alpha = move ? ex2_approx(-gap) : 1.0f;
          if constexpr (kSplit) {
            // The step before has read P, which is overwritten below, and every thread has made its arrivals of that step
            // (arrivals are anonymous: none of this step may come before one of the step before).
            if (g > 0) wait_on(smem_u32(&misc->o_full[i]), (g - 1) & 1, abort_flag, wait_info(kRoleSoftmax, kBarOFull, g), dead);
            tc_fence_after();
          }
          misc->alpha[i][row] = alpha;
          mbar_arrive(bar_a);
          delta *= alpha;
          uint64_t sum[2] = {0ull, 0ull};
          exp_chunk_in_place<kPoly, false>(&s[0], s, sum, ek, neg_m2, pk2);
          tmem_st16(p_tmem, pk2);
          exp_chunk_in_place<kPoly, true>(&s[32], &s[0], sum, ek, neg_m2, pk);
          tmem_st16(p_tmem + 16, pk);
          exp_chunk_in_place<kPoly, true>(&s[64], &s[32], sum, ek, neg_m2, pk2);
          if constexpr (kFirstK == 6) tmem_st16(p_tmem + 32, pk2);
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(bar_p);                          // P V may start on what has been written
          if constexpr (kFirstK == 4) tmem_st16(p_tmem + 32, pk2);
          exp_chunk_in_place<kPoly, true>(&s[96], &s[64], sum, ek, neg_m2, pk);
          tmem_st16(p_tmem + 48, pk);
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(bar_h);
#pragma unroll
          for (int j = 0; j < 16; ++j) sum[j & 1] = add_f32x2(sum[j & 1], pair_of(&s[96 + 2 * j]));
          float s0, s1;
          unpack_f32x2(add_f32x2(sum[0], sum[1]), s0, s1);
          delta += s0 + s1;
          if (any_dead(dead)) { ok = false; break; }
          // 2^gap > delta / kDominanceFactor, or gap > kRescaleThreshold; a maximum below the reference never moves it
          static_assert(kDominanceFactor == 16.0f, "its logarithm");
          lim = fminf(fmaxf(lg2_approx(delta) - 4.0f, 0.f), kRescaleThreshold);
        }
        if (!ok) break;
        // The denominators go to the correction warpgroup, which finishes the tile.  Its arrival on p_full of a tile's first
        // step says that it has read those of the tile before; from two steps on, the second step's scores come after it.  A
        // tile of one step waits for its only product instead.
        if (n == 1) {
          wait_on(smem_u32(&misc->o_full[i]), (kSplit ? g - 1 : done) & 1, abort_flag, wait_info(kRoleSoftmax, kBarOFull, g), dead);
          tc_fence_after();
        }
        misc->inv[i][row] = row_inverse(delta, m_run);
        mbar_arrive(smem_u32(&misc->fin_full[i]));
        ++done;
      }
      tile = next_tile(seq, kRoleSoftmax);
    }
  } else if (warp < 12) {
    // ================================================== correction warpgroup
    setmaxnreg_dec<64>();
    const int wq = warp & 3, row = wq * 32 + lane;
    const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
    const uint32_t stage_w = out_smem + wq * 8192;     // this warp's two staging chunks
    bool ok = run, dead = false;
    // steps of the sub-tiles; in bit i: sub-tile i's finished tiles mod 2, whether one waits for its epilogue (arrays would be
    // indexed at run time and live in local memory)
    uint32_t g0 = 0, g1 = 0, fin = 0, pending = 0, chunk_ctr = 0;
    int out_bh = 0, out_row0 = 0;                      // of the finished tile
    // A tile's end: normalise this warp's 32 rows of sub-tile i, 64 columns at a time through its two staging chunks in turn.
    auto finish = [&](int i) __attribute__((always_inline)) {
      wait_on(smem_u32(&misc->fin_full[i]), (fin >> i) & 1, abort_flag, wait_info(kRoleCorrection, kBarAlpha, 0x8000), dead);
      const float inv = misc->inv[i][row];
      wait_on(smem_u32(&misc->o_full[i]), kSplit ? ((i ? g1 : g0) - 1) & 1 : (fin >> i) & 1, abort_flag, wait_info(kRoleCorrection, kBarOFull, 0x8000), dead);
      fin ^= 1u << i;
      if (any_dead(dead)) return;                      // (nothing to store)
      tc_fence_after();
      const uint32_t o_tmem = lane_base + O_COL0 + i * D;
#pragma unroll 1
      for (int h = 0; h < KCH; ++h, ++chunk_ctr) {
        const uint32_t dst = stage_w + (chunk_ctr & 1) * 4096;
        // the store that last read this chunk (two chunks ago) must have finished reading it
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        __syncwarp();
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          uint32_t r[32];
          float v[32];
          tmem_ld32(o_tmem + h * 64 + c * 32, r);
#pragma unroll
          for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]) * inv;
          stage_row_chunk(dst, c, lane, v);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {                               // (rows past the end of the sequence are clipped by the tensor map)
          tma_store_3d(&tm_o, dst, h * 64, out_row0 + i * kSub + wq * 32, out_bh);
          tma_store_commit();
        }
      }
      tc_fence_before();                               // O has been read: this thread's next arrival on p_full says so
    };
    const volatile float* const alpha0 = &misc->alpha[0][row];
    const uint32_t bar_a = smem_u32(&misc->alpha_full[0]), bar_p = smem_u32(&misc->p_full[0]);
    // One step of sub-tile i: rescales its accumulator where a reference moved (a tile's first step starts it afresh).
    auto step = [&](int i, uint32_t& g, bool first) __attribute__((always_inline)) {
      wait_on(bar_a + 8 * i, g & 1, abort_flag, wait_info(kRoleCorrection, kBarAlpha, g), dead);
      const float a = alpha0[i * kSub];
      if (!first && __any_sync(0xffffffffu, a != 1.0f)) {
        // P V of the step before is complete (d = 128: these scores were issued behind it)
        if constexpr (kSplit) wait_on(smem_u32(&misc->o_full[i]), (g - 1) & 1, abort_flag, wait_info(kRoleCorrection, kBarOFull, g), dead);
        else wait_on(smem_u32(&misc->s_full[i]), g & 1, abort_flag, wait_info(kRoleCorrection, kBarSFull, g), dead);
        tc_fence_after();
        const uint32_t o_tmem = lane_base + O_COL0 + i * D;
#pragma unroll 1
        for (int c = 0; c < D / 16; ++c) {             // (16 columns at a time: 32 make this role spill)
          uint32_t r[16];
          tmem_ld16(o_tmem + c * 16, r);
#pragma unroll
          for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) * a);
          tmem_st16(o_tmem + c * 16, r);
        }
        tmem_wait_st();
        tc_fence_before();
      }
      mbar_arrive(bar_p + 8 * i);
      ++g;
    };
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const PipeWork w = pipe_work<CAUSAL>(tile, p);
#pragma unroll 1
      for (int i = 0; i < 2; ++i) {
        if ((pending >> i) & 1) finish(i);
        if (i == 0) step(0, g0, true);
        else if (w.n1 > 0) step(1, g1, true);
      }
      if (any_dead(dead)) { ok = false; break; }
      const int both = w.n0 < w.n1 ? w.n0 : w.n1;
#pragma unroll 1
      for (int j = 1; j < both; ++j) {
        step(0, g0, false);
        step(1, g1, false);
        if (any_dead(dead)) { ok = false; break; }
      }
      for (int j = both > 1 ? both : 1; ok && j < w.n; ++j) {
        if (w.n0 > w.n1) step(0, g0, false);
        else step(1, g1, false);
        if (any_dead(dead)) { ok = false; break; }
      }
      if (!ok) break;
      pending = 1u | (w.n1 > 0 ? 2u : 0u);
      out_bh = w.bh;
      out_row0 = w.q_row0;
      tile = next_tile(seq, kRoleCorrection);
    }
#pragma unroll 1
    for (int i = 0; i < 2; ++i)
      if (ok && tile == -1 && ((pending >> i) & 1)) finish(i);
    if (lane == 0) tma_store_wait_read();              // shared memory is read by the stores until here
    __syncwarp();
  } else if (warp < 14) {
    // ============================== MMA issuer of one sub-tile (the whole warp walks the loop, one lane issues)
    setmaxnreg_dec<40>();
    const int i = warp - 12;
    bool ok = run, dead = false;
    const uint32_t s_tmem = tmem_base + i * TKV, o_tmem = tmem_base + O_COL0 + i * D;
    const uint32_t p_tmem = kSplit ? tmem_base + P_COL0 + i * (TKV / 2) : s_tmem;
    uint32_t g = 0, q_uses = 0, slot = 0, qk = 0;      // steps; Q loads that have been read; turns taken; products Q K^T issued
    uint32_t k0_seen = 0;                              // bit s: tiles' first K tiles seen in stage s, mod 2
    int vs = 1;                                        // stage of V_j
    uint32_t vph = 0;
    auto wait = [&](uint64_t* bar, uint32_t parity, uint32_t id) __attribute__((always_inline)) {
      wait_on(smem_u32(bar), parity, abort_flag, wait_info(kRoleMma, id, 0x100 * i + (g & 0xFF)), dead);
    };
    // (one lane) Scores of the keys in stage k; last: no later step of the tile reads this Q.
    auto issue_scores = [&](int k, bool last) __attribute__((always_inline)) {
      issue_qk<D, TKV>(s_tmem, smem_base + i * SM::kSubBytes, ring_smem + k * SM::kStageBytes);
      umma_commit(smem_u32(&misc->s_full[i]));
      umma_commit(smem_u32(&misc->kv_empty[k]));
      if (last) umma_commit(smem_u32(&misc->q_empty[i]));
    };
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const PipeWork w = pipe_work<CAUSAL>(tile, p);
      const int n = w.n, ni = w.steps(i);
      // (both warps see every phase of every stage, also of tiles that have no second sub-tile: a wait by parity is exact only so)
      const int k0 = vs - 1;
      wait(&misc->kv_full[k0], (k0_seen >> k0) & 1, kBarKvFull);
      k0_seen ^= 1u << k0;
      if (ni > 0) {
        wait(&misc->q_full[i], q_uses & 1, kBarQ);
        ++q_uses;
        if (kSplit && qk > 0) wait(&misc->s_free[i], (qk - 1) & 1, kBarSFull);
        ++qk;
        tc_fence_after();
        if (may_issue(dead)) issue_scores(k0, ni == 1);
      } else if (lane == 0 && !dead) {
        mbar_arrive(smem_u32(&misc->kv_empty[k0]));
      }
      __syncwarp();
      for (int j = 0; j < n; ++j) {
        const uint32_t v = ring_smem + vs * SM::kStageBytes;
        const int ks = vs + 1 == p.stages ? 0 : vs + 1;          // stage of K_{j+1}
        wait(&misc->kv_full[vs], vph, kBarKvFull);               // V_j and K_{j+1}
        if (j < ni) {
          if constexpr (kSplit) {
            if (j + 1 < ni) {
              wait(&misc->s_free[i], (qk - 1) & 1, kBarSFull);
              ++qk;
              tc_fence_after();
              if (may_issue(dead)) issue_scores(ks, j + 2 == ni);
              __syncwarp();
            }
          } else {
            wait(&misc->turn[i], (slot + 1 + i) & 1, kBarSync);  // (sub-tile 0 begins)
          }
          wait(&misc->p_full[i], g & 1, kBarPFull);
          tc_fence_after();
          if (may_issue(dead)) issue_pv<D, TKV>(o_tmem, p_tmem, v, j > 0, TKV * 128, 1024, 0, kFirstK);
          __syncwarp();
          wait(&misc->p_half[i], g & 1, kBarPFull);
          tc_fence_after();
          if (may_issue(dead)) {
            issue_pv<D, TKV>(o_tmem, p_tmem, v, true, TKV * 128, 1024, kFirstK, 8);
            if (!kSplit && j + 1 < ni) issue_scores(ks, j + 2 == ni);
            else umma_commit(smem_u32(&misc->o_full[i]));
            if (!kSplit) mbar_arrive(smem_u32(&misc->turn[i ^ 1]));
            umma_commit(smem_u32(&misc->kv_empty[vs]));
            if (j + 1 == ni && j + 1 < n) mbar_arrive(smem_u32(&misc->kv_empty[ks]));   // a key tile after this sub-tile's rows
          }
          __syncwarp();
          ++g;
        } else {
          // a step that only the other sub-tile has
          if (!kSplit) wait(&misc->turn[i], (slot + 1 + i) & 1, kBarSync);
          if (lane == 0 && !dead) {
            if (!kSplit) mbar_arrive(smem_u32(&misc->turn[i ^ 1]));
            mbar_arrive(smem_u32(&misc->kv_empty[vs]));
            if (j + 1 < n) mbar_arrive(smem_u32(&misc->kv_empty[ks]));
          }
          __syncwarp();
        }
        ++slot;
        vs += 2;
        if (vs >= p.stages) { vs -= p.stages; vph ^= 1u; }
        if (any_dead(dead)) { ok = false; break; }
      }
      if (!ok) break;
      tile = next_tile(seq, kRoleMma);
    }
  } else if (warp == 14) {
    // ================================================== TMA producer, and the requests for the next tile
    setmaxnreg_dec<40>();
    bool ok = run;
    int asked = 0;                                     // requests made
    int stage = 0;                                     // of the next K tile; its V tile goes to the stage after it
    uint32_t phase = 0;
    uint32_t q_loads0 = 0, q_loads1 = 0, k0_loads = 0; // (k0_loads: bit s: tiles' first K tiles loaded into stage s, mod 2)
    // (the waits are taken by the whole warp, the copies issued by one lane)
    auto stage_free = [&](int st, uint32_t ph) __attribute__((always_inline)) -> bool {
      return wait_quiet_warp(smem_u32(&misc->kv_empty[st]), ph ^ 1u, abort_flag, wait_info(kRoleLoad, kBarKvEmpty, st));
    };
    // bytes: announced on `bar`, 0 where they have been
    auto load = [&](const CUtensorMap* tm, int st, int j, int bh, uint32_t bar, uint32_t bytes) __attribute__((always_inline)) {
      if (elect_one()) {
        if (bytes) mbar_arrive_expect_tx(bar, bytes);
#pragma unroll
        for (int c = 0; c < KCH; ++c) tma_load_3d(ring_smem + st * SM::kStageBytes + c * (TKV * 128), tm, c * 64, j * TKV, bh, bar);
      }
      __syncwarp();
    };
    auto load_q = [&](int i, const PipeWork& w) __attribute__((always_inline)) -> bool {
      const uint32_t u = i ? q_loads1 : q_loads0;
      if (u >= 1 && !wait_quiet_warp(smem_u32(&misc->q_empty[i]), (u - 1) & 1, abort_flag, wait_info(kRoleLoad, kBarQ, u))) return false;
      if (elect_one()) {
        const uint32_t bar = smem_u32(&misc->q_full[i]);
        mbar_arrive_expect_tx(bar, SM::kSubBytes);
#pragma unroll
        for (int c = 0; c < KCH; ++c)
          tma_load_3d(smem_base + i * SM::kSubBytes + c * (kSub * 128), &tm_q, c * 64, w.q_row0 + i * kSub, w.bh, bar);
      }
      __syncwarp();
      if (i) ++q_loads1; else ++q_loads0;
      return true;
    };
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const PipeWork w = pipe_work<CAUSAL>(tile, p);
      const int n = w.n;
      // the first product needs K_0 and Q of sub-tile 0; the first tile's Q buffer is free at once
      if (seq == 1) ok = load_q(0, w);
      if (ok) ok = stage_free(stage, phase);
      if (!ok) break;
      load(&tm_k, stage, 0, w.bh, smem_u32(&misc->kv_full[stage]), SM::kStageBytes);
      k0_loads ^= 1u << stage;
      if (seq > 1) ok = load_q(0, w);
      if (ok && w.n1 > 0) ok = load_q(1, w);
      for (int j = 0; ok && j < n; ++j) {
        const int vst = stage + 1;
        const uint32_t bar = smem_u32(&misc->kv_full[vst]), ph = phase;
        stage += 2;
        if (stage >= p.stages) { stage = 0; phase ^= 1u; }
        if (j + 1 < n) {
          // K_{j+1} and V_j are counted on one barrier: both stages are free before either is announced
          ok = stage_free(stage, phase) && stage_free(vst, ph);
          if (!ok) break;
          load(&tm_k, stage, j + 1, w.bh, bar, 2 * SM::kStageBytes);
          load(&tm_v, vst, j, w.bh, bar, 0);
        } else {
          // Ask for the tile after this one, into the slot that held the tile before this one -- as late as the answer is
          // sure to be back in time (a ring's depth ahead of the MMA warps): a tile asked for early would be tied to this
          // CTA while others run dry.
          if (seq >= 3) ok = wait_quiet_warp(smem_u32(&misc->sched_empty[seq & 1]), ((seq - 3) >> 1) & 1, abort_flag, wait_info(kRoleLoad, kBarSync, seq));
          if (!ok) break;
          if (elect_one()) {
            mbar_arrive_expect_tx(smem_u32(&misc->sched_full[seq & 1]), 16);
            clc_try_cancel(smem_u32(&misc->sched[seq & 1]), smem_u32(&misc->sched_full[seq & 1]));
          }
          __syncwarp();
          asked = seq;
          ok = stage_free(vst, ph);
          if (!ok) break;
          load(&tm_v, vst, j, w.bh, bar, SM::kStageBytes);
        }
      }
      if (!ok) break;
      tile = next_tile(seq, kRoleLoad);
    }
    grid_release();
    if (tile == -2) ok = false;
    if (!ok && lane == 0) {
      // Drain: every copy started here must land before the CTA may exit, and so must an answer still on its way.
      for (int s = 0; s < p.stages; s += 2) {
        drain_bar(smem_u32(&misc->kv_full[s]), ((k0_loads >> s) & 1) ^ 1u);
        drain_bar(smem_u32(&misc->kv_full[s + 1]), s + 1 < stage ? phase : phase ^ 1u);
      }
      for (int i = 0; i < 2; ++i)
        if (const uint32_t q = i ? q_loads1 : q_loads0) drain_bar(smem_u32(&misc->q_full[i]), (q - 1) & 1);
      if (asked > 0) drain_bar(smem_u32(&misc->sched_full[asked & 1]), ((asked - 1) >> 1) & 1);
    }
  } else {
    setmaxnreg_dec<40>();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 15) {
    tc_fence_after();
    if (*abort_flag) products_end();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0) report_abort(&misc->abort);
}

}  // namespace attn

// attn_narrow_kernel: fused attention in which every Q tile is worked on by one CTA from its first key to its last (nothing to
// merge between CTAs) by several softmax streams, causal or not: d = 64, and at d = 128 tiles of 128 rows.
//
// At d = 64 the step is bound by the softmax warps' instructions: 256 x 128 exponentials, maxima, conversions and sums take a
// scheduler partition about 1930 cycles however they are written (2040 beside the matrix products), the products 1300.
// attn_fwd_kernel gives a partition two softmax warps of 128 scores a row and takes 2800 cycles a step.  Here it has four, of
// 64 scores a row: a tile of 256 query rows is worked on as four streams, two sub-tiles of 128 rows times the two halves of
// every 128-key tile.  A stream has its own scores, reference, denominator and accumulator in tensor memory (4 x (64 + 64)
// columns: all 512; P overwrites the front of its scores) and its own softmax warpgroup; the two streams of a sub-tile meet
// when the tile is finished, in the epilogue warpgroup, which reads both accumulators.  2600 cycles a step.  In loops of 0.8 s
// (us, attn_fwd_kernel / this kernel): causal 128 heads x 8192 1708 / 1499, 128 x 4096 454 / 413; not causal 900 x 1025 544 / 490, 256 x 1000
// 122 / 117, 128 x 8192 2898 / 2842 (attn_pipe_kernel 2886), 148 x 4096 855 / 864: the power limit takes back a part of what bursts gain (128 x 8192
// 3009 / 2760 in graphs).  In graphs: causal 128 x 2048 141 / 114, 256 x 300 39.1 / 22.2.  Where another kernel is the faster one stands at
// narrow_subs and pipe_tiles (attn_api.cu).
// SUBS = 1 works on tiles of 128 query rows, one sub-tile: its four streams are the two halves of the even and of the odd key
// tiles.  A tile then takes half as long, which evens out the CTAs where a launch has few tiles for each (narrow_subs in
// attn_api.cu), at twice the K and V loads for a row.  At d = 128, where a stream needs 256 columns of tensor memory, two
// streams take the even and the odd key tiles, in that form only.
//   * One barrier each way per step: scores ready (commit of Q K^T, which also says that the stream's P V of the step before
//     is complete) and P ready.  A softmax warp whose reference moved rescales its accumulator itself: that is rare, and
//     no other warp has to be asked.
//     Its waits, and the MMA warps', are those of attn_pipe_kernel, without a vote, and so is its decision to move the reference: with a vote
//     at each wait, the factor computed in every step and the threshold compared after it, 24 shapes of two sub-tiles took 1.02 times as
//     long, 244 of one 1.01 (d = 64), 119 1.02 (d = 128), causal ones 1.01 (us, before / now: 592 x 384 50.9 / 49.4, 1000 x 256 35.1 / 34.6, 32 x 1111, d = 128 31.7 / 31.0).
//   * Every stream has an MMA warp of its own, which issues P V of a step and then Q K^T of the stream's next step: what is in
//     flight for one stream runs under the exponentials of the other three.  One MMA warp that served the streams in turn took
//     800 cycles a turn, waits and instruction issue together, and bound the step at 3200 cycles.
//   * A stage of the K and V ring is waited for by parity, which is exact only for a warp that has seen every phase of the stage:
//     SUBS = 1 has a ring for each parity of the key tiles, and its MMA warps never pass over an item (kv_ring.h).  In loops (us):
//     causal 32 x 1111 16.4, 8 x 4096 30.5 (d = 64), 16 x 2048 27.3 (d = 128); one ring that they stepped through took 16.5, 30.2, 28.2.
//   * Tiles come from the hardware's queue of CTAs not yet started, and the epilogue of a tile runs under the next one, as in
//     attn_pipe_kernel (pipe_kernel.cuh).
#pragma once

#include "attn_kernels.cuh"
#include "kv_ring.h"

namespace attn {

struct NarrowParams {
  int Lq, Lk;              // query rows and keys per head
  int q_tiles;             // Q tiles per head = ceil(Lq / (SUBS * 128))
  int n_steps;             // key steps per head = ceil(Lk / 128)
  int heads;               // B * H
  int group_heads;         // causal: heads whose tiles are dealt out together, longest first
  int stages;              // stages of a ring (kv_ring.h)
  float scale_log2;        // log2(e) / sqrt(d)
  unsigned int* status;    // as in FwdParams
};

// d = 64: four streams, the halves of a key tile; d = 128: two, whole key tiles (SUBS = 1 only).
template <int D>
struct NarrowShape {
  static constexpr int kHalves = D == 64 ? 2 : 1;                // streams that share a key tile
  static constexpr int kStreams = 2 * kHalves;
  static constexpr int kKeys = 128 / kHalves;                    // keys of a stream's step
  static constexpr int kEpiWarp = 4 * kStreams, kMmaWarp = kEpiWarp + 4, kLoadWarp = kMmaWarp + kStreams, kAllocWarp = kLoadWarp + 1;
  // d = 64: 16 softmax warps, 4 epilogue, 4 MMA, TMA, tensor-memory allocation, 2 idle; registers 896 x 72 at launch, then 512 x 96
  // and 384 x 40.  d = 128: 8, 4, 2, 1, 1; 512 x 128 at launch, then 256 x 192 and 256 x 64.
  static constexpr int kThreads = D == 64 ? 896 : 512;
  static constexpr int kSoftmaxRegs = D == 64 ? 96 : 192, kOtherRegs = D == 64 ? 40 : 64;
  static constexpr int kSchedReaders = kLoadWarp + 1;            // warps that read a tile's index
};
template <int D, int SUBS>
struct NarrowSmem {
  static_assert(D == 64 || SUBS == 1, "no room for the second sub-tile");
  static constexpr int kSubBytes = kSub * D * 2;                 // one sub-tile of Q
  static constexpr int kQBytes = 2 * SUBS * kSubBytes;           // two tiles
  static constexpr int kStageBytes = 128 * D * 2;
  static constexpr int kChunks = D == 64 ? 2 : 1;                // [32 rows][64 columns] bf16 output chunks per epilogue warp
  static constexpr int kOutBytes = 4 * kChunks * 4096;
  static constexpr int kMiscBytes = 9216;
  __host__ __device__ static constexpr int total(int stages) { return kQBytes + stages * kStageBytes + kOutBytes + kMiscBytes; }   // of all rings
};

struct NarrowMisc {
  float2 stat[2][4][kSub];                 // [the sub-tile's tiles mod 2][stream][row] reference and denominator of a finished tile
  uint4 sched[2];                          // answers of try_cancel (16 bytes each)
  uint64_t sched_full[2], sched_empty[2];
  uint64_t q_full[2][2], q_empty[2][2];    // [sub-tile][buffer]
  uint64_t kv_full[kMaxStages], kv_empty[kMaxStages];
  uint64_t s_full[4], p_full[4];           // per stream
  uint64_t fin_full[4];                    // per stream
  uint64_t o_full[2], o_free[2];           // per sub-tile
  AbortCell abort;
  uint32_t tmem_slot;
};
static_assert(sizeof(NarrowMisc) <= NarrowSmem<64, 2>::kMiscBytes, "misc region too large");

// A tile: its head, first row, key tiles and the number of them that each of its streams works on.  Stream st: sub-tile st / 2,
// half st % 2 of every key tile; SUBS = 1: half st % 2 of the key tiles j with j % 2 = st / 2.
template <int SUBS>
struct NarrowWork {
  int bh, q_row0, n, n0, n1;               // n: key tiles; n0, n1: those of streams 0, 1 and of streams 2, 3
  __device__ __forceinline__ int steps(int group) const { return group ? n1 : n0; }
};
template <bool CAUSAL, int SUBS>
__device__ __forceinline__ NarrowWork<SUBS> narrow_work(int index, const NarrowParams& p) {
  NarrowWork<SUBS> w;
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
  w.q_row0 = q * SUBS * kSub;
  if constexpr (SUBS == 2) {
    // (causal: a sub-tile's last key tile is the one that holds its own rows)
    w.n0 = CAUSAL ? 2 * q + 1 : p.n_steps;
    w.n1 = w.q_row0 + kSub >= p.Lq ? 0 : CAUSAL ? 2 * q + 2 : p.n_steps;
    w.n = w.n1 > w.n0 ? w.n1 : w.n0;
  } else {
    w.n = CAUSAL ? q + 1 : p.n_steps;
    w.n0 = (w.n + 1) / 2;
    w.n1 = w.n / 2;
  }
  return w;
}

template <int D, bool CAUSAL, int SUBS>
__global__ void __launch_bounds__(NarrowShape<D>::kThreads, 1)
attn_narrow_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o, const NarrowParams p) {
  using SH = NarrowShape<D>;
  using SM = NarrowSmem<D, SUBS>;
  using RINGS = KvRings<SUBS>;
  constexpr int TKV = 128, HKV = SH::kKeys, KCH = D / 64, NCH = HKV / 32, HALVES = SH::kHalves;
  constexpr int O_COL0 = SH::kStreams * HKV;
  constexpr int kPoly = kPolyPairsPer8;
  constexpr int kParts = SH::kStreams / SUBS;         // streams of a sub-tile

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t ring_smem = smem_base + SM::kQBytes;
  const uint32_t out_smem = ring_smem + RINGS::kRings * p.stages * SM::kStageBytes;
  NarrowMisc* const misc = reinterpret_cast<NarrowMisc*>(smem_raw + SM::kQBytes + RINGS::kRings * p.stages * SM::kStageBytes + SM::kOutBytes);
  volatile int* abort_flag = &misc->abort.flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    abort_cell_init(&misc->abort, p.status);
    if (smem_base & 1023u) note_timeout(wait_info(kRoleLoad, 0, 0xFFFF), &misc->abort.flag);   // swizzled tiles need 1024-byte alignment
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&misc->kv_full[s]), 1);
      mbar_init(smem_u32(&misc->kv_empty[s]), HALVES * SUBS);     // the streams that read a stage
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(smem_u32(&misc->s_full[i]), 1);
      mbar_init(smem_u32(&misc->p_full[i]), kSub);
      mbar_init(smem_u32(&misc->fin_full[i]), kSub);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&misc->sched_full[i]), 1);
      mbar_init(smem_u32(&misc->sched_empty[i]), SH::kSchedReaders);
      for (int b = 0; b < 2; ++b) {
        mbar_init(smem_u32(&misc->q_full[i][b]), 1);
        mbar_init(smem_u32(&misc->q_empty[i][b]), kParts);        // the sub-tile's streams
      }
      mbar_init(smem_u32(&misc->o_full[i]), kParts);
      mbar_init(smem_u32(&misc->o_free[i]), kSub);
    }
    fence_mbar_init();
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
    prefetch_tmap(&tm_o);
  }
  if (warp == SH::kAllocWarp) {
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

  if (warp < SH::kEpiWarp) {
    // ===================================================== softmax warpgroup of one stream
    setmaxnreg_inc<SH::kSoftmaxRegs>();
    const int st = warp >> 2, group = st / HALVES, half = st % HALVES, i = SUBS == 2 ? group : 0;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_tmem = lane_base + st * HKV;      // P goes to the front of it
    const uint32_t bar_s = smem_u32(&misc->s_full[st]);
    const uint32_t bar_p = smem_u32(&misc->p_full[st]);
    const float scale = p.scale_log2;
    const ExpConsts ek = make_exp_consts(scale);
    const int kv_tail = CAUSAL ? 0 : p.Lk & (TKV - 1);
    bool ok = run, dead = false;
    uint32_t g = 0, done = 0;                          // steps of this stream over all tiles; finished tiles
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const NarrowWork<SUBS> w = narrow_work<CAUSAL, SUBS>(tile, p);
      const int n = w.steps(group);
      if (n > 0) {
        // whether this stream's last key tile is the tile's last (SUBS = 1: the last tile is one parity's)
        const bool ends = SUBS == 2 || ((w.n - 1) & 1) == group;
        float m_run = -INFINITY, delta = 0.f, lim_move = 0.f;   // lim_move: as in attn_pipe_kernel
        // One key step.  The masked variant (the causal diagonal, a ragged last key tile) is compiled separately so that the
        // common step pays nothing for it; `lim` is the last key column of this half the thread's row may attend to.
        auto softmax_step = [&](auto mask_tag, int lim, bool first, bool last) __attribute__((always_inline)) -> bool {
          constexpr bool kMasked = decltype(mask_tag)::value;
          wait_on(bar_s, g & 1, abort_flag, wait_info(kRoleSoftmax, kBarSFull, g), dead);
          tc_fence_after();
          uint32_t s[HKV];
          // load the row in two halves: the maximum of the first half is taken while the second is in flight
#pragma unroll
          for (int c = 0; c < NCH / 2; ++c) tmem_ld32_nowait(s_tmem + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
#pragma unroll
          for (int c = 0; c < NCH / 2; ++c) tmem_ld_fence(*reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
#pragma unroll
          for (int c = NCH / 2; c < NCH; ++c) tmem_ld32_nowait(s_tmem + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
          // keys past the end or after the query's position: score -inf, never zero
          if constexpr (kMasked) {
#pragma unroll
            for (int k = 0; k < HKV / 2; ++k)
              if (k > lim) s[k] = 0xFF800000u;
          }
          const float mx_a = max_nan(chain_max<0, HKV / 4>(s), chain_max<HKV / 4, HKV / 2>(s));
#pragma unroll
          for (int c = NCH / 2; c < NCH; ++c) tmem_ld_fence(*reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
          if constexpr (kMasked) {
#pragma unroll
            for (int k = HKV / 2; k < HKV; ++k)
              if (k > lim) s[k] = 0xFF800000u;
          }
          const float mx = max3_nan(mx_a, chain_max<HKV / 2, 3 * HKV / 4>(s), chain_max<3 * HKV / 4, HKV>(s));
          // Lazy rescale, as in attn_fwd_kernel.  The reference is finite from the first step on, also where a stream's
          // half of the keys holds none that the row may attend to.
          const float m_cand = max_nan(mx * scale, kEmptyReference);
          const float gap = m_cand - m_run;
          const bool move = !(gap <= lim_move);        // (a NaN moves it)
          m_run = move ? m_cand : m_run;
          // The step before is complete (see s_full), so the accumulator may be rescaled here; P V of this step waits for P.
          if (__any_sync(0xffffffffu, move)) {
            const float alpha = move ? ex2_approx(-gap) : 1.0f;
            delta *= alpha;
            if (!first) {
              const uint32_t o_tmem = lane_base + O_COL0 + st * D;
#pragma unroll 1
              for (int c = 0; c < D / 16; ++c) {
                uint32_t r[16];
                tmem_ld16(o_tmem + c * 16, r);
#pragma unroll
                for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) * alpha);
                tmem_st16(o_tmem + c * 16, r);
              }
            }
          }
          const uint64_t neg_m2 = pack_f32x2(-m_run, -m_run);
          uint64_t sum2 = 0ull;                        // packed (0.f, 0.f)
#pragma unroll
          for (int c = 0; c < NCH; ++c) {
            uint32_t pk[16];
            exp_chunk<kPoly>(&s[c * 32], ek, neg_m2, sum2, pk);
            tmem_st16(s_tmem + c * 16, pk);
          }
          float sum0, sum1;
          unpack_f32x2(sum2, sum0, sum1);
          delta += sum0 + sum1;
          if (last) {
            // The epilogue warpgroup finishes the tile.  It has read what stood here two tiles ago: this tile's first scores
            // came after the first P V of the tile before, which waited for that (o_free).  The arrival stands before the one
            // on p_full: a thread that is a tile ahead has seen scores that came after every thread's p_full, so it cannot
            // make its next arrival here before a slow thread has made this one.
            // (A tile of one step: its only scores did not wait for the epilogue of the tile before, which may still be
            // waiting for that tile's arrivals here.)
            if (first && done > 0 && !wait_quiet_warp(smem_u32(&misc->o_free[i]), (done - 1) & 1, abort_flag, wait_info(kRoleSoftmax, kBarOFull, g))) return false;
            misc->stat[done & 1][st][row] = make_float2(m_run, delta);
            mbar_arrive(smem_u32(&misc->fin_full[st]));
          }
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(bar_p);
          lim_move = fminf(fmaxf(lg2_approx(delta) - 4.0f, 0.f), kRescaleThreshold);
          return !any_dead(dead);
        };
        for (int jj = 0; ok && jj < n; ++jj, ++g) {
          // Only the last step may need a mask: the causal diagonal, which starts at the sub-tile's first row and ends, in a
          // ragged last key tile, before the padding for every row of the sequence; else a ragged last key tile.
          const bool last = jj == n - 1;
          if (last && ends && (CAUSAL || kv_tail != 0)) ok = softmax_step(MaskTag<true>{}, (CAUSAL ? row : kv_tail - 1) - half * HKV, jj == 0, true);
          else ok = softmax_step(MaskTag<false>{}, HKV - 1, jj == 0, (!CAUSAL || SUBS == 1) && last);
        }
        if (!ok) break;
        ++done;
      } else if (SUBS == 1) {
        // (no key tile of this parity: an empty part, so that the epilogue finds four)
        if (done > 0 && !wait_quiet_warp(smem_u32(&misc->o_free[0]), (done - 1) & 1, abort_flag, wait_info(kRoleSoftmax, kBarOFull, g))) { ok = false; break; }
        misc->stat[done & 1][st][row] = make_float2(-INFINITY, 0.f);
        mbar_arrive(smem_u32(&misc->fin_full[st]));
        ++done;
      }
      tile = next_tile(seq, kRoleSoftmax);
    }
  } else if (warp < SH::kMmaWarp) {
    // ================================================== epilogue warpgroup
    setmaxnreg_dec<SH::kOtherRegs>();
    const int wq = warp & 3, row = wq * 32 + lane;
    const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
    const uint32_t stage_w = out_smem + wq * (SM::kChunks * 4096);     // this warp's staging chunks
    bool ok = run;
    uint32_t fin = 0, chunk = 0;                       // bit i: finished tiles of sub-tile i, mod 2; next staging chunk
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const NarrowWork<SUBS> w = narrow_work<CAUSAL, SUBS>(tile, p);
#pragma unroll 1
      for (int i = 0; ok && i < SUBS; ++i) {
        if (SUBS == 2 && w.steps(i) == 0) continue;
        const uint32_t ph = (fin >> i) & 1;
        fin ^= 1u << i;
        float wt[kParts], m = -INFINITY, sum = 0.f;
#pragma unroll
        for (int k = 0; k < kParts; ++k)
          if (ok && !wait_quiet_warp(smem_u32(&misc->fin_full[HALVES * i + k]), ph, abort_flag, wait_info(kRoleCorrection, kBarAlpha, HALVES * i + k))) ok = false;
        if (!ok) break;
        // the streams' parts on the common reference, normalised
#pragma unroll
        for (int k = 0; k < kParts; ++k) m = fmaxf(m, misc->stat[ph][HALVES * i + k][row].x);
#pragma unroll
        for (int k = 0; k < kParts; ++k) {
          const float2 a = misc->stat[ph][HALVES * i + k][row];
          wt[k] = ex2_approx(a.x - m);                 // (an empty part: -inf, weight 0)
          sum += a.y * wt[k];
        }
        const float inv = row_inverse(sum, m);
#pragma unroll
        for (int k = 0; k < kParts; ++k) wt[k] *= inv;
        if (!wait_quiet_warp(smem_u32(&misc->o_full[i]), ph, abort_flag, wait_info(kRoleCorrection, kBarOFull, i))) { ok = false; break; }
        tc_fence_after();
        const bool empty = SUBS == 1 && w.n1 == 0;     // the streams of the odd key tiles have no accumulator
        const uint32_t o_tmem = lane_base + O_COL0 + HALVES * i * D;
#pragma unroll 1
        for (int h = 0; h < KCH; ++h) {
          const uint32_t dst = stage_w + chunk * 4096;
          chunk = chunk + 1 < SM::kChunks ? chunk + 1 : 0;
          // the store that last read this chunk must have finished reading it
          if (lane == 0) {
            if (SM::kChunks == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            else tma_store_wait_read();
          }
          __syncwarp();
#pragma unroll 1
          for (int c = 0; c < 8; ++c) {                // 8 columns at a time
            const uint32_t col = o_tmem + h * 64 + c * 8;
            uint32_t ra[8], rb[8];
            float v[8];
            tmem_ld8x2(col, col + D, ra, rb);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              v[e] = __uint_as_float(ra[e]) * wt[0];
              if (HALVES == 2 || !empty) v[e] += __uint_as_float(rb[e]) * wt[1];
            }
            if (kParts == 4 && !empty) {
              tmem_ld8x2(col + 2 * D, col + 3 * D, ra, rb);
#pragma unroll
              for (int e = 0; e < 8; ++e) v[e] += __uint_as_float(ra[e]) * wt[kParts - 2] + __uint_as_float(rb[e]) * wt[kParts - 1];
            }
            uint32_t q[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) q[e] = pack_bf16x2(v[2 * e], v[2 * e + 1]);
            st_shared_u4(dst + lane * 128 + (((uint32_t)c ^ (uint32_t)(lane & 7)) << 4), q);   // 128-byte swizzle
          }
          if (h == KCH - 1) {
            tc_fence_before();
            mbar_arrive(smem_u32(&misc->o_free[i]));   // every accumulator has been read
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {                             // (rows past the end of the sequence are clipped by the tensor map)
            tma_store_3d(&tm_o, dst, h * 64, w.q_row0 + i * kSub + wq * 32, w.bh);
            tma_store_commit();
          }
        }
      }
      if (!ok) break;
      tile = next_tile(seq, kRoleCorrection);
    }
    if (lane == 0) tma_store_wait_read();              // shared memory is read by the stores until here
    __syncwarp();
  } else if (warp < SH::kLoadWarp) {
    // ============================== MMA issuer of one stream (the whole warp walks the loop, one lane issues)
    setmaxnreg_dec<SH::kOtherRegs>();
    const int st = warp - SH::kMmaWarp, group = st / HALVES, half = st % HALVES, i = SUBS == 2 ? group : 0;
    bool ok = run, dead = false;
    const uint32_t s_tmem = tmem_base + st * HKV, o_tmem = tmem_base + O_COL0 + st * D;
    const uint32_t k_smem = ring_smem + half * (HKV * 128);       // this stream's keys in a ring item
    uint32_t g = 0, done = 0, q_uses = 0;              // steps; finished tiles; Q loads that have been read
    const int first_stage = RINGS::of_group(group) * p.stages;
    KvRing ring = {first_stage, 0u};                   // K and V of this stream's key tiles, one after another, over all tiles
    auto wait = [&](uint64_t* bar, uint32_t parity, uint32_t id) __attribute__((always_inline)) {
      wait_on(smem_u32(bar), parity, abort_flag, wait_info(kRoleMma, id, 0x100 * st + (g & 0xFF)), dead);
    };
    // Waits for the ring's next item and passes it; its stage.
    auto take = [&]() __attribute__((always_inline)) -> int {
      const int stage = ring.pos;
      wait(&misc->kv_full[stage], ring.phase, kBarKvFull);
      ring.advance(first_stage, p.stages);
      return stage;
    };
    // (one lane) Scores of the keys in stage k; last: no later step of the tile reads this Q.
    auto issue_scores = [&](int k, bool last) __attribute__((always_inline)) {
      const int b = (q_uses - 1) & 1;
      issue_qk<D, HKV>(s_tmem, smem_base + (b * SUBS + i) * SM::kSubBytes, k_smem + k * SM::kStageBytes);
      umma_commit(smem_u32(&misc->s_full[st]));
      umma_commit(smem_u32(&misc->kv_empty[k]));
      if (last) umma_commit(smem_u32(&misc->q_empty[i][b]));
    };
    // Key steps that this stream's sub-tile does not run: their ring items are passed on as soon as they have arrived.
    auto skip = [&](int steps) __attribute__((always_inline)) {
#pragma unroll 1
      for (int x = 0; x < 2 * steps; ++x) {
        const int stage = take();
        if (lane == 0 && !dead) mbar_arrive(smem_u32(&misc->kv_empty[stage]));
      }
    };
    // A tile's first scores.
    auto start = [&](int steps) __attribute__((always_inline)) {
      wait(&misc->q_full[i][q_uses & 1], (q_uses >> 1) & 1, kBarQ);
      const int k = take();
      ++q_uses;
      tc_fence_after();
      if (may_issue(dead)) issue_scores(k, steps == 1);
      __syncwarp();
    };
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const NarrowWork<SUBS> w = narrow_work<CAUSAL, SUBS>(tile, p);
      const int n = w.steps(group);
      if (n > 0) start(n);
      for (int j = 0; ok && j < n; ++j, ++g) {
        const int v = take();
        const bool more = j + 1 < n;
        const int k = more ? take() : 0;
        // the tile before has left the accumulator
        if (j == 0 && done > 0) wait(&misc->o_free[i], (done - 1) & 1, kBarOFull);
        wait(&misc->p_full[st], g & 1, kBarPFull);
        tc_fence_after();
        if (may_issue(dead)) {
          issue_pv<D, HKV>(o_tmem, s_tmem, k_smem + v * SM::kStageBytes, j > 0, TKV * 128, 1024);
          umma_commit(smem_u32(&misc->kv_empty[v]));
          if (more) issue_scores(k, j + 2 == n);
          else umma_commit(smem_u32(&misc->o_full[i]));
        }
        __syncwarp();
        if (any_dead(dead)) ok = false;
      }
      if (!ok) break;
      if constexpr (SUBS == 2) {
        done += n > 0 ? 1u : 0u;
        if (CAUSAL || n == 0) skip(w.n - n);
      } else {
        ++done;
        if (n == 0) {
          // nothing to add to the tile, nothing read of its Q (the arrivals of the tile before must all have been made: o_free)
          if (done > 1) wait(&misc->o_free[0], (done - 2) & 1, kBarOFull);
          wait(&misc->q_full[0][q_uses & 1], (q_uses >> 1) & 1, kBarQ);
          if (lane == 0 && !dead) {
            mbar_arrive(smem_u32(&misc->q_empty[0][q_uses & 1]));
            mbar_arrive(smem_u32(&misc->o_full[0]));
          }
          ++q_uses;
        }
      }
      if (any_dead(dead)) break;
      tile = next_tile(seq, kRoleMma);
    }
  } else if (warp == SH::kLoadWarp) {
    // ================================================== TMA producer, and the requests for the next tile
    setmaxnreg_dec<SH::kOtherRegs>();
    bool ok = run;
    int asked = 0;                                     // requests made
    KvRing ring0 = {0, 0u}, ring1 = {p.stages, 0u};
    uint32_t q_loads0 = 0, q_loads1 = 0;
    // (the waits are taken by the whole warp, the copies issued by one lane)
    auto load_kv = [&](const CUtensorMap* tm, int j, int bh) __attribute__((always_inline)) -> bool {
      const int r = RINGS::of_key_tile(j);
      KvRing ring = r ? ring1 : ring0;
      const int stage = ring.pos;
      if (!wait_quiet_warp(smem_u32(&misc->kv_empty[stage]), ring.phase ^ 1u, abort_flag, wait_info(kRoleLoad, kBarKvEmpty, j))) return false;
      if (elect_one()) {
        const uint32_t bar = smem_u32(&misc->kv_full[stage]);
        mbar_arrive_expect_tx(bar, SM::kStageBytes);
#pragma unroll
        for (int c = 0; c < KCH; ++c) tma_load_3d(ring_smem + stage * SM::kStageBytes + c * (TKV * 128), tm, c * 64, j * TKV, bh, bar);
      }
      __syncwarp();
      ring.advance(r * p.stages, p.stages);
      if (r) ring1 = ring; else ring0 = ring;
      return true;
    };
    auto load_q = [&](int i, const NarrowWork<SUBS>& w) __attribute__((always_inline)) -> bool {
      const uint32_t u = i ? q_loads1 : q_loads0, b = u & 1;
      if (u >= 2 && !wait_quiet_warp(smem_u32(&misc->q_empty[i][b]), (u / 2 - 1) & 1, abort_flag, wait_info(kRoleLoad, kBarQ, u))) return false;
      if (elect_one()) {
        const uint32_t bar = smem_u32(&misc->q_full[i][b]);
        mbar_arrive_expect_tx(bar, SM::kSubBytes);
#pragma unroll
        for (int c = 0; c < KCH; ++c)
          tma_load_3d(smem_base + (b * SUBS + i) * SM::kSubBytes + c * (kSub * 128), &tm_q, c * 64, w.q_row0 + i * kSub, w.bh, bar);
      }
      __syncwarp();
      if (i) ++q_loads1; else ++q_loads0;
      return true;
    };
    int tile = blockIdx.x;
    for (int seq = 1; ok && tile >= 0; ++seq) {
      const NarrowWork<SUBS> w = narrow_work<CAUSAL, SUBS>(tile, p);
      const int n = w.n;
      // the first product needs K_0 and Q of sub-tile 0; the first tile's Q buffer is free at once
      if (seq == 1) ok = load_q(0, w);
      if (ok) ok = load_kv(&tm_k, 0, w.bh);
      if (ok && seq > 1) ok = load_q(0, w);
      if (ok && SUBS == 2 && w.n1 > 0) ok = load_q(1, w);
      for (int j = 0; ok && j < n; ++j) {
        if (j > 0) ok = load_kv(&tm_k, j, w.bh);
        if (ok && j == n - 1) {
          // Ask for the tile after this one, into the slot that held the tile before this one -- as late as the answer is
          // sure to be back in time (a ring's depth ahead of the MMA warp): a tile asked for early would be tied to this
          // CTA while others run dry.
          if (seq >= 3)
            ok = wait_quiet_warp(smem_u32(&misc->sched_empty[seq & 1]), ((seq - 3) >> 1) & 1, abort_flag, wait_info(kRoleLoad, kBarSync, seq));
          if (!ok) break;
          if (elect_one()) {
            mbar_arrive_expect_tx(smem_u32(&misc->sched_full[seq & 1]), 16);
            clc_try_cancel(smem_u32(&misc->sched[seq & 1]), smem_u32(&misc->sched_full[seq & 1]));
          }
          __syncwarp();
          asked = seq;
        }
        if (ok) ok = load_kv(&tm_v, j, w.bh);
      }
      if (!ok) break;
      tile = next_tile(seq, kRoleLoad);
    }
    grid_release();
    if (tile == -2) ok = false;
    if (!ok && lane == 0) {
      // Drain: every copy started here must land before the CTA may exit, and so must an answer still on its way.
      for (int s = 0; s < RINGS::kRings * p.stages; ++s)
        drain_bar(smem_u32(&misc->kv_full[s]), (s < p.stages ? ring0 : ring1).last_parity(s));
      for (int i = 0; i < SUBS; ++i)
        for (uint32_t q = i ? q_loads1 : q_loads0, u = q > 2u ? q - 2u : 0; u < q; ++u) drain_bar(smem_u32(&misc->q_full[i][u & 1]), (u / 2) & 1);
      if (asked > 0) drain_bar(smem_u32(&misc->sched_full[asked & 1]), ((asked - 1) >> 1) & 1);
    }
  } else {
    setmaxnreg_dec<SH::kOtherRegs>();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == SH::kAllocWarp) {
    tc_fence_after();
    if (*abort_flag) products_end();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0) report_abort(&misc->abort);
}

}  // namespace attn

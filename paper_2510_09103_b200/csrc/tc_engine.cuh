// A persistent, warp-specialised tcgen05 engine that runs a table of "items".  An item is a short
// list of K-loops ("segments") that accumulate into 128-row accumulators in tensor memory,
// followed by an epilogue that turns the accumulators into the result of one step of Algorithm 2.
// It has two forms: panel items run on pairs of CTAs (cta_group::2, M = 256), Gram items on single ones.
//
//   refit of L (row panels of 128 rows of a block, Algorithm 2's L update):
//       D = g R^T + [L hi | L lo] X + [L0 hi | L0 lo] Y     X = [Bop1; Bop1], Bop1 = -(R R^T)/(1-b1)
//       L' = L + eta (1-b1) D                               Y = [Bop2; Bop2], Bop2 = b1 (R0 R^T)/(1-b1)
//   refit of R (column panels of 128 columns, the R update, computed transposed):
//       D = g^T L + [R^T hi | R^T lo] X' + [R0^T hi | R0^T lo] Y'   with -(L^T L)/(1-b1), b1 (L0^T L)/(1-b1)
//       R'^T = R^T + eta (1-b1) D
//   Gram item: one of the r x r matrices above, scaled and stored as a split-bf16 operand, twice, one
//       copy below the other, so that the hi and the lo columns of a factor meet the same rows.
//
// fp32 factors are carried into the bf16 tensor cores as hi + lo pairs (two bf16 numbers whose sum
// has ~16 significant bits); gradients are bf16 already and enter unchanged.  Operands with hi and
// lo parts are stored side by side ([rows, 2 half]: hi columns from 0, lo columns from `half`;
// half = rp = r rounded up to 16 while 2 rp <= 256, else rp rounded up to 64), so that used as the
// N side of an MMA the two parts land in two column ranges of the accumulator, which the epilogue
// adds.  In a pair the CTA of rank 0 holds the hi columns of B and the other one the lo columns; one MMA of N = 2 rp takes
// both up to rank 128, above that the first takes N = 256 (128 columns of each part) and a second one the rest.  A Gram item
// above rank 128 takes one MMA of N = rp for the hi and one for the lo part, which starts at a chunk of its own.
// (Letting both add to the same columns would free half of the accumulator, but the small products then meet the
// rounding of the large sums: errors of L R against 64 bits up to twice as large at ranks 128 to 256.)
//
// A stage of the shared-memory ring holds `stage_k` (64 or 128) of K:
//   A  up to three operands of 128 rows x stage_k (K along x: boxes of 64 x 128) or stage_k x 128
//      columns (K along y: two boxes of 64 x stage_k).  All are multiplied with the same B and fill
//      one accumulator each: the more operands share a B, the fewer bytes a flop brings in
//   B  stage_k rows of 64-column chunks of a [rows, 2 half] array, i.e. the N side read MN-major with its chunks one box
//      apart; in a pair each CTA's own part
// Why pairs: with M = 128 every MMA reads A and all of B from the shared memory of its SM and every CTA brings in all of
// B, 115 of the 128 bytes a cycle an SM's shared memory delivers at rank 80 before the fills; at rank 204, where tensor
// memory has room for one panel, four fifths of the fills are B.  A pair reads and fills half of B per SM.  A panel launch,
// one CTA -> pair: 3.65 -> 2.5 ms on eight layers of the 8B shapes, 1.20 -> 1.11 ms on the 1.5B set, 437 -> 370 us on the
// 350M set at rank 128, 172 -> 147 at rank 8.  What is left there: the power cap (SM clocks of 1.3 to 1.5 GHz while these
// launches run) and, per stage, the serial path of the warp that issues the MMAs.
// Warp roles (512 threads, 128 registers each): warp 0 loads A, warp 3 loads B, warp 1 issues the MMAs (in a pair that of
// rank 0, for both), warps 4-7 add up g^2 per row from the gradient tiles of the first segment when the launch asks for it
// (the second-moment statistic of the block-mean form then needs no pass of its own over g), warps 8-15 drain the
// accumulators (two groups of four warps that take the 16-column pieces of an item alternately).  The issuing warps run
// dependent scalar code, so their per-stage instruction count bounds the rate; all lanes run the loops on values that the
// compiler knows to be uniform (mbar_wait_warp, uniform).
// The copies of both CTAs of a pair are counted at the barriers of rank 0, whose MMAs read them; rank 1 learns from the commit
// of those MMAs that a stage of its own has been filled and multiplied.  The row sums of rank 1 are therefore made between the
// MMAs of a stage and its next fill, those of rank 0 beside the MMAs.  (A commit ahead of the MMAs, to let rank 1 start with
// them: 871 -> 862 us per step where the ring has three stages, 9.11 -> 9.16 ms on the 1.5B set.)
// With two accumulator buffers the epilogue of one item overlaps the K-loops of the next.
// Every wait is bounded; when one runs out the CTA records a status bit, stops taking work, tells the other CTA of its
// pair to do the same and leaves through the common exit (which frees its tensor memory).  A launch that finds the status
// word set on entry does nothing.
#pragma once

#include <cuda.h>

#include "tc_common.cuh"

namespace adapm {
namespace tc {

constexpr int kMaxSegs = 4;
constexpr int kMaxA = 3;
constexpr int kEngineThreads = 512;
constexpr uint32_t kTeamSpinDefault = 1u << 22;   // polls of 256 ns each: about a second
constexpr uint32_t kDrainSpins = 1u << 16;         // for the copies in flight when a CTA gives up: 4 to 70 milliseconds in all
constexpr uint32_t kWaitSpinDefault = 1u << 23;   // mbarrier polls of 0.3 to 1.3 us: 2 to 10 seconds, longer than a team wait

enum : int32_t { EPI_FACTOR = 0, EPI_GRAM = 1, EPI_NONE = 2 };   // EPI_NONE: a filler that only keeps a CTA in step

struct Seg {
  int32_t map_a;             // 2-D tensor map: boxes of 64 x 128 (a_mode 0) or 64 x stage_k (a_mode 1)
  int32_t map_b;             // one CTA: 3-D tensor map (64, rows, chunks), box 64 x stage_k x chunks; pair: 2-D, boxes of 64 x stage_k
  int32_t ax[kMaxA], ay[kMaxA];   // element coordinates of the first box of each A operand
  int32_t k;                 // K extent, multiple of 16
  uint32_t tx_bytes;         // bytes one stage of this segment brings into a CTA
  int16_t a_mode;            // 0: K runs along x (K-major A), 1: K runs along y (MN-major A)
  int16_t n;                 // N of one MMA (multiple of 16, <= 256)
  int16_t n_a;               // A operands of a CTA (1..kMaxA)
  int16_t n2;                // N of a second MMA per K step that reads B from chunk b2_chunk and adds at +d_part, or 0
  int16_t d_col[kMaxA];      // accumulator column of each A operand
  int16_t first;             // 1: its first MMA overwrites the accumulators
  int16_t b2_chunk, d_part;
  int16_t same_acc;          // 1: the A operands share one accumulator (all but the first always accumulate)
  int16_t n_b, b_x;          // pair: boxes of B per CTA, and the column of B at which the part of the CTA of rank 1 starts
};

struct Item {
  Seg seg[kMaxSegs];
  int32_t n_seg;
  int32_t epi;
  // EPI_FACTOR: a CTA has n_pan panels, those of the CTA of rank 1 (and its A operands) follow on those of rank 0, and
  // panels beyond own_count do not exist.  Panel p has its accumulator at column acc_stride * p; the thread that owns
  // accumulator row q of panel p updates factor entries (owner = first + 128 p + q, k):
  //   new[owner][k] = old[owner][k] + coef * (D hi[q][k] + D lo[q][k])                 k < r
  //   dst[owner][k] = hi, dst[owner][half + k] = lo                                    k < rp
  // Old and new fp32 values live in the state, f32[own_stride * owner + k_stride * k], or in the workspace in the order
  // in which the epilogue's threads take them (iter_at).
  // EPI_GRAM: G[own0 + q][k] = coef * sum over n_sum parts (rp columns apart) of D[q][k]; stored like dst above,
  //   and once more stack_rows rows below                                              own0 + q, k < rp
  int32_t own0, own_count;   // first owner of the item and number of owners of the whole matrix
  int32_t n_pan, acc_stride;
  int32_t r, rp, half;
  int32_t n_sum, stack_rows;
  int32_t dst_ld;            // row pitch of the destination in elements
  int64_t f32_off;           // float offset of the factor in the state buffer
  int64_t iter_off;          // float offset in the workspace of its values between two passes
  int32_t from_iter, to_iter;   // 1: old values come from there, new values go there
  int64_t own_stride, k_stride;
  int64_t dst_off;           // bf16 element offset of the destination array in the workspace
  int64_t sumsq_off;         // float offset in the workspace of the row sums of g^2 (row own0 first), or -1
  // Pacing of a team of CTAs that work through the same blocks (so that their reads of g meet in L2): before its
  // first load the item waits until team_counters[team] >= wait_count, after its last load it adds `signal`.
  // Pacing only: no data depends on it.
  int16_t team, signal;
  int32_t wait_count;
  float coef;
  int32_t cost;              // stages, for scheduling
};

// the fields of an Item its epilogue needs
struct ItemEpi {
  int32_t epi, own0, own_count, n_pan, acc_stride, r, rp, half, n_sum, stack_rows, dst_ld;
  int32_t from_iter, to_iter;
  int64_t f32_off, iter_off, own_stride, k_stride, dst_off;
  float coef;
};

struct EngineArgs {
  const Item* items;
  int32_t n_items;
  const CUtensorMap* maps;
  float* f32_base;           // state buffer
  uint16_t* work_bf16;       // workspace viewed as bf16
  float* work_f32;           // workspace viewed as fp32 (row sums of g^2)
  int32_t* status;
  int32_t stage_k;           // 64 or 128
  int32_t stage_bytes;       // a_bytes + stage_k * 128 * (largest number of 64-column chunks of B)
  int32_t a_bytes;           // room for the A operands of a stage: (most operands of any segment) * 256 * stage_k
  int32_t n_stages;
  int32_t acc_cols;          // tensor-memory columns per accumulator buffer
  int32_t n_acc;             // 1 or 2 accumulator buffers
  const int32_t* cta_begin;  // CTA c runs items [cta_begin[c], cta_begin[c + 1]) in order
  int32_t sum_col;           // EPI_FACTOR: first of the tensor-memory columns the epilogue parks D0 + D1 in, or -1
  int32_t sumsq_on;          // 1: warps 4-7 follow the stages and sum g^2 for items that have sumsq_off >= 0
  int32_t* team_counters;    // one counter per team, zero at launch (nullptr when no item waits)
  uint32_t team_spin_limit[2];   // of the CTAs of a pair
  uint32_t wait_spin_limit;
  const float* gscale;       // device scalar: every gradient counts as gscale[0] * g (nullptr: 1)
};

struct __align__(8) EngineShared {
  uint64_t full[8], empty[8], summed[8], tfull[2], tempty[2];
  uint32_t tmem_base;
  int abort, skip;
};

// The A operands of one stage, NBOX boxes each.  Compile-time counts keep the issuing thread's instruction stream short (it
// runs dependent scalar code; its rate bounds the pipeline).
template <bool PAIR, int NA, int NBOX>
__device__ __forceinline__ void load_operands(uint8_t* sa, int a_tile, int box_bytes, const CUtensorMap* ma, const int* x,
                                              const int* y, uint64_t* bar, uint32_t pair_bar) {
#pragma unroll
  for (int p = 0; p < NA; ++p)
#pragma unroll
    for (int j = 0; j < NBOX; ++j) {
      if (PAIR) tma_load_box_pair(sa + p * a_tile + j * box_bytes, ma, x[p] + 64 * j, y[p], pair_bar);
      else tma_load_box(sa + p * a_tile + j * box_bytes, ma, x[p] + 64 * j, y[p], bar);
    }
}

// Lets the copies already issued into a ring of `n_stages` land before the CTA exits.  (stage, phase): where the next would go.
// (Rank 1 of a pair has no barrier that counts its own: it allows them a few milliseconds, a thousand times what a copy takes.)
template <bool PAIR>
__device__ __forceinline__ void drain_ring(uint64_t* full, int stage, uint32_t phase, uint32_t issued, int n_stages, uint32_t rank) {
  if (PAIR && rank != 0) {
    for (uint32_t spin = 0; issued > 0 && spin < kDrainSpins; ++spin) __nanosleep(64);
    return;
  }
  const int back = issued < (uint32_t)n_stages ? (int)issued : n_stages;
  uint32_t spin = 0;       // (a stage that the other CTA of a pair has not loaded never completes)
  for (int q = 0; q < back; ++q) {
    int st = stage - 1 - q;
    uint32_t ph = phase;
    if (st < 0) { st += n_stages; ph ^= 1u; }
    for (; spin < kDrainSpins && !mbar_try_wait<PAIR ? WAIT_PAIR : WAIT_CTA>(&full[st], ph); ++spin) __nanosleep(64);
  }
}

// What the warp that issues the MMAs carries from stage to stage (the same in all lanes).
struct MmaCursor {
  int stage;
  uint32_t phase;
};
struct MmaSeg {
  uint32_t dcol[kMaxA], d_part, same, accumulate, idesc, idesc2, b2, b_lbo;
  int k;
};

// The stages of one segment: KS K steps each (less in the last one), NA operands, NM MMAs per operand and step.  The loop is
// instantiated for the counts and all lanes run it on uniform values: the warp issues in program order, and what it does
// beside the MMAs of a stage (300 to 800 cycles of tensor work) has to fit in the same time.
template <bool PAIR, int NA, int NM, bool MN_MAJOR_A, int KS>
__device__ __forceinline__ bool mma_segment(const EngineArgs& a, EngineShared& sh, MmaCursor& cur, const MmaSeg& S, uint32_t ring,
                                            bool leader) {
  constexpr int kStageK = 16 * KS;
  const uint32_t dhi = desc_hi();
  const uint32_t a_lbo = MN_MAJOR_A ? S.b_lbo : 16u;
  uint32_t accumulate = S.accumulate;
  for (int k_left = S.k; k_left > 0; k_left -= kStageK) {
    if (!mbar_wait_warp<PAIR ? WAIT_PAIR : WAIT_CTA>(&sh.full[cur.stage], cur.phase, &sh.abort, a.status, ST_WAIT_FULL,
                                                     a.wait_spin_limit)) return false;
    tc_fence_after();
    // per K step of 16, in 16-byte units: K along x walks 32 B inside a box and 16 KB to the next box; K along y walks 16
    // rows of 128 B
    const uint32_t slot = ring + (uint32_t)(cur.stage * a.stage_bytes);
    const uint32_t alo = desc_lo(slot, a_lbo);
    const uint32_t blo = desc_lo(slot + (uint32_t)a.a_bytes, S.b_lbo);
    if (leader) {
#pragma unroll
      for (int q = 0; q < KS; ++q) {
        if (16 * q < k_left) {
          const uint32_t astep = MN_MAJOR_A ? (uint32_t)(q * 128) : (uint32_t)((q >> 2) * (kBoxBytes >> 4) + (q & 3) * 2);
          const uint64_t bd = desc_join(blo + (uint32_t)(q * 128), dhi);
#pragma unroll
          for (int p = 0; p < NA; ++p) {
            const uint64_t ad = desc_join(alo + (uint32_t)(p * (256 * kStageK >> 4)) + astep, dhi);
            const uint32_t acc_p = q > 0 ? 1u : ((p > 0 && S.same) ? 1u : accumulate);
            mma_bf16<PAIR>(S.dcol[p], ad, bd, S.idesc, acc_p);
            if (NM == 2) mma_bf16<PAIR>(S.dcol[p] + S.d_part, ad, desc_join(blo + S.b2 + (uint32_t)(q * 128), dhi), S.idesc2, acc_p);
          }
        }
      }
      mma_commit<PAIR>(&sh.empty[cur.stage]);
    }
    __syncwarp();
    accumulate = 1u;
    if (++cur.stage == a.n_stages) { cur.stage = 0; cur.phase ^= 1u; }
  }
  return true;
}

// The form of a segment: the operand counts that the items of a launch have (one panel per CTA where two MMAs are needed; A of
// a Gram item always has K along y).
template <bool PAIR, int KS>
__device__ __forceinline__ bool mma_segment_any(const EngineArgs& a, EngineShared& sh, MmaCursor& cur, const MmaSeg& S, int n_a,
                                                bool two, bool mn_major, uint32_t ring, bool leader) {
#define ADAPM_MMA(NA, NM, MN) return mma_segment<PAIR, NA, NM, MN, KS>(a, sh, cur, S, ring, leader)
  if (!PAIR) {
    if (two) ADAPM_MMA(2, 2, true);          // (above rank 128 always both parts of A)
    if (n_a == 2) ADAPM_MMA(2, 1, true);
    ADAPM_MMA(1, 1, true);
  }
  if (two) { if (mn_major) ADAPM_MMA(1, 2, true); ADAPM_MMA(1, 2, false); }
  if (mn_major) {
    if (n_a == 2) ADAPM_MMA(2, 1, true);
    if (n_a == 3) ADAPM_MMA(3, 1, true);
    ADAPM_MMA(1, 1, true);
  }
  if (n_a == 2) ADAPM_MMA(2, 1, false);
  if (n_a == 3) ADAPM_MMA(3, 1, false);
  ADAPM_MMA(1, 1, false);
#undef ADAPM_MMA
}

template <bool PAIR>
__global__ void __launch_bounds__(kEngineThreads, 1) tc_items_kernel(EngineArgs a) {
  extern __shared__ uint8_t dyn_smem[];
  __shared__ EngineShared sh;
  wait_for_previous_kernel();
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn_smem) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &sh.abort;
  const uint32_t wlim = a.wait_spin_limit;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 8; ++i) {
      mbar_init(&sh.full[i], 2);                              // A and B (of a pair: those of rank 0, for both CTAs)
      mbar_init(&sh.empty[i], PAIR && a.sumsq_on && rank == 0 ? 5 : 1);
      mbar_init(&sh.summed[i], 4);
    }
    for (int i = 0; i < 2; ++i) { mbar_init(&sh.tfull[i], 1); mbar_init(&sh.tempty[i], PAIR ? 16 : 8); }
    sh.abort = 0;
    sh.skip = *reinterpret_cast<volatile int32_t*>(a.status) != 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc<PAIR>(&sh.tmem_base, 512);
    tmem_relinquish<PAIR>();
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;
  // an earlier launch gave up: write nothing (the CTAs that work together decide together)
  const bool skip = (PAIR ? load_shared_of(&sh.skip, 0) : sh.skip) != 0;
  const int it_begin = uniform(skip ? 0 : a.cta_begin[unit]), it_end = uniform(skip ? 0 : a.cta_begin[unit + 1]);
  const int stage_k = a.stage_k;
  const int a_tile = 256 * stage_k;                 // bytes of one A operand of a stage
  constexpr Wait kWait = PAIR ? WAIT_PAIR : WAIT_CTA, kTensorWait = PAIR ? WAIT_PAIR_TC : WAIT_CTA;
  // what a producer waits for: in rank 1 the row sums come after the MMAs, in rank 0 they arrive at the same barrier
  uint64_t* const free_bar = PAIR && rank != 0 && a.sumsq_on ? sh.summed : sh.empty;
  const uint32_t pair_full = PAIR ? uniform(shared_of(sh.full, 0)) : 0u;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (all lanes run, one issues)
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued = 0;
    bool ok = true;
    for (int it = it_begin; it < it_end && ok; ++it) {
      const Item& I = a.items[it];
      const int wait_count = uniform(I.wait_count), signal = uniform((int)I.signal), n_seg = uniform(I.n_seg);
      int32_t* const team = a.team_counters + uniform((int)I.team);
      if (wait_count > 0) {
        // Bounded like every wait here: a team member that never arrives ends this CTA with a status, not a
        // hang.  The bound is generous (about a second), because a member may start late when other work
        // holds SMs; the consumers' own bounds are longer still, so this is the wait that reports.
        volatile int32_t* cnt = team;
        uint32_t spin = 0;
        while (__any_sync(0xffffffffu, *cnt < wait_count)) {
          if (++spin >= (rank == 0 ? a.team_spin_limit[0] : a.team_spin_limit[1])) {
            give_up<PAIR>(abort);
            if (leader) atomicOr(a.status, ST_WAIT_TEAM);
            ok = false;
            break;
          }
          if ((spin & 255u) == 0 && __any_sync(0xffffffffu, *abort != 0)) { ok = false; break; }
          __nanosleep(256);
        }
        if (!ok) break;
      }
      for (int s = 0; s < n_seg && ok; ++s) {
        const Seg& S = I.seg[s];
        const CUtensorMap* ma = a.maps + uniform(S.map_a);
        const int nst = (uniform(S.k) + stage_k - 1) / stage_k, a_mode = uniform((int)S.a_mode), n_a = uniform((int)S.n_a);
        const uint32_t tx_bytes = (uint32_t)(n_a * a_tile);
        const int after = (int)rank * 128 * n_a;      // rank 1's operands follow on those of rank 0
        int x[kMaxA], y[kMaxA];
#pragma unroll
        for (int p = 0; p < kMaxA; ++p) { x[p] = uniform(S.ax[p]) + (a_mode ? after : 0); y[p] = uniform(S.ay[p]) + (a_mode ? 0 : after); }
        const int dx = a_mode ? 0 : stage_k, dy = a_mode ? stage_k : 0;
        // K along x: stage_k / 64 boxes of 64 x 128, 16 KB apart; K along y: two boxes of 64 x stage_k
        const int n_box = a_mode ? 2 : (stage_k >> 6);
        const int box_bytes = a_mode ? stage_k * 128 : kBoxBytes;
        for (int c = 0; c < nst; ++c) {
          if (!mbar_wait_warp<kWait>(&free_bar[stage], phase ^ 1u, abort, a.status, ST_WAIT_EMPTY, wlim)) { ok = false; break; }
          uint8_t* sa = stages + stage * a.stage_bytes;
          uint64_t* bar = &sh.full[stage];
          if (leader) {
            if (!PAIR || rank == 0) mbar_arrive_expect_tx(bar, PAIR ? 2 * tx_bytes : tx_bytes);
            const uint32_t pair_bar = pair_full + 8u * (uint32_t)stage;
#define ADAPM_LOAD(NA, NBOX) load_operands<PAIR, NA, NBOX>(sa, a_tile, box_bytes, ma, x, y, bar, pair_bar)
            if (!PAIR) {
              if (n_a == 2) ADAPM_LOAD(2, 2); else ADAPM_LOAD(1, 2);
            } else if (n_box == 2) {
              if (n_a == 2) ADAPM_LOAD(2, 2); else if (n_a == 3) ADAPM_LOAD(3, 2); else ADAPM_LOAD(1, 2);
            } else {
              if (n_a == 2) ADAPM_LOAD(2, 1); else if (n_a == 3) ADAPM_LOAD(3, 1); else ADAPM_LOAD(1, 1);
            }
#undef ADAPM_LOAD
          }
          __syncwarp();
#pragma unroll
          for (int p = 0; p < kMaxA; ++p) { x[p] += dx; y[p] += dy; }
          ++issued;
          if (++stage == a.n_stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (ok && signal && leader && rank == 0) atomicAdd(team, signal);
    }
    if (!ok) drain_ring<PAIR>(sh.full, stage, phase, issued, a.n_stages, rank);
  } else if (warp == 3) {
    // ------------------------------------------------------------------ producer of B (a warp of its own: an expected
    // count and a box take 100 cycles each to issue, and a stage of 64 K is multiplied in 300 to 800)
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued = 0;
    bool ok = true;
    const int b_box = stage_k * 128;
    for (int it = it_begin; it < it_end && ok; ++it) {
      const Item& I = a.items[it];
      const int n_seg = uniform(I.n_seg);
      for (int s = 0; s < n_seg && ok; ++s) {
        const Seg& S = I.seg[s];
        const CUtensorMap* mb = a.maps + uniform(S.map_b);
        const int nst = (uniform(S.k) + stage_k - 1) / stage_k, n_b = uniform((int)S.n_b), xb = rank ? uniform((int)S.b_x) : 0;
        const uint32_t tx_bytes = uniform(S.tx_bytes) - (uint32_t)(uniform((int)S.n_a) * a_tile);
        for (int c = 0; c < nst; ++c) {
          if (!mbar_wait_warp<kWait>(&free_bar[stage], phase ^ 1u, abort, a.status, ST_WAIT_EMPTY, wlim)) { ok = false; break; }
          uint8_t* sb = stages + stage * a.stage_bytes + a.a_bytes;
          uint64_t* bar = &sh.full[stage];
          if (leader) {
            if (!PAIR || rank == 0) mbar_arrive_expect_tx(bar, PAIR ? 2 * tx_bytes : tx_bytes);
            if (PAIR) {
              const uint32_t pair_bar = pair_full + 8u * (uint32_t)stage;
              tma_load_box_pair(sb, mb, xb, c * stage_k, pair_bar);
              if (n_b > 1) tma_load_box_pair(sb + b_box, mb, xb + 64, c * stage_k, pair_bar);
              if (n_b > 2) tma_load_box_pair(sb + 2 * b_box, mb, xb + 128, c * stage_k, pair_bar);
              if (n_b > 3) tma_load_box_pair(sb + 3 * b_box, mb, xb + 192, c * stage_k, pair_bar);
            } else {
              tma_load_box3(sb, mb, 0, c * stage_k, 0, bar);
            }
          }
          __syncwarp();
          ++issued;
          if (++stage == a.n_stages) { stage = 0; phase ^= 1u; }
        }
      }
    }
    if (!ok) drain_ring<PAIR>(sh.full, stage, phase, issued, a.n_stages, rank);
  } else if (warp == 1 && rank == 0) {
    // ------------------------------------------------------------------ MMA issuer (all lanes run, one issues)
    const bool leader = elect_one();
    MmaCursor cur = {0, 0u};
    bool ok = true;
    int j = 0;
    const uint32_t ring = uniform(smem_u32(stages)), d0 = uniform(tmem_base);
    for (int it = it_begin; it < it_end && ok; ++it, ++j) {
      const Item& I = a.items[it];
      const int acc = j % a.n_acc;
      const uint32_t acc_phase = (uint32_t)(j / a.n_acc) & 1u;
      if (!mbar_wait_warp<kTensorWait>(&sh.tempty[acc], acc_phase ^ 1u, abort, a.status, ST_WAIT_TMEM_EMPTY, wlim)) break;
      tc_fence_after();
      const uint32_t d_base = d0 + (uint32_t)(acc * a.acc_cols);
      const int n_seg = uniform(I.n_seg);
      for (int s = 0; s < n_seg && ok; ++s) {
        const Seg& G = I.seg[s];
        const int n_a = uniform((int)G.n_a), n2 = uniform((int)G.n2), a_mode = uniform((int)G.a_mode);
        MmaSeg S;
        S.k = uniform(G.k);
        S.idesc = uniform(make_idesc(G.n, a_mode != 0, true, false, PAIR ? 256 : 128));
        S.idesc2 = make_idesc(n2, a_mode != 0, true, false, PAIR ? 256 : 128);
        S.b_lbo = (uint32_t)stage_k * 128u;               // bytes between the 64-column chunks of B
        S.b2 = (uniform((uint32_t)G.b2_chunk) * S.b_lbo) >> 4;
        S.accumulate = uniform((uint32_t)G.first) ? 0u : 1u;
        S.d_part = uniform((uint32_t)G.d_part); S.same = uniform((uint32_t)G.same_acc);
#pragma unroll
        for (int p = 0; p < kMaxA; ++p) S.dcol[p] = d_base + uniform((uint32_t)G.d_col[p]);
        ok = stage_k == 64 ? mma_segment_any<PAIR, 4>(a, sh, cur, S, n_a, n2 != 0, a_mode != 0, ring, leader)
                           : mma_segment_any<PAIR, 8>(a, sh, cur, S, n_a, n2 != 0, a_mode != 0, ring, leader);
      }
      if (ok && leader) mma_commit<PAIR>(&sh.tfull[acc]);
      __syncwarp();
    }
  } else if (warp < 4) {
    // no work
  } else if (warp < 8) {
    // ------------------------------------------------------------------ row sums of g^2
    // The four warps follow every stage of the launch (their arrivals are part of each stage's release); for an
    // item with sumsq_off >= 0 they read the gradient tiles of the first segment (K along x), each warp 32 rows
    // of every panel.  Eight lanes share a row of a box (its eight 16-byte pieces,
    // whatever order the swizzle put them in), so a warp reads four rows per access without bank conflicts; a
    // lane keeps one partial sum per row it visits, and the eight partial sums of a row are added in a fixed
    // order at the end of the item.
    if (PAIR && a.sumsq_on) {
      uint64_t* const ready = rank == 0 ? sh.full : sh.empty;      // (empty: filled, and multiplied as well)
      uint64_t* const done = rank == 0 ? sh.empty : sh.summed;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      const int rsub = 32 * (warp - 4) + (lane >> 3), piece = lane & 7;
      for (int it = it_begin; it < it_end && ok; ++it) {
        const Item& I = a.items[it];
        const bool mine = I.sumsq_off >= 0;
        float acc[kMaxA][8];
#pragma unroll
        for (int p = 0; p < kMaxA; ++p)
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[p][i] = 0.f;
        int n_a0 = 0;
        for (int s = 0; s < I.n_seg && ok; ++s) {
          const int k = I.seg[s].k, n_a = I.seg[s].n_a;
          if (s == 0) n_a0 = n_a;
          const int nst = (k + stage_k - 1) / stage_k;
          const int n_box = stage_k >> 6;
          for (int c = 0; c < nst; ++c) {
            bool got = true;
            if (lane == 0) got = mbar_wait<WAIT_PAIR>(&ready[stage], phase, abort, a.status, ST_WAIT_FULL, wlim);
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) { ok = false; break; }
            if (mine && s == 0) {
              const uint8_t* sa = stages + stage * a.stage_bytes;
#pragma unroll
              for (int p = 0; p < kMaxA; ++p) {
                if (p < n_a) {
                  for (int jb = 0; jb < n_box; ++jb) {
                    const uint8_t* box = sa + p * a_tile + jb * kBoxBytes + piece * 16;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                      const uint4 v = *reinterpret_cast<const uint4*>(box + (4 * i + rsub) * 128);
                      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                      float s2 = acc[p][i];
#pragma unroll
                      for (int e = 0; e < 4; ++e) {
                        const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
                        s2 = fmaf(lo, lo, s2);
                        s2 = fmaf(hi, hi, s2);
                      }
                      acc[p][i] = s2;
                    }
                  }
                }
              }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&done[stage]);
            if (++stage == a.n_stages) { stage = 0; phase ^= 1u; }
          }
        }
        if (mine && ok) {
          const int after = (int)rank * 128 * n_a0;
          float* out = a.work_f32 + I.sumsq_off + after;
#pragma unroll
          for (int p = 0; p < kMaxA; ++p) {
            if (p < n_a0) {
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                float s2 = acc[p][i];
                s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
                s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
                s2 += __shfl_xor_sync(0xffffffffu, s2, 4);
                const int row = 128 * p + 4 * i + rsub;
                if (piece == 0 && I.own0 + after + row < I.own_count) out[row] = s2;
              }
            }
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    const int q = 32 * (warp & 3) + lane;               // accumulator row (= TMEM lane) of this thread
    const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
    const int grp = (warp - 8) >> 2;                    // the two groups take the pieces of an item alternately
    const float gs = a.gscale ? *a.gscale : 1.f;
    int j = 0;
    for (int it = it_begin; it < it_end; ++it, ++j) {
      // scalar fields are copied once: the stores below could alias the item table as far as the
      // compiler can tell, and every re-read would be a round trip to global memory
      ItemEpi I;
      {
        const Item& G = a.items[it];
        I.epi = G.epi; I.own0 = G.own0; I.own_count = G.own_count; I.n_pan = G.n_pan; I.acc_stride = G.acc_stride;
        I.r = G.r; I.rp = G.rp; I.half = G.half; I.n_sum = G.n_sum; I.stack_rows = G.stack_rows;
        I.from_iter = G.from_iter; I.to_iter = G.to_iter; I.iter_off = G.iter_off;
        I.f32_off = G.f32_off; I.own_stride = G.own_stride; I.k_stride = G.k_stride;
        I.dst_off = G.dst_off; I.dst_ld = G.dst_ld; I.coef = G.coef;
        if (PAIR) {                                     // rank 1's panels follow on those of rank 0; some may not exist
          I.own0 += (int)rank * 128 * I.n_pan;
          I.n_pan = max(0, min(I.n_pan, (I.own_count - I.own0 + 127) >> 7));
        }
      }
      const int acc = j % a.n_acc;
      const uint32_t acc_phase = (uint32_t)(j / a.n_acc) & 1u;
      const int rp = I.rp, r = I.r, half = I.half;
      const int np = rp >> 4;                             // 16-column pieces per panel
      const int total = PAIR && I.epi == EPI_FACTOR ? I.n_pan * np : 0;
      // Gradients scaled by gs (global norm clipping): the factor update is linear in g, so the Gram operands
      // are divided by gs where they are made and the whole accumulator is multiplied by it here.
      const float coef = PAIR ? I.coef * gs : I.coef / gs;
      const bool factor = PAIR && grp < total;
      const bool has_work = PAIR ? factor : (I.epi == EPI_GRAM && grp == 0);
      const int qc = lane & 3;
      float* const fbase = a.f32_base + I.f32_off;
      float* const ibase = a.work_f32 + I.iter_off;
      // EPI_FACTOR works in one of two arrangements.  Straight: a thread keeps its accumulator row.  Old and new values
      // are 32-byte accesses per lane in the workspace's order, where a warp's 32 rows are one run of memory, and for a
      // row-stored factor of the state (L, [m, r]) whose rows start on 32 bytes and hold a multiple of eight values; a
      // factor whose consecutive owners are adjacent (R, [r, n]) goes column by column, 32 rows = one 128-byte run.
      // Turned, for any other L: every quad of lanes transposes its 4 x 16 piece with shuffles, after which lane c of
      // the quad holds columns 4c .. 4c+3 of the quad's four rows, so that rows are 64-byte runs instead of one per lane.
      // Only the first pass of a step reads the state and only the last one writes it.  A piece of 16 columns took 1.6
      // thousand cycles by rows and 3.5 thousand by columns, whether or not memory was busy: a warp's 32-byte accesses touch 32
      // cache lines by rows and 8 in the workspace's order, and columns take 16 narrow accesses.  Panel launches of a step,
      // state in every pass -> workspace in between: 2.01 -> 1.79 ms on the 350M set at rank 128, 418 -> 376 us on
      // 1024 x 2730, 137 -> 127 us on the 60M set, 16.3 -> 15.7 ms on 8 layers of the 8B shapes.
      const bool by_column = I.own_stride == 1;
      const bool by_row = I.k_stride == 1 && ((I.own_stride | r | I.f32_off) & 7) == 0;
      const bool turned = factor && !by_column && !by_row && !(I.from_iter && I.to_iter);
      // workspace order: [panel][piece][8 columns][128 rows][8]
      auto iter_at = [&](int u, int h, int row) { return ibase + (((int64_t)u * 2 + h) * 128 + row) * 8; };
      const int own_u0 = I.own0 >> 7;                     // panels before this item's (its pieces start at own_u0 * np)
      auto fetch = [&](int u, float* o) {
        const int pan = u / np, p = 16 * (u - pan * np);
        const int own_row = I.own0 + 128 * pan + q;
        if (I.from_iter) {
          ldcg_f32x8(iter_at(own_u0 * np + u, 0, q), o);
          if (p + 8 < r) {
            ldcg_f32x8(iter_at(own_u0 * np + u, 1, q), o + 8);
          } else {                       // (no traffic for padding)
#pragma unroll
            for (int e = 8; e < 16; ++e) o[e] = 0.f;
          }
          return;
        }
        const bool row_ok = own_row < I.own_count;
        if (by_row) {
          const float* fp = fbase + I.own_stride * own_row + p;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (row_ok && p + 8 * h < r) {
              ldcg_f32x8(fp + 8 * h, o + 8 * h);
            } else {
#pragma unroll
              for (int e = 0; e < 8; ++e) o[8 * h + e] = 0.f;
            }
          }
        } else {
          const float* fp = fbase + own_row + I.k_stride * p;
          const int n = row_ok ? r - p : 0;
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            o[e] = e < n ? __ldcg(fp) : 0.f;
            fp += I.k_stride;
          }
        }
      };
      // the turned arrangement: o[4 i + e] = column p + 4 qc + e of quad row i
      auto fetch_turned = [&](int u, float* o) {
        const int pan = u / np, p = 16 * (u - pan * np);
        const int row_quad = 32 * (warp & 3) + (lane & ~3), own_quad = I.own0 + 128 * pan + row_quad;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int owner = own_quad + i, k = p + 4 * qc;
          if (I.from_iter) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(iter_at(own_u0 * np + u, qc >> 1, row_quad + i) + 4 * (qc & 1)));
            o[4 * i] = v.x; o[4 * i + 1] = v.y; o[4 * i + 2] = v.z; o[4 * i + 3] = v.w;
          } else {
            const float* fp = fbase + I.own_stride * owner + k;
            const int n = owner < I.own_count ? r - k : 0;
#pragma unroll
            for (int e = 0; e < 4; ++e) o[4 * i + e] = e < n ? __ldcg(fp + e) : 0.f;
          }
        }
      };
      // old values travel one piece ahead in two register sets that swap roles (no copies, which
      // would wait for the loads); the first set is requested before the accumulator is waited for
      float oldA[16], oldB[16];
      if (PAIR && turned) fetch_turned(grp, oldA);
      else if (PAIR && factor) fetch(grp, oldA);
      // one lane per warp polls (fewer pollers on the barrier), then the warp agrees: the
      // tensor-memory loads below need all 32 lanes
      bool got = true;
      if (lane == 0) got = mbar_wait<kTensorWait>(&sh.tfull[acc], acc_phase, abort, a.status, ST_WAIT_TMEM_FULL, wlim);
      got = __shfl_sync(0xffffffffu, got, 0);
      if (!got) break;
      tc_fence_after();
      const uint32_t t0 = tmem_base + lane_addr + (uint32_t)(acc * a.acc_cols);
      // With one accumulator buffer the next item's MMAs wait for this epilogue.  Its memory traffic is the slow
      // part, so the sums D0 + D1 are first parked in spare tensor-memory columns (this warp's own lanes, the
      // same columns for every item) and the accumulator is handed back at once; the pieces below then read the
      // parked sums while the next main loop runs.  Each group parks the pieces it will work on.
      const bool parked = factor && a.sum_col >= 0;
      const uint32_t ts = parked ? tmem_base + lane_addr + (uint32_t)a.sum_col : t0;
      const uint32_t ts_stride = (uint32_t)(parked ? rp : I.acc_stride);
      // Where column p of a panel and its lo part are: the first MMA of a K step makes [hi | lo] of columns below 128, the
      // second one (ranks above 128) the same of the others, from column 256.
      auto hi_col = [&](int p) { return p < 128 ? p : p + 128; };
      auto lo_col = [&](int p) { return p < 128 ? p + min(rp, 128) : p + rp; };
      if (parked) {
#pragma unroll 1
        for (int u = grp; u < total; u += 2) {
          const int pan = u / np, p = 16 * (u - pan * np);
          float d0[16], d1[16];
          tmem_ld16(t0 + (uint32_t)(pan * I.acc_stride + hi_col(p)), d0);
          tmem_ld16(t0 + (uint32_t)(pan * I.acc_stride + lo_col(p)), d1);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 16; ++e) d0[e] += d1[e];
          tmem_st16(ts + (uint32_t)pan * ts_stride + (uint32_t)p, d0);
        }
        tmem_st_wait();
      }
      // D0 + D1 of columns [p, p + 16) of this thread's row of a panel
      auto sum16 = [&](int pan, int p, float* x) {
        tmem_ld16(ts + (uint32_t)pan * ts_stride + (uint32_t)(parked ? p : hi_col(p)), x);
        if (!parked) {
          float d1[16];
          tmem_ld16(ts + (uint32_t)pan * ts_stride + (uint32_t)lo_col(p), d1);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 16; ++e) x[e] += d1[e];
        } else {
          tmem_ld_wait();
        }
      };
      // the accumulator goes back to the warp that issues the MMAs: one arrival per warp, at rank 0
      auto hand_back = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR) mbar_arrive_relaxed_at(shared_of(&sh.tempty[acc], 0));
          else mbar_arrive(&sh.tempty[acc]);
        }
      };
      const bool early = parked || !has_work;   // (a warp without work never reads the accumulator)
      if (early) hand_back();
      if (PAIR && factor) {
        uint16_t* const dst = a.work_bf16 + I.dst_off;
        auto piece = [&](int u, const float* o) {
          const int pan = u / np, p = 16 * (u - pan * np);
          const int own_row = I.own0 + 128 * pan + q;
          float x[16];
          sum16(pan, p, x);
          const bool row_ok = own_row < I.own_count;
          uint32_t hi[8], lo[8];
#pragma unroll
          for (int e = 0; e < 16; e += 2) {
            x[e] = p + e < r ? o[e] + coef * x[e] : 0.f;
            x[e + 1] = p + e + 1 < r ? o[e + 1] + coef * x[e + 1] : 0.f;
            split_bf16x2(x[e], x[e + 1], hi[e >> 1], lo[e >> 1]);
          }
          if (I.to_iter) {
            st_f32x8(iter_at(own_u0 * np + u, 0, q), x);
            if (p + 8 < r) st_f32x8(iter_at(own_u0 * np + u, 1, q), x + 8);
          } else if (by_row) {
            float* fp = fbase + I.own_stride * own_row + p;
            if (row_ok && p < r) st_f32x8(fp, x);
            if (row_ok && p + 8 < r) st_f32x8(fp + 8, x + 8);
          } else {
            float* fp = fbase + own_row + I.k_stride * p;
            const int n = row_ok ? r - p : 0;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              if (e < n) __stcg(fp, x[e]);
              fp += I.k_stride;
            }
          }
          if (row_ok) {
            uint16_t* drow = dst + (int64_t)I.dst_ld * own_row + p;
            st_b32x8(drow, hi);
            st_b32x8(drow + half, lo);
          }
        };
        // one piece in the turned arrangement
        auto piece_turned = [&](int u, const float* o) {
          const int pan = u / np, p = 16 * (u - pan * np);
          const int row_quad = 32 * (warp & 3) + (lane & ~3), own_quad = I.own0 + 128 * pan + row_quad;
          float v[16];                   // columns of this thread's row
          sum16(pan, p, v);
          // quad transpose, first exchange (partner lane ^ 2): keep the half of the columns this lane's
          // final column group lies in, hand over the other half
          const bool up = (qc & 2) != 0, odd = (qc & 1) != 0;
          float k0[4], k1[4], g0[4], g1[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            k0[e] = up ? v[8 + e] : v[e];
            k1[e] = up ? v[12 + e] : v[4 + e];
            const float s0 = up ? v[e] : v[8 + e], s1 = up ? v[4 + e] : v[12 + e];
            g0[e] = __shfl_xor_sync(0xffffffffu, s0, 2);
            g1[e] = __shfl_xor_sync(0xffffffffu, s1, 2);
          }
          // second exchange (partner lane ^ 1): keep this lane's column group of the two rows held so far,
          // hand over the neighbour's; t[0..3] then belong to quad rows qc, qc^2, qc^1, qc^3
          float t[4][4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            t[0][e] = odd ? k1[e] : k0[e];
            t[1][e] = odd ? g1[e] : g0[e];
            const float s0 = odd ? k0[e] : k1[e], s1 = odd ? g0[e] : g1[e];
            t[2][e] = __shfl_xor_sync(0xffffffffu, s0, 1);
            t[3][e] = __shfl_xor_sync(0xffffffffu, s1, 1);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            // order by row, so that in every access below the four lanes of a quad address one row:
            // row i is t[0], t[1], t[2] or t[3] as i ^ qc is 0, 2, 1 or 3
            const int w = i ^ qc, owner = own_quad + i, k = p + 4 * qc;
            float x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float sd = w == 0 ? t[0][e] : (w == 2 ? t[1][e] : (w == 1 ? t[2][e] : t[3][e]));
              x[e] = k + e < r ? o[4 * i + e] + coef * sd : 0.f;
            }
            if (owner >= I.own_count) continue;
            if (I.to_iter) {
              __stcg(reinterpret_cast<float4*>(iter_at(own_u0 * np + u, qc >> 1, row_quad + i) + 4 * (qc & 1)),
                     make_float4(x[0], x[1], x[2], x[3]));
            } else {
              float* fp = fbase + I.own_stride * owner + k;
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (k + e < r) fp[e] = x[e];
            }
            uint32_t h01, l01, h23, l23;
            split_bf16x2(x[0], x[1], h01, l01);
            split_bf16x2(x[2], x[3], h23, l23);
            uint16_t* drow = dst + (int64_t)I.dst_ld * owner + k;
            *reinterpret_cast<uint2*>(drow) = make_uint2(h01, h23);
            *reinterpret_cast<uint2*>(drow + half) = make_uint2(l01, l23);
          }
        };
        // this group's pieces grp, grp + 2, ...: two per trip, the old values of the next one on their way
        if (!turned) {
#pragma unroll 1
          for (int u = grp; u < total; u += 4) {
            if (u + 2 < total) fetch(u + 2, oldB);
            piece(u, oldA);
            if (u + 2 < total) {
              if (u + 4 < total) fetch(u + 4, oldA);
              piece(u + 2, oldB);
            }
          }
        } else {
#pragma unroll 1
          for (int u = grp; u < total; u += 4) {
            if (u + 2 < total) fetch_turned(u + 2, oldB);
            piece_turned(u, oldA);
            if (u + 2 < total) {
              if (u + 4 < total) fetch_turned(u + 4, oldA);
              piece_turned(u + 2, oldB);
            }
          }
        }
      } else if (!PAIR && has_work) {  // EPI_GRAM
        uint16_t* dst = a.work_bf16 + I.dst_off;
        const int row = I.own0 + q;
#pragma unroll 1
        for (int p = 0; p < rp; p += 16) {
          float d0[16], d1[16];
          tmem_ld16(t0 + (uint32_t)p, d0);
          tmem_ld_wait();
#pragma unroll 1
          for (int part = 1; part < I.n_sum; ++part) {
            tmem_ld16(t0 + (uint32_t)(part * rp + p), d1);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 16; ++e) d0[e] += d1[e];
          }
          if (row < rp) {
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) split_bf16x2(coef * d0[e], coef * d0[e + 1], hi[e >> 1], lo[e >> 1]);
            for (int copy = 0; copy < (I.stack_rows > 0 ? 2 : 1); ++copy) {
              uint16_t* drow = dst + (int64_t)I.dst_ld * (row + copy * I.stack_rows) + p;
              uint4* dh = reinterpret_cast<uint4*>(drow);
              uint4* dl = reinterpret_cast<uint4*>(drow + half);
              dh[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
              dh[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
              dl[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
              dl[1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
            }
          }
        }
      }
      if (!early) hand_back();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();      // neither CTA leaves while the other may still reach into it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<PAIR>(tmem_base, 512);
  }
}

}  // namespace tc
}  // namespace adapm

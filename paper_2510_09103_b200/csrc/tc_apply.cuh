// Tensor-core "apply" kernel of the low-rank path: rebuilds the corrected momentum tile by tile and
// writes the parameters (Algorithm 1 lines 4, 6, 8 and 9 combined):
//
//   m^c = cg g + c0 L0 R0 - c1 L R          (= g + c (P_{t-1} - P_t) with the correction on)
//   W  <- W - lr s_b ( clamp( m^c / (sqrt(v) + eps) ) + lambda_b W )
//
// An item is a 128-row panel of one block times a run of column tiles.  Up to rank 128 the split-bf16 rows
// [L0 hi | L0 lo | L hi | L lo] of the panel are the A operand and stay in tensor memory for the whole run
// (two bf16 per column, the refitted set with its sign turned: 2 rp + two accumulators of 128 <= 512
// columns); per column tile the matching rows of [R0^T hi | R0^T lo | R^T hi | R^T lo] arrive one 64-column
// box at a time through a ring of 16 KB stages, and every 16 columns of a box are multiplied at once with
// the L columns they pair with (hi*hi and lo*hi for columns of a hi part, hi*lo for columns of a lo part),
// so the accumulator ends up holding D = L0 R0 - L R.  Four warps load the L panel of the next item when
// the last MMA of the present one is through.  With L in shared memory instead (4 rp columns x 128 rows: 80
// KB at rank 80, 128 KB at rank 128) the operand reads of A share the shared memory's bandwidth and the ring
// below has room for two or three buffers: 2.42 -> 1.36 ms at rank 128, 8.3 -> 6.6 ms on the 1.5B shapes with
// a per-element v; with a group v, where the ring had four buffers, as fast as before.
//
// Ranks above 128 leave no room for L in tensor memory.  The kernel's second form (kStream) streams L as
// well: a stage of its ring holds four boxes - 64 columns of L hi, L lo, R^T hi and R^T lo of one factor
// set - and feeds hi*hi, lo*hi and hi*lo for those columns; the previous set is always taken first, the
// refitted set second.  (Tiles of 96 columns would fit L up to rank 208 beside one accumulator; measured,
// that was slower, 8.3 against 6.3 ms on eight layers of the 8B shapes.)
//
// kTma (parameter rows start on 16 bytes: cols a multiple of 8): g and W never pass through registers on
// their way in or out.  A mover thread brings them in quarters (128 rows x 32 columns: 16 KB of W, 8 KB of
// g) by TMA into a ring of shared-memory buffers, several quarters ahead of their use, and writes the
// updated W back from the same buffer by TMA.  The groups of 128 epilogue threads take the quarters in
// turn; a thread owns one row of the panel: it reads its accumulator row from tensor memory, its columns of g
// and W from the (swizzled) buffer, and puts the new W back in place.  A per-element v, where a block has
// one, travels like W.
// (Quarters of 32 rows x 128 columns take four times as many boxes: 4.4 ms instead of 3.0 on the 1.5B shapes.)
// Otherwise an epilogue warp turns a 32 x 32 chunk of the accumulator through a patch of shared memory and
// works along the rows of the parameters, one column per lane, whatever the alignment of the rows.
// Four groups where the arithmetic or the latency of that form sets the pace, two where the ring of buffers does (with four it
// has to be four deep instead of six, or the ring of R half as deep): per-element v 5.30 -> 4.90 ms on the 1.5B shapes and 1.18
// -> 1.05 on the 350M set at rank 128, rows of 2730 184 -> 140 us; group scalars 2.50 -> 2.71 or 3.15 ms, kept at two.  The form
// with TMA is chosen for the set: one low-rank block with a per-element v makes its launch take four groups for all blocks.
// The m x n matrices m_t, r_t and m^c are never stored.
#pragma once

#include <cuda.h>

#include "adapm_internal.h"
#include "device_math.cuh"
#include "tc_common.cuh"

namespace adapm {
namespace tc {

// producer, MMA, epilogue warps in groups of four, mover, four warps that load L
constexpr int apply_threads(int groups) { return 32 * (2 + 4 * groups + 1 + 4); }
constexpr int kApplyNT = 128;              // columns per tile
constexpr int kApplyQC = 32;               // columns per quarter tile
constexpr int kApplyMaxStages = 8;         // R ring depth limit
constexpr int kApplyMaxBufs = 8;           // g / W ring depth limit
constexpr int kWBoxBytes = 128 * kApplyQC * 4;   // a quarter tile of W: 128 rows of 128 bytes
constexpr int kGBoxBytes = 128 * kApplyQC * 2;   // and of g: 128 rows of 64 bytes
constexpr int kApplyBufBytes = kWBoxBytes + kGBoxBytes;    // + kWBoxBytes where a block has a per-element v
constexpr int kPatchPitch = 33;            // floats per row of an epilogue warp's patch
constexpr int kPatchBytes = 32 * kPatchPitch * 4;

struct ApplyItem {
  int64_t off;               // element offset of the block in params / grads
  int64_t v_off;             // float offset of v in state
  int64_t l_off;             // bf16 element offset of the L array in the workspace (row pitch 4 half)
  int32_t rows, cols, r, rp;
  int32_t half;              // column at which the lo part of a factor set starts (a set is 2 half columns wide)
  int32_t map_l, map_r;      // split factors, previous and final set side by side: [rows, 4 half] and [cols, 4 half]
                             // = [hi0 | lo0 | hi1 | lo1], boxes of 64 x 128
  int32_t map_w, map_g;      // params and grads of the block, boxes of 32 x 128
  int32_t map_v;             // per-element v of the block (same boxes as params); unused with a group v
  int32_t map_sh;            // bf16 copy of the params (same boxes as grads); used when the launch has a shadow
  int32_t row0;              // first row of the panel
  int32_t tile0, n_tiles;    // column tiles [tile0, tile0 + n_tiles) of 128 columns
  int32_t v_mode, v_group_rows;
  float lr_scale, wd;
};

struct ApplyArgs {
  const ApplyItem* items;
  int32_t n_items;
  const CUtensorMap* maps;
  const uint16_t* work;      // workspace viewed as bf16
  float* params;             // params, grads and shadow by address (!kTma; kTma goes through the maps)
  const uint16_t* grads;
  uint16_t* shadow_out;
  float* state;
  int32_t* status;
  StepScalars sc;
  int32_t use_new;           // 0: c1 == 0, the refitted factors are not needed
  int32_t parity;            // 0: the left half of the operands holds the previous factors, 1: the right half
  const float* gscale;       // device scalar: every gradient counts as gscale[0] * g (nullptr: 1)
  int32_t shadow;            // 1: the bf16 copy of the parameters is written with W
  int32_t n_rstages;         // R ring depth (1..kApplyMaxStages); a stage is one 64 x 128 box of R^T (kStream: four boxes)
  int32_t w_region_off;      // byte offset of the g / W ring (kTma) or of the patches inside the dynamic shared memory
  int32_t n_bufs;            // g / W ring depth (up to kApplyMaxBufs, a multiple of the groups: see the epilogue)
  int32_t buf_bytes;         // one buffer: W, g and, if any block of the launch has a per-element v, v
};

struct __align__(8) ApplyShared {
  uint64_t lfull, lempty, rfull[kApplyMaxStages], rempty[kApplyMaxStages], tfull[2], tempty[2];
  uint64_t wfull[kApplyMaxBufs];   // a quarter's g and W have landed
  uint64_t wdone[kApplyMaxBufs];   // a group of four epilogue warps has put its new W back
  uint32_t tmem_base;
  int abort;
};

// The epilogue of one warp without TMA: 32 x 32 chunks of the accumulator, one column per lane.  (Rows in flight: a warp has 80
// registers in this form.)
template <int kGroups>
__device__ __forceinline__ void apply_rows_epilogue(const ApplyArgs& a, ApplyShared& sh, float* patch, uint32_t tmem_acc) {
  constexpr int kChunks = kApplyNT / 32, kBatch = 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = warp & 3, grp = (warp - 2) >> 2;           // which 32 accumulator rows; chunks grp, grp + kGroups, ...
  const uint32_t lane_addr = (uint32_t)(32 * sub) << 16;
  const StepScalars& sc = a.sc;
  const float gs = a.gscale ? *a.gscale : 1.f;
  int j = 0;
  for (int it = blockIdx.x; it < a.n_items; it += gridDim.x) {
    const ApplyItem I = a.items[it];
    const bool grouped = I.v_mode == ADAPM_V_BLOCKMEAN;
    const float lr_s = sc.lr * I.lr_scale;
    const int row0 = I.row0 + 32 * sub, rows = I.rows - row0;
    // one denominator per row when v is a group scalar (lane = row of the chunk): m^c / (sqrt(v) + eps) is a product
    float kr = 0.f;
    if (grouped && lane < rows) {
      const float v_row = a.state[I.v_off + (row0 + lane) / I.v_group_rows];
      kr = sc.inv_bc1 / (sqrtf(v_row * sc.inv_bc2) + sc.eps);
    }
    for (int t = 0; t < I.n_tiles; ++t, ++j) {
      const int acc = j & 1;
      for (int c = grp; c < kChunks; c += kGroups) {
        const int col = (I.tile0 + t) * kApplyNT + 32 * c + lane;
        const bool cok = col < I.cols;
        const int64_t o = (int64_t)row0 * I.cols + col;
        float* W = a.params + I.off + o;
        const uint16_t* G = a.grads + I.off + o;
        float* V = a.state + I.v_off + o;
#pragma unroll
        for (int r0 = 0; r0 < 32; r0 += kBatch) {
          float w[kBatch], v[kBatch];
          uint16_t g[kBatch];
#pragma unroll
          for (int r = 0; r < kBatch; ++r) {
            const int64_t at = (int64_t)(r0 + r) * I.cols;
            w[r] = 0.f; v[r] = 0.f; g[r] = 0;
            if (cok && r0 + r < rows) {
              w[r] = W[at];
              g[r] = G[at];
              if (!grouped) v[r] = V[at];
            }
          }
          if (r0 == 0) {
            // one lane polls, then the warp agrees: the tensor-memory loads need all 32 lanes
            bool got = true;
            if (lane == 0) got = mbar_wait(&sh.tfull[acc], (uint32_t)(j >> 1) & 1u, &sh.abort, a.status, ST_WAIT_TMEM_FULL);
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) return;
            tc_fence_after();
#pragma unroll
            for (int x = 0; x < 32; x += 16) {
              float d[16];
              tmem_ld16(tmem_acc + lane_addr + (uint32_t)(acc * kApplyNT + 32 * c + x), d);
              tmem_ld_wait();
#pragma unroll
              for (int e = 0; e < 16; ++e) patch[lane * kPatchPitch + x + e] = d[e];
            }
            __syncwarp();
          }
#pragma unroll
          for (int r = 0; r < kBatch; ++r) {
            const float k_row = __shfl_sync(0xffffffffu, kr, r0 + r);
            if (cok && r0 + r < rows) {
              const int64_t at = (int64_t)(r0 + r) * I.cols;
              const float d = patch[(r0 + r) * kPatchPitch + lane], g1 = gs * bf16_bits_to_float(g[r]);
              const float mc = sc.cg * g1 + sc.c0 * d;
              if (grouped) {
                w[r] = w[r] - lr_s * (clamp_keep_nan(mc * k_row, sc.clip) + I.wd * w[r]);
              } else {
                v[r] = sc.beta2 * v[r] + (1.f - sc.beta2) * (g1 * g1);
                adapm_param_update_n<1>(&w[r], &mc, &v[r], sc, lr_s, I.wd);
                V[at] = v[r];
              }
              W[at] = w[r];
              if (a.shadow) a.shadow_out[I.off + o + at] = (uint16_t)(pack_bf16x2(w[r], 0.f) & 0xffffu);
            }
          }
        }
        __syncwarp();                                        // the patch is free again
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.tempty[acc]);
    }
  }
}

template <bool kStream, bool kTma, int kGroups>
__global__ void __launch_bounds__(apply_threads(kGroups), 1) tc_apply_kernel(ApplyArgs a) {
  constexpr int kStageBytes = kStream ? 4 * kBoxBytes : kBoxBytes;
  constexpr int kQ = kApplyNT / kApplyQC;                    // quarters per tile
  extern __shared__ uint8_t dyn_smem[];
  __shared__ ApplyShared sh;
  __shared__ int skip_launch;
  wait_for_previous_kernel();
  if (threadIdx.x == 0) skip_launch = *reinterpret_cast<volatile int32_t*>(a.status) != 0;
  __syncthreads();
  if (skip_launch) return;   // an earlier launch of the step gave up: leave W and v untouched
  uint8_t* smem_r = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn_smem) + 1023) & ~(uintptr_t)1023);
  uint8_t* smem_w = smem_r + a.w_region_off;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &sh.abort;
  const int n_sets = a.use_new ? 2 : 1;

  if (threadIdx.x == 0) {
    mbar_init(&sh.lfull, 4); mbar_init(&sh.lempty, 1);
    for (int i = 0; i < kApplyMaxStages; ++i) { mbar_init(&sh.rfull[i], 1); mbar_init(&sh.rempty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&sh.tfull[i], 1); mbar_init(&sh.tempty[i], 4 * kGroups); }
    for (int i = 0; i < kApplyMaxBufs; ++i) { mbar_init(&sh.wfull[i], 1); mbar_init(&sh.wdone[i], 4); }
    sh.abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;                   // A from column 0, accumulators at the end
  const uint32_t tmem_acc = tmem_base + 512 - 2 * kApplyNT;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (all lanes run, one issues)
    const bool leader = elect_one();
    uint32_t rphase = 0;
    int rs = 0;
    bool ok = true;
    int r_loads = 0;
    for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
      const ApplyItem& I = a.items[it];
      const CUtensorMap* const ml = a.maps + I.map_l;
      const CUtensorMap* const mr = a.maps + I.map_r;
      const int n_tiles = I.n_tiles, row0 = I.row0, half = I.half, rp = I.rp;
      // the columns of all parts in one run; with only the previous set in use, and that set in the right half, the
      // run starts there
      const int x0 = (n_sets == 1 && a.parity) ? 2 * half : 0;
      const int nb = kStream ? (rp + 63) >> 6 : (n_sets * 2 * rp + 63) >> 6;
      int col0 = I.tile0 * kApplyNT;
      for (int t = 0; t < n_tiles && ok; ++t, col0 += kApplyNT) {
        for (int si = 0; si < (kStream ? n_sets : 1) && ok; ++si) {
          const int xs = (si == 0 ? a.parity : 1 - a.parity) * 2 * half;
          for (int bc = 0; bc < nb; ++bc) {
            if (!mbar_wait_warp(&sh.rempty[rs], rphase ^ 1u, abort, a.status, ST_WAIT_EMPTY)) { ok = false; break; }
            uint8_t* st = smem_r + rs * kStageBytes;
            if (leader) {
              mbar_arrive_expect_tx(&sh.rfull[rs], (uint32_t)kStageBytes);
              if (kStream) {
                tma_load_box(st, ml, xs + 64 * bc, row0, &sh.rfull[rs]);
                tma_load_box(st + kBoxBytes, ml, xs + half + 64 * bc, row0, &sh.rfull[rs]);
                tma_load_box(st + 2 * kBoxBytes, mr, xs + 64 * bc, col0, &sh.rfull[rs]);
                tma_load_box(st + 3 * kBoxBytes, mr, xs + half + 64 * bc, col0, &sh.rfull[rs]);
              } else {
                tma_load_box(st, mr, x0 + 64 * bc, col0, &sh.rfull[rs]);
              }
            }
            __syncwarp();
            ++r_loads;
            if (++rs == a.n_rstages) { rs = 0; rphase ^= 1u; }
          }
        }
      }
    }
    if (!ok) {   // let the copies already issued land before the CTA exits
      const int back = r_loads < a.n_rstages ? r_loads : a.n_rstages;
      for (int q = 0; q < back; ++q) {
        int st = rs - 1 - q;
        uint32_t ph = rphase;
        if (st < 0) { st += a.n_rstages; ph ^= 1u; }
        for (uint32_t spin = 0; spin < kSpinLimit && !mbar_try_wait(&sh.rfull[st], ph); ++spin) __nanosleep(64);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (all lanes run, one issues)
    const bool leader = elect_one();
    uint32_t item_phase = 0, rphase = 0;
    int rs = 0;
    int j = 0;   // running tile count of this CTA
    bool ok = true;
    const uint32_t r_base = uniform(smem_u32(smem_r)), a_base = uniform(tmem_base), acc_base = uniform(tmem_acc);
    const uint32_t dhi = desc_hi();
    const uint32_t idesc_pos = make_idesc(kApplyNT, false, false, false);
    const uint32_t idesc_neg = make_idesc(kApplyNT, false, false, true);
    for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
      const int n_tiles = uniform(a.items[it].n_tiles);
      const int ks = uniform(a.items[it].rp >> 4);     // 16-wide K steps per part (hi or lo of one set)
      if (!kStream && !mbar_wait_warp(&sh.lfull, item_phase, abort, a.status, ST_WAIT_FULL)) break;
      for (int t = 0; t < n_tiles && ok; ++t, ++j) {
        const int acc = j & 1;
        if (!mbar_wait_warp(&sh.tempty[acc], ((uint32_t)(j >> 1) & 1u) ^ 1u, abort, a.status, ST_WAIT_TMEM_EMPTY)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d = acc_base + (uint32_t)(acc * kApplyNT);
        if (kStream) {
          const int nbh = (ks + 3) >> 2;
          for (int si = 0; si < n_sets && ok; ++si) {
            const uint32_t idesc = si ? idesc_neg : idesc_pos;      // the refitted set enters negated
            for (int jb = 0; jb < nbh; ++jb) {
              if (!mbar_wait_warp(&sh.rfull[rs], rphase, abort, a.status, ST_WAIT_FULL)) { ok = false; break; }
              tc_fence_after();
              const uint32_t st = r_base + (uint32_t)(rs * kStageBytes);
              const uint32_t ahi = desc_lo(st, 16), alo = desc_lo(st + kBoxBytes, 16);
              const uint32_t bhi = desc_lo(st + 2 * kBoxBytes, 16), blo = desc_lo(st + 3 * kBoxBytes, 16);
              if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                  if (4 * jb + kk < ks) {
                    const uint32_t o = (uint32_t)(kk * 2);
                    mma_bf16(d, desc_join(ahi + o, dhi), desc_join(bhi + o, dhi), idesc, (si | jb | kk) != 0);
                    mma_bf16(d, desc_join(alo + o, dhi), desc_join(bhi + o, dhi), idesc, 1u);
                    mma_bf16(d, desc_join(ahi + o, dhi), desc_join(blo + o, dhi), idesc, 1u);
                  }
                }
                mma_commit(&sh.rempty[rs]);
              }
              __syncwarp();
              if (++rs == a.n_rstages) { rs = 0; rphase ^= 1u; }
            }
          }
        } else {
          int part = 0, w = 0;         // the box's first K step: part (hi, lo of one set, hi, lo of the other), step inside it
          while (part < 2 * n_sets) {
            if (!mbar_wait_warp(&sh.rfull[rs], rphase, abort, a.status, ST_WAIT_FULL)) { ok = false; break; }
            tc_fence_after();
            const uint32_t rb = desc_lo(r_base + (uint32_t)(rs * kStageBytes), 16);
            if (leader) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                int pp = part, ww = w + kk;
                if (ww >= ks) { ww -= ks; ++pp; }
                if (ww >= ks) { ww -= ks; ++pp; }
                if (ww >= ks) { ww -= ks; ++pp; }
                if (pp < 2 * n_sets) {
                  const uint64_t b = desc_join(rb + (uint32_t)(kk * 2), dhi);
                  const uint32_t at = a_base + (uint32_t)(8 * (pp * ks + ww));
                  const uint32_t odd = (uint32_t)pp & 1u;
                  // hi * hi and lo * hi, or hi * lo
                  mma_bf16_ta(d, at - (odd ? (uint32_t)(8 * ks) : 0u), b, idesc_pos, (pp | ww) != 0);
                  if (!odd) mma_bf16_ta(d, at + (uint32_t)(8 * ks), b, idesc_pos, 1u);
                }
              }
              mma_commit(&sh.rempty[rs]);
            }
            __syncwarp();
            w += 4;
            while (w >= ks) { w -= ks; ++part; }
            if (++rs == a.n_rstages) { rs = 0; rphase ^= 1u; }
          }
        }
        if (ok && leader) mma_commit(&sh.tfull[acc]);
        __syncwarp();
      }
      if (!kStream && ok && leader) mma_commit(&sh.lempty);
      __syncwarp();
      item_phase ^= 1u;
    }
  } else if (warp < 2 + 4 * kGroups) {
    // ------------------------------------------------------------------ epilogue
    if constexpr (!kTma) {
      apply_rows_epilogue<kGroups>(a, sh, reinterpret_cast<float*>(smem_w) + (warp - 2) * 32 * kPatchPitch, tmem_acc);
    } else {
      const int wq4 = warp & 3;                             // which 32 accumulator rows this warp may read
      // The groups of four warps take the quarters in turn.  With a multiple of kGroups of buffers a buffer belongs to one
      // group: a group that waited on the other's buffers could be a whole phase ahead of a barrier, whose parity then
      // reads as complete.
      const int grp = (warp - 2) >> 2;
      const uint32_t lane_addr = (uint32_t)(32 * wq4) << 16;
      const int rloc = 32 * wq4 + lane;                     // this thread's row of the panel
      StepScalars sc = a.sc;
      const float gs = a.gscale ? *a.gscale : 1.f;
      sc.cg *= gs;               // m^c = cg (gs g) + c0 D
      // byte offsets of a 16-byte chunk of this thread's row inside a buffer: the 128-byte swizzle turns chunk c of
      // row r into chunk c ^ (r % 8), the 64-byte swizzle chunk c of a 64-byte row into c ^ ((r / 2) % 4)
      auto w_at = [&](int c) { return (uint32_t)(rloc * 128 + ((c ^ (rloc & 7)) << 4)); };
      auto g_at = [&](int c) { return (uint32_t)(kWBoxBytes + rloc * 64 + ((c ^ ((rloc >> 1) & 3)) << 4)); };
      int j = 0, b = grp;   // running tile count of this CTA, g / W buffer
      uint32_t wphase = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
        const ApplyItem I = a.items[it];
        const bool grouped = I.v_mode == ADAPM_V_BLOCKMEAN;
        const float lr_s = sc.lr * I.lr_scale;
        const int row = I.row0 + rloc;
        const bool rok = row < I.rows;
        // one denominator per row when v is a group scalar: m^c / (sqrt(v) + eps) becomes a product.  (m^c first: a group
        // that never had a gradient has v = 0, and 0 * (1 / 0) + ... would be NaN with eps = 0 where m^c is not zero.)
        const float v_row = (rok && grouped) ? a.state[I.v_off + row / I.v_group_rows] : 0.f;
        const float kr = sc.inv_bc1 / (sqrtf(v_row * sc.inv_bc2) + sc.eps);
        for (int t = 0; t < I.n_tiles && ok; ++t, ++j) {
          const int acc = j & 1;
          // one lane per warp polls, then the warp agrees: the tensor-memory loads need all 32 lanes
          bool got = true;
          if (lane == 0) got = mbar_wait(&sh.tfull[acc], (uint32_t)(j >> 1) & 1u, abort, a.status, ST_WAIT_TMEM_FULL);
          got = __shfl_sync(0xffffffffu, got, 0);
          if (!got) { ok = false; break; }
          tc_fence_after();
#pragma unroll 1
          for (int q = grp; q < kQ; q += kGroups) {
            if (!mbar_wait(&sh.wfull[b], wphase, abort, a.status, ST_WAIT_FULL)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            uint8_t* buf = smem_w + (size_t)b * a.buf_bytes;
            const int col = (I.tile0 + t) * kApplyNT + q * kApplyQC;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              float d[16];
              tmem_ld16(tmem_acc + lane_addr + (uint32_t)(acc * kApplyNT + q * kApplyQC + 16 * half), d);
              float gf[16];
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const uint4 gg = *reinterpret_cast<const uint4*>(buf + g_at(2 * half + i));
                const uint32_t gw[4] = {gg.x, gg.y, gg.z, gg.w};
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                  gf[8 * i + 2 * x] = __uint_as_float(gw[x] << 16);
                  gf[8 * i + 2 * x + 1] = __uint_as_float(gw[x] & 0xffff0000u);
                }
              }
              tmem_ld_wait();
              uint32_t shw[8];
              if (grouped) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  float4* wp = reinterpret_cast<float4*>(buf + w_at(4 * half + i));
                  const float4 wo = *wp;
                  float w[4] = {wo.x, wo.y, wo.z, wo.w};
#pragma unroll
                  for (int x = 0; x < 4; ++x) {
                    const float ratio = clamp_keep_nan((sc.cg * gf[4 * i + x] + sc.c0 * d[4 * i + x]) * kr, sc.clip);
                    w[x] = w[x] - lr_s * (ratio + I.wd * w[x]);
                  }
                  *wp = make_float4(w[0], w[1], w[2], w[3]);
                  shw[2 * i] = pack_bf16x2(w[0], w[1]);
                  shw[2 * i + 1] = pack_bf16x2(w[2], w[3]);
                }
              } else {
                // kBatch elements at a time: their chains of a root and a quotient each run side by side.  Four at a time, with
                // the rare elements in a loop that kept them in local memory, a quarter took 8.1 thousand cycles of its group:
                // 7.5 -> 5.7 ms on the 1.5B shapes, 1.65 -> 1.25 on the 350M set at rank 128; group scalars 3.0 -> 2.5 ms.
                constexpr int kBatch = kGroups == 4 ? 8 : 16;
#pragma unroll
                for (int i0 = 0; i0 < 4; i0 += kBatch / 4) {
                  float w[kBatch], vv[kBatch], mc[kBatch];
#pragma unroll
                  for (int i = 0; i < kBatch / 4; ++i) {
                    const float4 wo = *reinterpret_cast<const float4*>(buf + w_at(4 * half + i0 + i));
                    const float4 vo = *reinterpret_cast<const float4*>(buf + kApplyBufBytes + w_at(4 * half + i0 + i));   // v lies like W
                    w[4 * i] = wo.x; w[4 * i + 1] = wo.y; w[4 * i + 2] = wo.z; w[4 * i + 3] = wo.w;
                    vv[4 * i] = vo.x; vv[4 * i + 1] = vo.y; vv[4 * i + 2] = vo.z; vv[4 * i + 3] = vo.w;
                  }
#pragma unroll
                  for (int x = 0; x < kBatch; ++x) {
                    const float g1 = gf[4 * i0 + x];
                    vv[x] = sc.beta2 * vv[x] + (1.f - sc.beta2) * ((gs * g1) * (gs * g1));
                    mc[x] = sc.cg * g1 + sc.c0 * d[4 * i0 + x];
                    // (rows and columns out of range hold zeros, are not stored, and would all take the rare path)
                    if (!rok || col + 16 * half + 4 * i0 + (x & 8) >= I.cols) vv[x] = 1.f;
                  }
                  adapm_param_update_n<kBatch>(w, mc, vv, sc, lr_s, I.wd);
#pragma unroll
                  for (int i = 0; i < kBatch / 4; ++i) {
                    *reinterpret_cast<float4*>(buf + kApplyBufBytes + w_at(4 * half + i0 + i)) =
                        make_float4(vv[4 * i], vv[4 * i + 1], vv[4 * i + 2], vv[4 * i + 3]);
                    *reinterpret_cast<float4*>(buf + w_at(4 * half + i0 + i)) =
                        make_float4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
                    shw[2 * (i0 + i)] = pack_bf16x2(w[4 * i], w[4 * i + 1]);
                    shw[2 * (i0 + i) + 1] = pack_bf16x2(w[4 * i + 2], w[4 * i + 3]);
                  }
                }
              }
              if (a.shadow) {
                // The bf16 copy of the new W takes the place of the gradient in the buffer (this thread's two 16-byte
                // pieces, already read): it has g's box shape and swizzle, and is stored with the same kind of tensor
                // map.
                *reinterpret_cast<uint4*>(buf + g_at(2 * half)) = make_uint4(shw[0], shw[1], shw[2], shw[3]);
                *reinterpret_cast<uint4*>(buf + g_at(2 * half + 1)) = make_uint4(shw[4], shw[5], shw[6], shw[7]);
              }
            }
            fence_async_smem();   // every lane orders its own writes, the warp meets, one arrival per warp
            if (q + kGroups >= kQ) tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              mbar_arrive(&sh.wdone[b]);
              if (q + kGroups >= kQ) mbar_arrive(&sh.tempty[acc]);
            }
            b += kGroups;
            if (b >= a.n_bufs) { b = grp; wphase ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 2 + 4 * kGroups) {
    // ------------------------------------------------------------------ g / W mover
    if (kTma && lane == 0) {
      // load cursor: runs n_bufs quarters ahead of the quarter being stored
      int ld_it = blockIdx.x, ld_q = 0, ld_nq = 0, n_loaded = 0;
      ApplyItem LI;
      if (ld_it < a.n_items) { LI = a.items[ld_it]; ld_nq = kQ * LI.n_tiles; }
      auto load_next = [&]() {
        const int b = n_loaded % a.n_bufs;
        uint8_t* buf = smem_w + (size_t)b * a.buf_bytes;
        const int col = LI.tile0 * kApplyNT + ld_q * kApplyQC;
        const bool with_v = LI.v_mode == ADAPM_V_ELEMENT;
        mbar_arrive_expect_tx(&sh.wfull[b], (uint32_t)(kApplyBufBytes + (with_v ? kWBoxBytes : 0)));
        tma_load_box(buf, a.maps + LI.map_w, col, LI.row0, &sh.wfull[b]);
        tma_load_box(buf + kWBoxBytes, a.maps + LI.map_g, col, LI.row0, &sh.wfull[b]);
        if (with_v) tma_load_box(buf + kApplyBufBytes, a.maps + LI.map_v, col, LI.row0, &sh.wfull[b]);
        ++n_loaded;
        if (++ld_q == ld_nq) {
          ld_it += gridDim.x; ld_q = 0; ld_nq = 0;
          if (ld_it < a.n_items) { LI = a.items[ld_it]; ld_nq = kQ * LI.n_tiles; }
        }
      };
      for (int i = 0; i < a.n_bufs && ld_it < a.n_items; ++i) load_next();
      int k = 0;   // running quarter count of this CTA
      bool ok = true;
      for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
        const ApplyItem I = a.items[it];
        for (int q = 0; q < kQ * I.n_tiles; ++q, ++k) {
          const int b = k % a.n_bufs;
          if (!mbar_wait(&sh.wdone[b], (uint32_t)(k / a.n_bufs) & 1u, abort, a.status, ST_WAIT_DRAIN)) { ok = false; break; }
          const int col = I.tile0 * kApplyNT + q * kApplyQC;
          // (a quarter that lies past the last column is not stored)
          if (col < I.cols) {
            const uint8_t* buf = smem_w + (size_t)b * a.buf_bytes;
            tma_store_box(a.maps + I.map_w, col, I.row0, buf);
            if (a.shadow) tma_store_box(a.maps + I.map_sh, col, I.row0, buf + kWBoxBytes);
            if (I.v_mode == ADAPM_V_ELEMENT) tma_store_box(a.maps + I.map_v, col, I.row0, buf + kApplyBufBytes);
          }
          bulk_commit_group();
          if ((k & 1) && ld_it < a.n_items) {
            // two quarters at a time: their rows are neighbours in memory, and requests that reach DRAM
            // together share its open pages (one at a time, by a thread of its own: 8.2 instead of 6.8 ms on the 1.5B
            // shapes with a per-element v).  They go into this buffer and the one stored before it, once both
            // stores have read them.
            bulk_wait_group_read<0>();
            load_next();
            if (ld_it < a.n_items) load_next();
          }
        }
      }
      bulk_wait_group<0>();
      if (!ok) {   // let the loads already issued land before the CTA exits
        for (int kk = k; kk < n_loaded; ++kk) {
          const uint32_t ph = (uint32_t)(kk / a.n_bufs) & 1u;
          for (uint32_t spin = 0; spin < kSpinLimit && !mbar_try_wait(&sh.wfull[kk % a.n_bufs], ph); ++spin)
            __nanosleep(64);
        }
      }
    }
  } else if (!kStream) {
    // ------------------------------------------------------------------ L panel -> tensor memory, one row per thread
    // The loads of 64 columns are in flight together, and those of an item's first 64 before the tensor memory is free:
    // the MMAs wait for this between two items.  (160 columns at a time: 2.86 instead of 2.80 ms on the 1.5B shapes, 6.85
    // instead of 6.58 with a per-element v, 1.39 instead of 1.36 on the 350M set at rank 128; 32: 2.89, 6.65 and 1.37.)
    const int sub = warp & 3;                                // which 32 lanes of tensor memory this warp may write
    const uint32_t lane_addr = (uint32_t)(32 * sub) << 16;
    uint32_t item_phase = 0;
    for (int it = blockIdx.x; it < a.n_items; it += gridDim.x) {
      const int rp = a.items[it].rp, row = a.items[it].row0 + 32 * sub + lane;
      const bool rok = row < a.items[it].rows;
      // [hi0 | lo0 | hi1 | lo1] without gaps (half = rp); with one set in use, that set alone
      const int width = n_sets * 2 * rp;
      const uint16_t* src = a.work + a.items[it].l_off + (int64_t)row * (4 * rp) + (n_sets == 2 ? 0 : a.parity * 2 * rp);
      // the refitted set enters negated
      const int neg0 = n_sets == 2 ? (1 - a.parity) * 2 * rp : width, neg1 = neg0 + 2 * rp;
      uint4 x[8];
      auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          x[i] = make_uint4(0, 0, 0, 0);
          if (rok && k0 + 8 * i < width) x[i] = *reinterpret_cast<const uint4*>(src + k0 + 8 * i);
        }
      };
      fetch(0);
      if (!mbar_wait_warp(&sh.lempty, item_phase ^ 1u, abort, a.status, ST_WAIT_EMPTY)) break;
      tc_fence_after();
      for (int k0 = 0; k0 < width; k0 += 64) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = k0 + 16 * i;
          if (k < width) {
            const uint32_t flip = k >= neg0 && k < neg1 ? 0x80008000u : 0u;
            const uint4 p = x[2 * i], q = x[2 * i + 1];
            const uint32_t v[8] = {p.x ^ flip, p.y ^ flip, p.z ^ flip, p.w ^ flip, q.x ^ flip, q.y ^ flip, q.z ^ flip, q.w ^ flip};
            tmem_st8(tmem_base + lane_addr + (uint32_t)(k >> 1), v);
          }
        }
        if (k0 + 64 < width) fetch(k0 + 64);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.lfull);
      item_phase ^= 1u;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace tc
}  // namespace adapm

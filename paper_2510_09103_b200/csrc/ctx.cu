// Context creation (validation, state / workspace layout, the static per-step launch program) and
// the step driver.  The driver only orders kernels on the caller's stream: it never allocates,
// copies to the host or synchronises.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <exception>
#include <new>

#include <nvtx3/nvToolsExt.h>

#include "adapm_internal.h"

namespace adapm {

static thread_local std::string g_cuda_error;

void set_cuda_error(cudaError_t e, const char* where) {
  g_cuda_error = std::string(cudaGetErrorName(e)) + ": " + cudaGetErrorString(e) + " at " + where;
}

void set_error_text(const char* text) { g_cuda_error = text ? text : ""; }

namespace {

template <typename T>
int64_t append_table(std::vector<unsigned char>& blob, const std::vector<T>& tab) {
  const size_t off = (blob.size() + 15) / 16 * 16;
  blob.resize(off + tab.size() * sizeof(T));
  if (!tab.empty()) std::memcpy(blob.data() + off, tab.data(), tab.size() * sizeof(T));
  return (int64_t)off;
}

double inner_eta(int k, int K) { return 0.5 * (1.0 + std::cos(M_PI * (double)k / (double)K)); }

int validate(const adapm_block* blocks, int64_t n, const adapm_hparams& hp) {
  if (!(hp.beta1 >= 0.f && hp.beta1 < 1.f) || !(hp.beta2 >= 0.f && hp.beta2 < 1.f)) return ADAPM_ERANGE;
  if (!(hp.eps >= 0.f) || !(hp.clip > 0.f) || hp.inner_iters < 0 || hp.inner_iters > 64) return ADAPM_ERANGE;
  if (!std::isfinite(hp.lr) || !std::isfinite(hp.inner_lr_scale)) return ADAPM_EINVAL;
  if (hp.grad_dtype != ADAPM_GRAD_F32 && hp.grad_dtype != ADAPM_GRAD_BF16) return ADAPM_EINVAL;
  if (hp.lowrank_path < ADAPM_PATH_AUTO || hp.lowrank_path > ADAPM_PATH_TENSOR) return ADAPM_EINVAL;
  if (hp.refresh_period < 0) return ADAPM_ERANGE;
  if (!(hp.max_grad_norm >= 0.f)) return ADAPM_ERANGE;      // 0 and +inf both mean "no clipping"; NaN is refused
  if (hp.tune_panels < 0 || hp.tune_panels > 3) return ADAPM_ERANGE;
  if (hp.tune_stage_k != 0 && hp.tune_stage_k != 64 && hp.tune_stage_k != 128) return ADAPM_ERANGE;
  if (hp.inner_precond != 0 && hp.inner_precond != 1) return ADAPM_EINVAL;
  if (hp.inner_precond && !(hp.precond_damping >= 0.f && std::isfinite(hp.precond_damping))) return ADAPM_ERANGE;
  std::vector<std::pair<int64_t, int64_t>> spans;
  spans.reserve((size_t)n);
  for (int64_t i = 0; i < n; ++i) {
    const adapm_block& b = blocks[i];
    if (b.rows < 1 || b.cols < 1 || b.offset < 0) return ADAPM_ERANGE;
    if (b.offset % kAlignElems) return ADAPM_EALIGN;
    if (b.mom_mode < ADAPM_MOM_NONE || b.mom_mode > ADAPM_MOM_LOWRANK) return ADAPM_EINVAL;
    if (b.v_mode != ADAPM_V_ELEMENT && b.v_mode != ADAPM_V_BLOCKMEAN) return ADAPM_EINVAL;
    if (b.mom_mode == ADAPM_MOM_LOWRANK) {
      if (b.rank < 1 || b.rank > std::min(b.rows, b.cols)) return ADAPM_ERANGE;
    } else if (b.rank != 0) {
      return ADAPM_EINVAL;
    }
    if (b.v_mode == ADAPM_V_BLOCKMEAN) {
      if (b.v_group_rows < 0 || b.v_group_rows > b.rows) return ADAPM_ERANGE;
      if (b.v_group_rows > 0 && b.rows % b.v_group_rows) return ADAPM_ERANGE;
    }
    if (!std::isfinite(b.lr_scale) || !std::isfinite(b.weight_decay)) return ADAPM_EINVAL;
    spans.emplace_back(b.offset, b.offset + (int64_t)b.rows * b.cols);
  }
  std::sort(spans.begin(), spans.end());
  for (size_t i = 1; i < spans.size(); ++i)
    if (spans[i].first < spans[i - 1].second) return ADAPM_EINVAL;   // overlapping blocks
  return ADAPM_OK;
}


// The apply launch of the CUDA-core blocks; previous L and R and the refitted pair at the given bases (floats).
void add_simt_apply(adapm_ctx* c, const std::vector<int64_t>& ids, int phase, int l0_base, int64_t l0_shift, int r0_base,
                    int64_t r0_shift, int l1_base, int64_t l1_shift, int r1_base, int64_t r1_shift) {
  std::vector<ApplyBlk> ab;
  std::vector<int32_t> tile_blk;
  for (int64_t i : ids) {
    const adapm_block& b = c->blocks[i];
    ApplyBlk a;
    std::memset(&a, 0, sizeof(a));
    a.off = b.offset;
    a.l0_base = l0_base; a.l0_off = l0_shift + c->l_off[i];
    a.r0_base = r0_base; a.r0_off = r0_shift + c->r_off[i];
    a.l1_base = l1_base; a.l1_off = l1_shift + c->l_off[i];
    a.r1_base = r1_base; a.r1_off = r1_shift + c->r_off[i];
    a.v_off = c->v_off[i]; a.rows = b.rows; a.cols = b.cols; a.rank = b.rank; a.v_mode = b.v_mode;
    a.v_group_rows = b.v_group_rows == 0 ? b.rows : b.v_group_rows;
    a.lr_scale = b.lr_scale; a.wd = b.weight_decay;
    a.tiles_n = (b.cols + kApplyTile - 1) / kApplyTile; a.first_tile = (int64_t)tile_blk.size();
    tile_blk.insert(tile_blk.end(), (size_t)((b.rows + kApplyTile - 1) / kApplyTile) * a.tiles_n, (int32_t)ab.size());
    ab.push_back(a);
  }
  Launch L{LK_APPLY_SIMT, append_table(c->h_tables, ab), (int64_t)ab.size(), (int64_t)tile_blk.size()};
  L.aux0 = append_table(c->h_tables, tile_blk);
  L.phase = phase;
  c->program.push_back(L);
}

// The refitted factors go back to the state, sub-buffer by sub-buffer (the padding between them is not touched).
void add_commit(adapm_ctx* c, const std::vector<int64_t>& ids, int phase) {
  std::vector<NormRange> ranges;
  std::vector<int32_t> cta_range;
  for (int64_t i : ids) {
    const adapm_block& b = c->blocks[i];
    for (int which = phase == 2 ? 1 : 0; which < 2; ++which) {      // (a step that holds L has only R to bring back)
      NormRange r{which ? c->r_off[i] : c->l_off[i], (int64_t)b.rank * (which ? b.cols : b.rows), (int64_t)cta_range.size()};
      for (int64_t q = 0; q < (r.numel + kNormChunk - 1) / kNormChunk; ++q) cta_range.push_back((int32_t)ranges.size());
      ranges.push_back(r);
    }
  }
  Launch CM{LK_COMMIT, append_table(c->h_tables, ranges), (int64_t)ranges.size(), (int64_t)cta_range.size()};
  CM.aux0 = append_table(c->h_tables, cta_range);
  CM.phase = phase;
  c->program.push_back(CM);
}

// The preconditioned passes (scaled gradient descent) of the CUDA-core blocks, on the batched GEMM.
// Workspace: two copies of the [L,R] section (ping-pong iterates), A/B with the same layout, Gram matrices and inverses.
void build_precond_program(adapm_ctx* c, const std::vector<int64_t>& lowrank_ids, const std::vector<double>& etas,
                           int64_t& work_cursor) {
  const adapm_hparams* hp = &c->hp;
  auto& prog = c->program;
  const int n = (int)c->blocks.size(), K_eff = (int)etas.size();
  const bool with_hold = hp->refresh_period > 1 && K_eff > 0;
  {
    c->ws_lr[0] = work_cursor; work_cursor += c->lr_section_floats;
    c->ws_lr[1] = work_cursor; work_cursor += c->lr_section_floats;
    const int64_t ws_ab = work_cursor; work_cursor += c->lr_section_floats;
    std::vector<int64_t> gram_off(n, 0);
    for (int64_t i : lowrank_ids) {
      gram_off[i] = work_cursor;
      work_cursor += round_up(6LL * c->blocks[i].rank * c->blocks[i].rank, kStateAlign);
    }
    const float b1 = hp->beta1, a1 = 1.f - hp->beta1;
    int src_base = BASE_STATE; int64_t src_shift = 0;   // where the current iterate lives
    int dst_buf = 0;
    // with a refresh period the passes exist twice: refitting both factors (phase 1) and holding L (phase 2)
    for (int phase = (with_hold ? 1 : 0); phase <= (with_hold ? 2 : 0); ++phase) {
    const bool hold = phase == 2;
    src_base = BASE_STATE; src_shift = 0; dst_buf = 0;
    for (int it = 0; it < K_eff; ++it) {
      const float se = (float)etas[it];
      const int64_t dst_shift = c->ws_lr[dst_buf];
      std::vector<GemmProb> pAB, pG, pU1, pU2, pU3;
      std::vector<InverseJob> inv;
      int64_t tAB = 0, tG = 0, tU1 = 0, tU2 = 0, tU3 = 0;
      auto push = [](std::vector<GemmProb>& v, GemmProb p, int64_t& tiles) {
        p.tiles_n = (p.N + 63) / 64;
        p.first_tile = tiles;
        tiles += (int64_t)((p.M + 63) / 64) * p.tiles_n;
        v.push_back(p);
      };
      for (int64_t i : lowrank_ids) {
        const adapm_block& b = c->blocks[i];
        const int m = b.rows, nn = b.cols, r = b.rank;
        const int64_t Lc = src_shift + c->l_off[i], Rc = src_shift + c->r_off[i];   // current iterate
        const int64_t L0 = c->l_off[i], R0 = c->r_off[i];                             // previous factors (state)
        const int64_t Ld = dst_shift + c->l_off[i], Rd = dst_shift + c->r_off[i];
        const int64_t Aw = ws_ab + c->l_off[i], Bw = ws_ab + c->r_off[i];
        const int64_t G1 = gram_off[i], G2 = G1 + (int64_t)r * r, G3 = G2 + (int64_t)r * r, G4 = G3 + (int64_t)r * r;
        GemmProb p;
        auto reset = [&]() {
          std::memset(&p, 0, sizeof(p));
          p.z1_base = p.z2_base = BASE_NONE;
          p.alpha = 1.f;
        };
        // A = g R^T  (m x r), contraction over n
        reset(); p.x_base = BASE_GRADS; p.x_off = b.offset; p.sxi = nn; p.sxk = 1;
        p.y_base = (int8_t)src_base; p.y_off = Rc; p.syk = 1; p.syj = nn;
        p.c_base = BASE_WORK; p.c_off = Aw; p.M = m; p.N = r; p.K = nn; p.ldc = r; if (!hold) push(pAB, p, tAB);
        // B = L^T g  (r x n), contraction over m
        reset(); p.x_base = (int8_t)src_base; p.x_off = Lc; p.sxi = 1; p.sxk = r;
        p.y_base = BASE_GRADS; p.y_off = b.offset; p.syk = nn; p.syj = 1;
        p.c_base = BASE_WORK; p.c_off = Bw; p.M = r; p.N = nn; p.K = m; p.ldc = nn; push(pAB, p, tAB);
        // G1 = R R^T, G2 = R0 R^T  (contraction over n)
        reset(); p.x_base = (int8_t)src_base; p.x_off = Rc; p.sxi = nn; p.sxk = 1;
        p.y_base = (int8_t)src_base; p.y_off = Rc; p.syk = 1; p.syj = nn;
        p.c_base = BASE_WORK; p.c_off = G1; p.M = r; p.N = r; p.K = nn; p.ldc = r; if (!hold) push(pG, p, tG);
        p.x_base = BASE_STATE; p.x_off = R0; p.c_off = G2; if (!hold) push(pG, p, tG);
        // G3 = L^T L, G4 = L^T L0  (contraction over m)
        reset(); p.x_base = (int8_t)src_base; p.x_off = Lc; p.sxi = 1; p.sxk = r;
        p.y_base = (int8_t)src_base; p.y_off = Lc; p.syk = r; p.syj = 1;
        p.c_base = BASE_WORK; p.c_off = G3; p.M = r; p.N = r; p.K = m; p.ldc = r; push(pG, p, tG);
        p.y_base = BASE_STATE; p.y_off = L0; p.c_off = G4; push(pG, p, tG);
        // Preconditioned pass: A <- L G1 - a1 A, A <- A - b1 L0 G2 (= dl/dL), L' = L - se A S1 with
        // S1 = (G1 + d I)^-1; B <- G3 R - a1 B, B <- B - b1 G4 R0 (= dl/dR), R' = R - se S3 B, S3 = (G3 + d I)^-1.
        const int64_t S1 = G4 + (int64_t)r * r, S3 = S1 + (int64_t)r * r;
        if (!hold) inv.push_back({G1, S1, r, 0});
        inv.push_back({G3, S3, r, 0});
        if (!hold) {
          reset(); p.x_base = (int8_t)src_base; p.x_off = Lc; p.sxi = r; p.sxk = 1;
          p.y_base = BASE_WORK; p.y_off = G1; p.syk = r; p.syj = 1;
          p.c_base = BASE_WORK; p.c_off = Aw; p.M = m; p.N = r; p.K = r; p.ldc = r;
          p.z1_base = BASE_WORK; p.z1_off = Aw; p.c1 = -a1; push(pU1, p, tU1);
          reset(); p.x_base = BASE_STATE; p.x_off = L0; p.sxi = r; p.sxk = 1;
          p.y_base = BASE_WORK; p.y_off = G2; p.syk = r; p.syj = 1;
          p.c_base = BASE_WORK; p.c_off = Aw; p.M = m; p.N = r; p.K = r; p.ldc = r;
          p.alpha = -b1; p.beta = 1.f; push(pU2, p, tU2);
        }
        reset(); p.x_base = BASE_WORK; p.x_off = Aw; p.sxi = r; p.sxk = 1;
        p.y_base = BASE_WORK; p.y_off = S1; p.syk = r; p.syj = 1;
        p.c_base = BASE_WORK; p.c_off = Ld; p.M = m; p.N = r; p.K = r; p.ldc = r;
        p.alpha = -se; p.z1_base = (int8_t)src_base; p.z1_off = Lc; p.c1 = 1.f;
        if (hold) { p.K = 0; p.alpha = 0.f; }                                            // L' = L
        push(pU3, p, tU3);
        reset(); p.x_base = BASE_WORK; p.x_off = G3; p.sxi = r; p.sxk = 1;
        p.y_base = (int8_t)src_base; p.y_off = Rc; p.syk = nn; p.syj = 1;
        p.c_base = BASE_WORK; p.c_off = Bw; p.M = r; p.N = nn; p.K = r; p.ldc = nn;
        p.z1_base = BASE_WORK; p.z1_off = Bw; p.c1 = -a1; push(pU1, p, tU1);
        reset(); p.x_base = BASE_WORK; p.x_off = G4; p.sxi = r; p.sxk = 1;
        p.y_base = BASE_STATE; p.y_off = R0; p.syk = nn; p.syj = 1;
        p.c_base = BASE_WORK; p.c_off = Bw; p.M = r; p.N = nn; p.K = r; p.ldc = nn;
        p.alpha = -b1; p.beta = 1.f; push(pU2, p, tU2);
        reset(); p.x_base = BASE_WORK; p.x_off = S3; p.sxi = r; p.sxk = 1;
        p.y_base = BASE_WORK; p.y_off = Bw; p.syk = nn; p.syj = 1;
        p.c_base = BASE_WORK; p.c_off = Rd; p.M = r; p.N = nn; p.K = r; p.ldc = nn;
        p.alpha = -se; p.z1_base = (int8_t)src_base; p.z1_off = Rc; p.c1 = 1.f; push(pU3, p, tU3);
      }
      for (auto* pv : {&pAB, &pG, &pU1, &pU2, &pU3}) {
        if (pv == &pU1 && !inv.empty()) {       // the inverses need the Gram matrices and feed the last update
          Launch IL{LK_SPD_INVERSE, append_table(c->h_tables, inv), (int64_t)inv.size(), (int64_t)inv.size()};
          IL.phase = phase;
          prog.push_back(IL);
        }
        if (pv->empty()) continue;
        const int64_t tiles = pv == &pAB ? tAB : (pv == &pG ? tG : (pv == &pU1 ? tU1 : (pv == &pU2 ? tU2 : tU3)));
        Launch GL{LK_GEMM, append_table(c->h_tables, *pv), (int64_t)pv->size(), tiles};
        GL.phase = phase;
        prog.push_back(GL);
      }
      src_base = BASE_WORK; src_shift = dst_shift;
      c->final_lr_buf = dst_buf;
      dst_buf ^= 1;
    }
    }
    add_simt_apply(c, lowrank_ids, 0, BASE_STATE, 0, BASE_STATE, 0, src_base, src_shift, src_base, src_shift);
    if (c->final_lr_buf >= 0) add_commit(c, lowrank_ids, 0);
  }
}

// Algorithm 2 for the CUDA-core blocks: per pass one launch for the r x r matrices and one for the products with the
// gradient and the factor update.  The iterates alternate between two workspace copies of the [L,R] section; the first
// pass copies the step's previous factors to a third and the last pass writes the state, so that nothing is copied back.
// (A step with a single pass ends in the workspace and is committed after the apply.)
void build_fp32_program(adapm_ctx* c, const std::vector<int64_t>& ids, const std::vector<double>& etas, int64_t& work_cursor) {
  const adapm_hparams& hp = c->hp;
  const int K_eff = (int)etas.size();
  const bool with_hold = hp.refresh_period > 1 && K_eff > 0;
  for (int64_t& w : c->ws_lr) { w = work_cursor; work_cursor += K_eff > 0 ? c->lr_section_floats : 0; }
  const int64_t ws_prev = c->ws_lr[2];
  const int64_t scratch = work_cursor;           // matrices and partial products, every pass anew
  int64_t scratch_end = work_cursor;
  // columns per thread of a rank's tiles (8 tn columns each): as few tiles of up to 40 columns as cover it, all of one width
  auto tiles_of = [](int r) { return (r + 39) / 40; };
  auto tn_of = [&](int r) { return ((r + tiles_of(r) - 1) / tiles_of(r) + 7) / 8; };
  // K loops are cut so that a launch has about `waves` CTAs per SM and none is much longer than the rest; a chunk is
  // never below 128, where its partial products would cost as much as its share of the gradient.
  // Measured (us per step of fp32 sets; tiny 176 with every setting: its chunks are 128 long either way):
  //   waves of the refit launch    3     6     9     12    18       of the gram launch    1     2     4     8     16
  //   gpt2_124m                    3757  3628  3627  3636  3594                            3712  3644  3629  3600  3616
  //   12 layers of 768, rank 32    2780  2770  2771  2768  2782                            2916  2802  2770  2759  2774
  //   6 layers of 512              890   842   838   839   853                             858   838   837   850   849
  // Fewer leave the last wave uneven, more cost partial products; between 6 and 12, and 4 and 8, it hardly matters.
  struct Cut { int32_t k_chunk, splits; };
  auto cut = [](int K, int64_t chunk) {
    const int64_t n = std::max<int64_t>(1, (K + chunk / 2) / chunk);
    Cut q;
    q.k_chunk = (int32_t)round_up((K + n - 1) / n, 16);
    q.splits = (K + q.k_chunk - 1) / q.k_chunk;
    return q;
  };
  constexpr int64_t kWavesRefit = 9, kWavesGram = 4;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    sms = 148;

  for (int phase = (with_hold ? 1 : 0); phase <= (with_hold ? 2 : 0); ++phase) {
    const bool hold = phase == 2;
    for (int it = 0; it < K_eff; ++it) {
      const bool first = it == 0, last = it == K_eff - 1 && K_eff > 1;
      const int cur_base = first ? BASE_STATE : BASE_WORK;
      const int64_t cur = first ? 0 : c->ws_lr[(it - 1) & 1], prev = first ? 0 : ws_prev;
      const int out_base = last ? BASE_STATE : BASE_WORK;
      const int64_t out = last ? 0 : c->ws_lr[it & 1];
      int64_t k_refit = 0, k_gram = 0;            // K summed over the tiles
      for (int64_t i : ids) {
        const adapm_block& b = c->blocks[i];
        const int64_t tr = tiles_of(b.rank), tg = tr * tr * (first ? 1 : 2);
        k_refit += tr * ((hold ? 0 : (int64_t)(b.rows + 127) / 128 * b.cols) + (int64_t)(b.cols + 127) / 128 * b.rows);
        k_gram += tg * ((hold ? 0 : (int64_t)b.cols) + b.rows);
      }
      const int64_t chunk_refit = std::max<int64_t>(128, k_refit / (sms * kWavesRefit));
      const int64_t chunk_gram = std::max<int64_t>(128, k_gram / (sms * kWavesGram));
      std::vector<Fp32Gram> grams;
      std::vector<Fp32Refit> refits;
      int64_t at = scratch, counters = 0;
      for (int64_t i : ids) {
        const adapm_block& b = c->blocks[i];
        const int m = b.rows, n = b.cols, r = b.rank;
        for (int side = hold ? 1 : 0; side < 2; ++side) {          // 0: L, by rows; 1: R, by columns
          // the side's factor F (owners x r) and the other one Y (K x r): Q = g Y, Ga = Y^T Y, Gb = Y0^T Y
          const int64_t f_off = side ? c->r_off[i] : c->l_off[i], y_off = side ? c->l_off[i] : c->r_off[i];
          const int owners = side ? n : m, K = side ? m : n, along_k = side ? 0 : 1;
          // a held L stays where it is, in the state
          const int y_base = hold ? BASE_STATE : cur_base;
          const int64_t yc = (hold ? 0 : cur) + y_off, yp = (hold ? 0 : prev) + y_off;
          auto gram = [&](int64_t x_off) {
            Fp32Gram g;
            std::memset(&g, 0, sizeof(g));
            g.x_base = g.y_base = y_base; g.x_off = x_off; g.y_off = yc; g.ld = side ? r : n;
            g.r = r; g.K = K; g.along_k = along_k;
            const Cut q = cut(K, chunk_gram);
            g.k_chunk = q.k_chunk; g.splits = q.splits;
            g.tn = tn_of(r); g.tiles_n = tiles_of(r);
            const int tile_rows = 16 * ((g.tn + 1) / 2), tiles = g.tiles_n * ((r + tile_rows - 1) / tile_rows);
            g.out_off = at; at += round_up((int64_t)r * r, kStateAlign);
            g.part_off = at; if (q.splits > 1) at += (int64_t)tiles * q.splits * tile_rows * 8 * g.tn;
            at = round_up(at, kStateAlign);
            g.counter = (int32_t)counters; counters += tiles;
            grams.push_back(g);
            return g.out_off;
          };
          Fp32Refit u;
          std::memset(&u, 0, sizeof(u));
          u.g_off = b.offset; u.ldg = n; u.y_base = y_base; u.y_off = yc;
          u.cur_base = u.prev_base = cur_base; u.cur_off = cur + f_off; u.prev_off = prev + f_off;
          u.out_base = out_base; u.out_off = out + f_off;
          u.save_off = first && K_eff > 1 ? ws_prev + f_off : -1;
          u.owners = owners; u.r = r; u.K = K; u.along_k = along_k; u.eta = (float)etas[it]; u.b1 = hp.beta1;
          u.tn = tn_of(r); u.tiles_n = tiles_of(r);
          u.ga_off = gram(yc);
          u.gb_off = first ? -1 : (hold ? u.ga_off : gram(yp));
          if (!first && !hold) grams.back().x_base = BASE_WORK;
          const Cut q = cut(K, chunk_refit);
          u.k_chunk = q.k_chunk; u.splits = q.splits;
          const int tiles = u.tiles_n * ((owners + 127) / 128);
          u.part_off = at; if (q.splits > 1) at += (int64_t)tiles * q.splits * 128 * 8 * u.tn;
          at = round_up(at, kStateAlign);
          u.counter = (int32_t)counters; counters += tiles;
          refits.push_back(u);
        }
      }
      scratch_end = std::max(scratch_end, at);
      c->n_counters = std::max(c->n_counters, counters);
      // longest chunks first
      std::stable_sort(grams.begin(), grams.end(), [](const Fp32Gram& a, const Fp32Gram& b) { return a.k_chunk > b.k_chunk; });
      std::stable_sort(refits.begin(), refits.end(),
                       [](const Fp32Refit& a, const Fp32Refit& b) { return a.k_chunk * a.tn > b.k_chunk * b.tn; });
      std::vector<int32_t> unit_gram, unit_refit;
      for (size_t q = 0; q < grams.size(); ++q) {
        Fp32Gram& g = grams[q];
        const int tile_rows = 16 * ((g.tn + 1) / 2);
        g.first_unit = (int32_t)unit_gram.size();
        unit_gram.insert(unit_gram.end(), (size_t)g.tiles_n * ((g.r + tile_rows - 1) / tile_rows) * g.splits, (int32_t)q);
      }
      for (size_t q = 0; q < refits.size(); ++q) {
        Fp32Refit& u = refits[q];
        u.first_unit = (int32_t)unit_refit.size();
        unit_refit.insert(unit_refit.end(), (size_t)u.tiles_n * ((u.owners + 127) / 128) * u.splits, (int32_t)q);
      }
      Launch GL{LK_FP32_GRAM, append_table(c->h_tables, grams), (int64_t)grams.size(), (int64_t)unit_gram.size()};
      GL.aux0 = append_table(c->h_tables, unit_gram); GL.phase = phase;
      c->program.push_back(GL);
      Launch UL{LK_FP32_REFIT, append_table(c->h_tables, refits), (int64_t)refits.size(), (int64_t)unit_refit.size()};
      UL.aux0 = append_table(c->h_tables, unit_refit); UL.phase = phase;
      c->program.push_back(UL);
    }
    // where the step's previous factors and the refitted ones are when the passes are over
    const int old_base = K_eff > 1 ? BASE_WORK : BASE_STATE, new_base = K_eff == 1 ? BASE_WORK : BASE_STATE;
    const int64_t old_at = K_eff > 1 ? ws_prev : 0, new_at = K_eff == 1 ? c->ws_lr[0] : 0;
    add_simt_apply(c, ids, phase, hold ? BASE_STATE : old_base, hold ? 0 : old_at, old_base, old_at,
                   hold ? BASE_STATE : new_base, hold ? 0 : new_at, new_base, new_at);
    if (K_eff == 1) { c->final_lr_buf = 0; add_commit(c, ids, phase); }
  }
  work_cursor = scratch_end;
}

// A step's branch on the context's own stream: however the step ends, the caller's stream waits for it.
class SideBranch {
 public:
  SideBranch(adapm_ctx* c, cudaStream_t main) : c_(c), main_(main) {}
  ~SideBranch() { (void)join(); }
  cudaError_t fork() {
    cudaError_t e = cudaEventRecord(c_->fork_event, main_);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(c_->side_stream, c_->fork_event, 0);
    open_ = e == cudaSuccess;
    return e;
  }
  cudaError_t join() {
    if (!open_) return cudaSuccess;
    open_ = false;
    cudaError_t e = cudaEventRecord(c_->join_event, c_->side_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(main_, c_->join_event, 0);
    // without the event the host waits: what the caller enqueues after the error must not overtake the branch
    if (e != cudaSuccess) (void)cudaStreamSynchronize(c_->side_stream);
    return e;
  }

 private:
  adapm_ctx* c_;
  cudaStream_t main_;
  bool open_ = false;
};

}  // namespace

// the tensor-core program of the low-rank blocks; defined in lowrank_tc.cu
bool tensor_path_block_ok(const adapm_hparams& hp, const adapm_block& b);
int build_tensor_program(adapm_ctx* c, const std::vector<int64_t>& tc_ids, const std::vector<double>& etas,
                         int64_t& work_cursor, std::vector<ReduceJob>& row_jobs, int64_t& row_groups);
int tensor_prepare_step(adapm_ctx* c, const Bases& b, int64_t t, cudaStream_t s, int* parity, int* convert);
int run_tensor_launch(adapm_ctx* c, const Launch& L, const Bases& b, const StepScalars& sc, int parity,
                      cudaStream_t s);
void destroy_tensor_program(adapm_ctx* c);
void tensor_state_changed(adapm_ctx* c);
int run_expired_wait_probe(adapm_ctx* c, cudaStream_t s);
size_t probe_table(std::vector<unsigned char>& out);

}  // namespace adapm

using namespace adapm;

extern "C" const char* adapm_last_cuda_error(void) { return g_cuda_error.c_str(); }

// Fills in the context, or leaves it as far as it came for adapm_destroy.
static int create_context(adapm_ctx* c, const adapm_block* blocks, int64_t n_blocks, const adapm_hparams* hp) {
  int rc = ADAPM_OK;
  c->blocks.assign(blocks, blocks + n_blocks);
  c->hp = *hp;
  const int n = (int)n_blocks;
  const size_t gsz = hp->grad_dtype == ADAPM_GRAD_BF16 ? 2 : 4;

  // ---- which kernels run each low-rank block ----------------------------------------------------------
  std::vector<int64_t> lowrank_ids, tc_ids;     // lowrank_ids: the blocks of the CUDA-core path
  for (int i = 0; i < n; ++i) {
    const adapm_block& b = c->blocks[i];
    if (b.mom_mode != ADAPM_MOM_LOWRANK) continue;
    if (tensor_path_block_ok(*hp, b)) tc_ids.push_back(i);
    else if (hp->lowrank_path == ADAPM_PATH_TENSOR) return ADAPM_EUNSUPPORTED;
    else if (hp->inner_precond && b.rank > 4096) return ADAPM_EUNSUPPORTED;
    else lowrank_ids.push_back(i);
  }
  c->n_tensor_blocks = (int64_t)tc_ids.size();

  // ---- state layout: [L,R of the low-rank blocks TMA cannot address in place][L,R of the others]
  //                    [m^f of every full block][v of every block] --------------------------------------
  c->m_off.assign(n, -1); c->l_off.assign(n, -1); c->r_off.assign(n, -1); c->v_off.assign(n, -1); c->v_cnt.assign(n, 0);
  int64_t cur = 0;
  auto place_factors = [&](int64_t i) {
    const adapm_block& b = c->blocks[i];
    c->l_off[i] = cur; cur += round_up((int64_t)b.rows * b.rank, kStateAlign);
    c->r_off[i] = cur; cur += round_up((int64_t)b.rank * b.cols, kStateAlign);
    c->bytes_L += (size_t)b.rows * b.rank * 4;
    c->bytes_R += (size_t)b.rank * b.cols * 4;
  };
  // The layout does not depend on which kernels a block runs on today: blocks that TMA cannot address in place come
  // first whether they take the CUDA-core path or a padded copy, so that checkpoints stay readable.
  auto in_place = [&](const adapm_block& b) { return b.cols % 8 == 0 && tensor_path_block_ok(*hp, b); };
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = 0; i < n; ++i) {
      const adapm_block& b = c->blocks[i];
      if (b.mom_mode == ADAPM_MOM_LOWRANK && in_place(b) == (pass == 1)) place_factors(i);
    }
    if (pass == 0) c->lr_section_floats = cur;
  }
  for (int i = 0; i < n; ++i) {
    const adapm_block& b = c->blocks[i];
    if (b.mom_mode != ADAPM_MOM_FULL) continue;
    c->m_off[i] = cur; cur += round_up((int64_t)b.rows * b.cols, kStateAlign);
    c->bytes_m += (size_t)b.rows * b.cols * 4;
  }
  for (int i = 0; i < n; ++i) {
    const adapm_block& b = c->blocks[i];
    int64_t cnt;
    if (b.v_mode == ADAPM_V_ELEMENT) cnt = (int64_t)b.rows * b.cols;
    else cnt = b.v_group_rows == 0 ? 1 : b.rows / b.v_group_rows;
    c->v_off[i] = cur; c->v_cnt[i] = cnt; cur += round_up(cnt, kStateAlign);
    c->bytes_v += (size_t)cnt * 4;
  }
  c->state_floats = cur;

  // ---- algorithmic traffic and flops -----------------------------------------------------------
  int K_eff = 0;
  std::vector<double> etas;
  for (int k = 1; k <= hp->inner_iters; ++k) {
    const double e = inner_eta(k, hp->inner_iters) * (double)hp->inner_lr_scale;
    if (std::fabs(e) > 1e-12) { etas.push_back(e); ++K_eff; }
  }
  for (int i = 0; i < n; ++i) {
    const adapm_block& b = c->blocks[i];
    const size_t ne = (size_t)b.rows * b.cols;
    c->step_bytes += ne * (gsz + 8);
    if (b.mom_mode == ADAPM_MOM_FULL) c->step_bytes += ne * 8;
    if (b.mom_mode == ADAPM_MOM_LOWRANK) {
      c->step_bytes += (size_t)b.rank * (b.rows + b.cols) * 8;
      c->step_flops += (4.0 * K_eff + 4.0) * (double)b.rows * b.cols * b.rank;
    }
    c->step_bytes += (size_t)c->v_cnt[i] * 8;
  }

  // ---- streaming blocks and reduction jobs -------------------------------------------------------
  std::vector<StreamBlk> sblk;
  // two-stage group sums of g^2: `rjobs` run every step, `rjobs_hold` only in steps that hold L (there the
  // tensor path has no row panels to take the row sums from)
  struct ReduceSet { std::vector<ReduceJob> jobs; int64_t units = 0, groups = 0; };
  ReduceSet rset_all, rset_hold, rset_norm;      // of every step; of steps that hold L; of sums that the norm pass leaves
  int64_t cta_cursor = 0, work_cursor = 0;
  auto add_reduce_job = [&](ReduceSet& rs, int i, int64_t group_elems, int64_t n_groups) {
    std::vector<ReduceJob>& rjobs = rs.jobs;
    int64_t& unit_cursor = rs.units;
    int64_t& group_cursor = rs.groups;
    ReduceJob j;
    std::memset(&j, 0, sizeof(j));
    j.g_off = c->blocks[i].offset;
    j.group_elems = group_elems;
    j.n_groups = n_groups;
    j.v_off = c->v_off[i];
    j.chunks_per_group = (int32_t)((group_elems + kWarpUnitMax - 1) / kWarpUnitMax);
    j.part_off = work_cursor;
    work_cursor += round_up(n_groups * j.chunks_per_group, kStateAlign);
    j.first_unit = unit_cursor; unit_cursor += n_groups * j.chunks_per_group;
    j.first_group = group_cursor; group_cursor += n_groups;
    rjobs.push_back(j);
  };
  for (int i = 0; i < n; ++i) {
    const adapm_block& b = c->blocks[i];
    const int64_t numel = (int64_t)b.rows * b.cols;
    const int64_t group_elems = b.v_group_rows == 0 ? numel : (int64_t)b.v_group_rows * b.cols;
    const int64_t n_groups = numel / group_elems;
    if (b.mom_mode == ADAPM_MOM_LOWRANK) continue;
    StreamBlk s;
    std::memset(&s, 0, sizeof(s));
    s.off = b.offset; s.m_off = c->m_off[i]; s.v_off = c->v_off[i]; s.numel = numel;
    s.lr_scale = b.lr_scale; s.wd = b.weight_decay;
    s.units_per_group = 1; s.group_elems = group_elems;
    if (b.v_mode == ADAPM_V_ELEMENT) {
      s.v_mode = SV_ELEMENT; s.team = 32; s.unit_elems = kWarpUnitMax;
      s.n_units = (numel + kWarpUnitMax - 1) / kWarpUnitMax; s.vec_ok = 1;
    } else if (group_elems <= kCtaUnitMax) {
      s.v_mode = SV_GROUP_INLINE;
      s.team = group_elems <= kWarpUnitMax ? 32 : 256;
      s.unit_elems = (int32_t)group_elems; s.n_units = n_groups;
      s.vec_ok = (group_elems % kChunkElems == 0 || n_groups == 1) ? 1 : 0;
    } else {
      s.v_mode = SV_GROUP_READY; s.team = 32; s.unit_elems = kWarpUnitMax;
      s.units_per_group = (int32_t)((group_elems + kWarpUnitMax - 1) / kWarpUnitMax);
      s.n_units = n_groups * s.units_per_group;
      s.vec_ok = (group_elems % kChunkElems == 0 || n_groups == 1) ? 1 : 0;
      add_reduce_job(rset_all, i, group_elems, n_groups);
    }
    sblk.push_back(s);
  }
  // Groups of 2049 to 8192 elements (rows of wide models) in teams that just hold them, where they are a good part of the
  // set: a CTA per row of 4096 left three quarters of its registers empty and ran at 3.4 TB/s, two warps per row 6.1.  The
  // kernel form with these teams runs the other units a little slower, so it takes a share of 1/16 of the elements to pay.
  // Measured (us without | with, rows of 4096 among 300 M elements, bf16 gradients): rows of 768 at a share of 1 %
  // 970|984, 3 % 976|989, 1/16 986|983, 1/8 1001|974, 1/4 1033|955; rows of 1600 892|900, 900|906, 913|905, 935|904, 980|898.
  bool stream_teams = false;
  {
    int64_t wide = 0, all = 0;
    auto is_wide = [](const StreamBlk& s) { return s.v_mode == SV_GROUP_INLINE && s.team == 256 && s.group_elems <= kCtaUnitMax / 2; };
    for (const StreamBlk& s : sblk) {
      all += s.numel;
      if (is_wide(s)) wide += s.numel;
    }
    stream_teams = wide > all / 16;
    if (stream_teams)
      for (StreamBlk& s : sblk)
        if (is_wide(s)) s.team = s.group_elems <= kCtaUnitMax / 4 ? 64 : 128;
  }
  for (StreamBlk& s : sblk) {
    s.first_cta = cta_cursor;
    cta_cursor += (s.n_units + 256 / s.team - 1) / (256 / s.team);
  }

  // Group sums of g^2 of the low-rank blocks come from the norm pass where there is one (see norm_pass_sums_groups), else on
  // the tensor path with a refit pass from that: its row panels read every row of g anyway and leave the row sums behind.
  // Else, and on steps that hold L, from the reduction kernels.
  const bool fold_sumsq = K_eff > 0 && !(hp->flags & ADAPM_FLAG_NO_SUMSQ_FOLD);
  const bool with_hold = hp->refresh_period > 1 && K_eff > 0;
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1 && fold_sumsq && !with_hold) break;
    for (int64_t i : (pass == 0 ? lowrank_ids : tc_ids)) {
      const adapm_block& b = c->blocks[i];
      if (b.v_mode != ADAPM_V_BLOCKMEAN) continue;
      const int64_t numel = (int64_t)b.rows * b.cols;
      const int64_t group_elems = b.v_group_rows == 0 ? numel : (int64_t)b.v_group_rows * b.cols;
      if (norm_pass_sums_groups(*hp, b)) continue;
      add_reduce_job((pass == 1 && fold_sumsq) ? rset_hold : rset_all, (int)i, group_elems, numel / group_elems);
    }
  }

  auto& prog = c->program;
  // Global gradient-norm clipping (and the finite check, which rides on the same reduction) needs the norm of
  // every gradient before anything uses one: a pass of its own over g.
  if (norm_pass_on(*hp)) {
    std::vector<NormRange> ranges;
    std::vector<int32_t> cta_range;
    for (int i = 0; i < n; ++i) {
      const adapm_block& b = c->blocks[i];
      NormRange r{b.offset, (int64_t)b.rows * b.cols, (int64_t)cta_range.size()};
      int64_t ctas = (r.numel + kNormChunk - 1) / kNormChunk;
      if (norm_pass_sums_groups(*hp, b)) {
        r.group_elems = b.v_group_rows == 0 ? r.numel : (int64_t)b.v_group_rows * b.cols;
        add_reduce_job(rset_norm, i, r.group_elems, r.numel / r.group_elems);
        const ReduceJob& j = rset_norm.jobs.back();
        r.chunks = j.chunks_per_group; r.rows_off = j.part_off;          // (counted from the sums of the CTAs below)
        ctas = (j.n_groups * r.chunks + kNormUnits - 1) / kNormUnits;
      }
      cta_range.insert(cta_range.end(), (size_t)ctas, (int32_t)ranges.size());
      ranges.push_back(r);
    }
    for (NormRange& r : ranges) r.rows_off -= work_cursor;
    Launch GN{LK_GRADNORM, append_table(c->h_tables, ranges), (int64_t)ranges.size(), (int64_t)cta_range.size()};
    GN.aux0 = append_table(c->h_tables, cta_range);
    GN.aux1 = work_cursor;                                   // per-chunk sums
    work_cursor += round_up((int64_t)cta_range.size(), kStateAlign);
    prog.push_back(GN);
    c->use_gscale = 1;
  }
  for (int which = 0; which < 3; ++which) {
    const ReduceSet& rs = which == 0 ? rset_all : which == 1 ? rset_hold : rset_norm;
    const std::vector<ReduceJob>& rjobs = rs.jobs;
    if (rjobs.empty()) continue;
    const int64_t off = append_table(c->h_tables, rjobs);
    // CTA index -> job of the CTA's first unit (the job table is sorted by first_unit), so that a warp finds its job
    // with a step or two instead of a binary search
    std::vector<int32_t> cta_job((size_t)((rs.units + 7) / 8));
    for (size_t q = 0, j = 0; q < cta_job.size(); ++q) {
      while (j + 1 < rjobs.size() && rjobs[j + 1].first_unit <= (int64_t)q * 8) ++j;
      cta_job[q] = (int32_t)j;
    }
    Launch RP{LK_REDUCE_PARTIAL, off, (int64_t)rjobs.size(), (rs.units + 7) / 8, rs.units};
    RP.aux1 = append_table(c->h_tables, cta_job);
    RP.phase = which == 1 ? 2 : 0;
    if (which < 2) prog.push_back(RP);
    Launch RF{LK_REDUCE_FINAL, off, (int64_t)rjobs.size(), (rs.groups + 7) / 8, rs.groups};
    RF.phase = RP.phase;
    prog.push_back(RF);
  }
  if (!sblk.empty()) {
    const int64_t off = append_table(c->h_tables, sblk);
    std::vector<int32_t> cta_blk((size_t)cta_cursor);       // CTA index -> entry of the block table
    for (size_t i = 0; i < sblk.size(); ++i) {
      const int64_t end = i + 1 < sblk.size() ? sblk[i + 1].first_cta : cta_cursor;
      for (int64_t q = sblk[i].first_cta; q < end; ++q) cta_blk[(size_t)q] = (int32_t)i;
    }
    Launch SL{LK_STREAM, off, (int64_t)sblk.size(), cta_cursor};
    SL.aux0 = append_table(c->h_tables, cta_blk);
    SL.aux1 = stream_teams ? 1 : 0;
    prog.push_back(SL);
  }

  // ---- low-rank program --------------------------------------------------------------------------
  if (!lowrank_ids.empty() || !tc_ids.empty()) {
    std::vector<InitJob> ijobs;
    for (int pass = 0; pass < 2; ++pass)
      for (int64_t i : (pass == 0 ? lowrank_ids : tc_ids))
        ijobs.push_back({c->l_off[i], i, c->blocks[i].rows, c->blocks[i].rank});
    c->init_table_off = append_table(c->h_tables, ijobs);
    c->n_init_jobs = (int64_t)ijobs.size();
    // Y = g Omega -> the block's L in the state (data-driven L_0)
    c->omega_off.assign(n, -1);
    std::vector<GemmProb> rp;
    int64_t tiles = 0;
    for (int pass = 0; pass < 2; ++pass)
      for (int64_t i : (pass == 0 ? lowrank_ids : tc_ids)) {
        const adapm_block& b = c->blocks[i];
        c->omega_off[i] = c->omega_floats;
        c->omega_floats += round_up((int64_t)b.cols * b.rank, kStateAlign);
        GemmProb p;
        std::memset(&p, 0, sizeof(p));
        p.z1_base = p.z2_base = BASE_NONE;
        p.alpha = 1.f;
        p.x_base = BASE_GRADS; p.x_off = b.offset; p.sxi = b.cols; p.sxk = 1;
        p.y_base = BASE_WORK; p.y_off = c->omega_off[i]; p.syk = b.rank; p.syj = 1;
        p.c_base = BASE_STATE; p.c_off = c->l_off[i]; p.M = b.rows; p.N = b.rank; p.K = b.cols; p.ldc = b.rank;
        p.tiles_n = (p.N + 63) / 64;
        p.first_tile = tiles;
        tiles += (int64_t)((p.M + 63) / 64) * p.tiles_n;
        rp.push_back(p);
      }
    c->range_table_off = append_table(c->h_tables, rp);
    c->n_range_probs = (int64_t)rp.size();
    c->n_range_tiles = tiles;
  }
  if (!tc_ids.empty()) {
    std::vector<ReduceJob> row_jobs;
    int64_t row_groups = 0;
    rc = build_tensor_program(c, tc_ids, etas, work_cursor, row_jobs, row_groups);
    if (rc != ADAPM_OK) return rc;
    if (!row_jobs.empty()) {
      const int64_t off = append_table(c->h_tables, row_jobs);
      for (Launch& L : prog)
        if (L.kind == LK_REDUCE_ROWS) {
          L.table_off = off; L.n_items = (int64_t)row_jobs.size(); L.grid = (row_groups + 7) / 8; L.aux0 = row_groups;
        }
    }
  }
  if (!lowrank_ids.empty()) {
    if (hp->inner_precond) build_precond_program(c, lowrank_ids, etas, work_cursor);
    else build_fp32_program(c, lowrank_ids, etas, work_cursor);
  }
  c->work_floats = work_cursor;

  // ---- upload ------------------------------------------------------------------------------------
  cudaError_t e = cudaGetDevice(&c->device);
  if (e == cudaSuccess) e = cudaMalloc((void**)&c->d_tables, std::max<size_t>(c->h_tables.size(), 16));
  if (e == cudaSuccess && !c->h_tables.empty())
    e = cudaMemcpy(c->d_tables, c->h_tables.data(), c->h_tables.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc((void**)&c->d_status, 256);
  if (e == cudaSuccess) e = cudaMemset(c->d_status, 0, 256);
  if (e == cudaSuccess && c->use_gscale) {
    const float ones[2] = {1.f, 1.f};
    e = cudaMalloc((void**)&c->d_gscale, 256);
    if (e == cudaSuccess) e = cudaMemcpy(c->d_gscale, ones, sizeof(ones), cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess && c->n_counters > 0) {
    e = cudaMalloc((void**)&c->d_counters, (size_t)c->n_counters * 4);
    if (e == cudaSuccess) e = cudaMemset(c->d_counters, 0, (size_t)c->n_counters * 4);
  }
  {
    std::vector<unsigned char> probe;
    const size_t pb = probe_table(probe);
    if (e == cudaSuccess) e = cudaMalloc((void**)&c->d_probe, pb);
    if (e == cudaSuccess) e = cudaMemcpy(c->d_probe, probe.data(), pb, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess && c->n_init_jobs > 0 && !sblk.empty()) {
    int least = 0, greatest = 0;
    e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&c->side_stream, cudaStreamNonBlocking, least);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->fork_event, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->join_event, cudaEventDisableTiming);
  }
  if (e != cudaSuccess) {
    set_cuda_error(e, "adapm_create upload");
    return ADAPM_ECUDA;
  }
  return ADAPM_OK;
}

extern "C" int adapm_create(const adapm_block* blocks, int64_t n_blocks, const adapm_hparams* hp, adapm_ctx** out) {
  if (!blocks || n_blocks <= 0 || !hp || !out) return ADAPM_EINVAL;
  *out = nullptr;
  adapm_ctx* c = nullptr;
  int rc;
  try {
    rc = validate(blocks, n_blocks, *hp);
    if (rc != ADAPM_OK) return rc;
    c = new adapm_ctx();
    rc = create_context(c, blocks, n_blocks, hp);
  } catch (const std::exception&) {       // tables too large for the host's memory: a size no device holds either
    set_error_text("adapm_create: out of host memory");
    rc = ADAPM_EINVAL;
  }
  if (rc != ADAPM_OK) adapm_destroy(c);
  else *out = c;
  return rc;
}

extern "C" void adapm_destroy(adapm_ctx* c) {
  if (!c) return;
  destroy_tensor_program(c);
  for (auto e : c->prof_events) if (e) cudaEventDestroy(e);
  if (c->side_stream) cudaStreamDestroy(c->side_stream);
  if (c->fork_event) cudaEventDestroy(c->fork_event);
  if (c->join_event) cudaEventDestroy(c->join_event);
  if (c->d_tables) cudaFree(c->d_tables);
  if (c->d_status) cudaFree(c->d_status);
  if (c->d_probe) cudaFree(c->d_probe);
  if (c->d_gscale) cudaFree(c->d_gscale);
  if (c->d_counters) cudaFree(c->d_counters);
  delete c;
}

extern "C" size_t adapm_state_bytes(const adapm_ctx* c) { return c ? (size_t)c->state_floats * 4 : 0; }

extern "C" int adapm_state_breakdown(const adapm_ctx* c, size_t* full_m, size_t* L, size_t* R, size_t* v) {
  if (!c) return ADAPM_EINVAL;
  if (full_m) *full_m = c->bytes_m;
  if (L) *L = c->bytes_L;
  if (R) *R = c->bytes_R;
  if (v) *v = c->bytes_v;
  return ADAPM_OK;
}

extern "C" int adapm_state_layout(const adapm_ctx* c, int64_t block, int which, int64_t* offset, int64_t* count) {
  if (!c || !offset || !count) return ADAPM_EINVAL;
  if (block < 0 || block >= (int64_t)c->blocks.size()) return ADAPM_ERANGE;
  const adapm_block& b = c->blocks[block];
  int64_t off = -1, cnt = 0;
  switch (which) {
    case ADAPM_STATE_M: off = c->m_off[block]; cnt = off >= 0 ? (int64_t)b.rows * b.cols : 0; break;
    case ADAPM_STATE_L: off = c->l_off[block]; cnt = off >= 0 ? (int64_t)b.rows * b.rank : 0; break;
    case ADAPM_STATE_R: off = c->r_off[block]; cnt = off >= 0 ? (int64_t)b.rank * b.cols : 0; break;
    case ADAPM_STATE_V: off = c->v_off[block]; cnt = c->v_cnt[block]; break;
    default: return ADAPM_EINVAL;
  }
  *offset = off;
  *count = cnt;
  return ADAPM_OK;
}

extern "C" size_t adapm_workspace_bytes(const adapm_ctx* c) { return c ? (size_t)c->work_floats * 4 : 0; }

extern "C" int adapm_set_workspace(adapm_ctx* c, void* dev_ptr, size_t bytes) {
  if (!c) return ADAPM_EINVAL;
  if (c->work_floats > 0) {
    if (!dev_ptr) return ADAPM_EINVAL;
    if ((uintptr_t)dev_ptr % 256) return ADAPM_EALIGN;
    if (bytes < (size_t)c->work_floats * 4) return ADAPM_ENOWORKSPACE;
  }
  c->workspace = dev_ptr;
  c->workspace_bytes = bytes;
  return ADAPM_OK;
}

extern "C" int adapm_state_init(adapm_ctx* c, void* state, adapm_stream stream) {
  if (!c || !state) return ADAPM_EINVAL;
  if ((uintptr_t)state % 256) return ADAPM_EALIGN;
  cudaStream_t s = (cudaStream_t)stream;
  ADAPM_CUDA(cudaMemsetAsync(state, 0, (size_t)c->state_floats * 4, s));
  tensor_state_changed(c);
  if (c->n_init_jobs > 0)
    return launch_init_L0((const InitJob*)(c->d_tables + c->init_table_off), c->n_init_jobs, (float*)state, c->hp.seed, 1, s);
  return ADAPM_OK;
}

extern "C" int64_t adapm_init_omega_floats(const adapm_ctx* c) { return c ? c->omega_floats : 0; }

extern "C" int adapm_init_omega_layout(const adapm_ctx* c, int64_t block, int64_t* offset, int64_t* count) {
  if (!c || !offset || !count) return ADAPM_EINVAL;
  if (block < 0 || block >= (int64_t)c->blocks.size()) return ADAPM_ERANGE;
  const bool lowrank = !c->omega_off.empty() && c->omega_off[(size_t)block] >= 0;
  *offset = lowrank ? c->omega_off[(size_t)block] : 0;
  *count = lowrank ? (int64_t)c->blocks[(size_t)block].cols * c->blocks[(size_t)block].rank : 0;
  return ADAPM_OK;
}

extern "C" int adapm_state_init_from_grads(adapm_ctx* c, void* state, const void* grads, const float* omega,
                                           adapm_stream stream) {
  if (!c || !state || !grads) return ADAPM_EINVAL;
  if (c->n_init_jobs > 0 && !omega) return ADAPM_EINVAL;
  if ((uintptr_t)state % 256 || (uintptr_t)grads % 16 || (uintptr_t)omega % 16) return ADAPM_EALIGN;
  cudaStream_t s = (cudaStream_t)stream;
  ADAPM_CUDA(cudaMemsetAsync(state, 0, (size_t)c->state_floats * 4, s));
  tensor_state_changed(c);
  if (c->n_init_jobs == 0) return ADAPM_OK;
  Bases b;
  b.p[BASE_PARAMS] = nullptr; b.p[BASE_GRADS] = const_cast<void*>(grads); b.p[BASE_STATE] = state;
  b.p[BASE_WORK] = const_cast<float*>(omega);
  b.status = c->d_status; b.gscale = nullptr; b.shadow = nullptr;
  const int rc = launch_gemm((const GemmProb*)(c->d_tables + c->range_table_off), c->n_range_probs, c->n_range_tiles, b,
                             c->hp.grad_dtype, s);
  if (rc != ADAPM_OK) return rc;
  return launch_init_L0((const InitJob*)(c->d_tables + c->init_table_off), c->n_init_jobs, (float*)state, c->hp.seed, 0, s);
}

extern "C" int adapm_set_lr(adapm_ctx* c, float lr) {
  if (!c || !std::isfinite(lr)) return ADAPM_EINVAL;
  c->hp.lr = lr;
  return ADAPM_OK;
}

extern "C" size_t adapm_step_bytes(const adapm_ctx* c) { return c ? c->step_bytes : 0; }
extern "C" double adapm_step_flops(const adapm_ctx* c) { return c ? c->step_flops : 0.0; }
extern "C" int64_t adapm_launch_count(const adapm_ctx* c) {
  if (!c) return 0;
  if (c->last_step_launches > 0) return c->last_step_launches;
  int64_t n = 0;
  for (const Launch& L : c->program)
    if ((L.when == WHEN_ALWAYS || L.when == WHEN_EVEN) && !L.only_convert && L.phase != 2) ++n;
  return n;
}

extern "C" int adapm_set_shadow_params(adapm_ctx* c, void* bf16_dev_ptr) {
  if (!c) return ADAPM_EINVAL;
  if ((uintptr_t)bf16_dev_ptr % 256) return ADAPM_EALIGN;
  c->shadow = bf16_dev_ptr;
  return ADAPM_OK;
}

extern "C" int adapm_state_changed(adapm_ctx* c) {
  if (!c) return ADAPM_EINVAL;
  tensor_state_changed(c);
  return ADAPM_OK;
}

extern "C" int adapm_selftest_expired_wait(adapm_ctx* c, adapm_stream stream) {
  if (!c) return ADAPM_EINVAL;
  return run_expired_wait_probe(c, (cudaStream_t)stream);
}

static int enqueue_step(adapm_ctx* c, void* params, const void* grads, void* state, int64_t t, cudaStream_t s) {
  const adapm_hparams& hp = c->hp;

  StepScalars sc;
  sc.lr = hp.lr; sc.beta1 = hp.beta1; sc.beta2 = hp.beta2; sc.eps = hp.eps; sc.clip = hp.clip;
  if (hp.adam_debias) {
    sc.inv_bc1 = (float)(1.0 / (1.0 - std::pow((double)hp.beta1, (double)t)));
    sc.inv_bc2 = (float)(1.0 / (1.0 - std::pow((double)hp.beta2, (double)t)));
  } else {
    sc.inv_bc1 = sc.inv_bc2 = 1.f;
  }
  if (hp.correction) {            // m^c = g + c (P_{t-1} - P_t), c = beta1 / (1 - beta1): lines 4, 6, 8 combined
    const float cc = hp.beta1 / (1.f - hp.beta1);
    sc.cg = 1.f; sc.c0 = cc; sc.c1 = cc;
  } else {                        // m^c = m_t = (1-beta1) g + beta1 P_{t-1}
    sc.cg = 1.f - hp.beta1; sc.c0 = hp.beta1; sc.c1 = 0.f;
  }

  Bases b;
  b.p[BASE_PARAMS] = params; b.p[BASE_GRADS] = const_cast<void*>(grads); b.p[BASE_STATE] = state;
  b.p[BASE_WORK] = c->workspace;
  b.status = c->d_status; b.gscale = c->d_gscale; b.shadow = (uint16_t*)c->shadow;
  float* work = (float*)c->workspace;

  // refresh period T: both factors are refitted at steps 1, T+1, 2T+1, ...; the steps in between hold L
  const bool refresh = hp.refresh_period <= 1 || (t - 1) % hp.refresh_period == 0;
  int parity = 0, convert = 0;
  if (c->tc) {
    const int prc = tensor_prepare_step(c, b, t, s, &parity, &convert);
    if (prc != ADAPM_OK) return prc;
  }
  const bool prof = c->profiling && c->prof_events.size() == c->program.size() + 1;
  if (prof) {
    c->prof_kinds.clear();
    ADAPM_CUDA(cudaEventRecord(c->prof_events[0], s));
  }
  // The streaming update touches other blocks than the low-rank launches do.  Up to a few GB per step, where those leave
  // SMs idle, it runs beside them on the context's own stream, forked off before its launch and joined at the end of the
  // step (under stream capture the side stream becomes a branch of the graph): 150 -> 134 us on the tiny set, 270 -> 234
  // on a two-layer set of width 576, 1-2 % at 1 GB, nothing to be had above.  Per-launch profiling times the launches one
  // by one.
  const bool fork = c->side_stream && !prof && c->step_bytes < (size_t)4 << 30;
  cudaStream_t const main_stream = s;
  SideBranch branch(c, main_stream);
  size_t li = 0;
  for (const Launch& L : c->program) {
    if ((L.only_convert && !convert) || (L.when == WHEN_EVEN && parity != 0) || (L.when == WHEN_ODD && parity != 1) ||
        (L.phase == 1 && !refresh) || (L.phase == 2 && refresh))
      continue;
    const unsigned char* tab = c->d_tables + L.table_off;
    int rc = ADAPM_OK;
    if (prof) nvtxRangePushA(adapm_launch_kind_name((int32_t)L.kind));   // a named range per launch for timeline tools
    switch (L.kind) {
      case LK_GRADNORM:
        rc = launch_gradnorm((const NormRange*)tab, (const int32_t*)(c->d_tables + L.aux0), L.grid, grads, hp.grad_dtype,
                             work + L.aux1, std::isfinite(hp.max_grad_norm) ? hp.max_grad_norm : 0.f,
                             (hp.flags & ADAPM_FLAG_CHECK_FINITE) ? 1 : 0, c->d_gscale, c->d_status, s);
        break;
      case LK_REDUCE_PARTIAL:
        rc = launch_reduce_partial((const ReduceJob*)tab, (const int32_t*)(c->d_tables + L.aux1), L.n_items, L.aux0, grads,
                                   work, hp.grad_dtype, c->d_status, s);
        break;
      case LK_REDUCE_FINAL:
      case LK_REDUCE_ROWS:
        rc = launch_reduce_final((const ReduceJob*)tab, L.n_items, L.aux0, (float*)state, work, hp.beta2, c->d_status,
                                 c->d_gscale, c->step_bytes < kChainedBytes, s);
        break;
      case LK_STREAM:
        if (fork) {
          ADAPM_CUDA(branch.fork());
          s = c->side_stream;
        }
        rc = launch_stream((const StreamBlk*)tab, (const int32_t*)(c->d_tables + L.aux0), L.grid, L.aux1 != 0, b, sc,
                           hp.grad_dtype, s);
        break;
      case LK_SPD_INVERSE:
        rc = launch_spd_inverse((const InverseJob*)tab, L.n_items, work, hp.precond_damping, c->d_status, s); break;
      case LK_GEMM:
        rc = launch_gemm((const GemmProb*)tab, L.n_items, L.grid, b, hp.grad_dtype, s); break;
      case LK_FP32_GRAM:
        rc = launch_fp32_gram((const Fp32Gram*)tab, (const int32_t*)(c->d_tables + L.aux0), L.grid, b, c->d_counters, s); break;
      case LK_FP32_REFIT:
        rc = launch_fp32_refit((const Fp32Refit*)tab, (const int32_t*)(c->d_tables + L.aux0), L.grid, b, hp.grad_dtype,
                               c->d_counters, s);
        break;
      case LK_APPLY_SIMT:
        rc = launch_apply_simt((const ApplyBlk*)tab, (const int32_t*)(c->d_tables + L.aux0), L.grid, b, sc, hp.grad_dtype, s);
        break;
      case LK_COMMIT:
        rc = launch_copy_ranges((const NormRange*)tab, (const int32_t*)(c->d_tables + L.aux0), L.grid, (float*)state,
                                work + c->ws_lr[c->final_lr_buf], c->d_status, s);
        break;
      default:
        rc = run_tensor_launch(c, L, b, sc, parity, s); break;
    }
    if (prof) nvtxRangePop();
    s = main_stream;
    if (rc != ADAPM_OK) return rc;
    ++li;
    if (prof) {
      c->prof_kinds.push_back((int32_t)L.kind);
      ADAPM_CUDA(cudaEventRecord(c->prof_events[li], s));
    }
  }
  ADAPM_CUDA(branch.join());
  c->last_step_launches = (int64_t)li;
  if (prof) c->prof_valid = 1;
  return ADAPM_OK;
}

extern "C" int adapm_step(adapm_ctx* c, void* params, const void* grads, void* state, int64_t t, adapm_stream stream) {
  if (!c || !params || !grads || !state || t < 1) return ADAPM_EINVAL;
  if ((uintptr_t)params % 256 || (uintptr_t)grads % 256 || (uintptr_t)state % 256) return ADAPM_EALIGN;
  if (c->work_floats > 0 && (!c->workspace || c->workspace_bytes < (size_t)c->work_floats * 4)) return ADAPM_ENOWORKSPACE;
  const int rc = enqueue_step(c, params, grads, state, t, (cudaStream_t)stream);
  // some launches may be missing: the bf16 copies of the factors no longer follow the step number, whatever comes next
  if (rc != ADAPM_OK) tensor_state_changed(c);
  return rc;
}

extern "C" int adapm_set_profiling(adapm_ctx* c, int32_t on) {
  if (!c) return ADAPM_EINVAL;
  if (on && c->prof_events.empty()) {
    c->prof_events.resize(c->program.size() + 1, nullptr);
    for (auto& e : c->prof_events) ADAPM_CUDA(cudaEventCreate(&e));
  }
  c->profiling = on ? 1 : 0;
  c->prof_valid = 0;
  return ADAPM_OK;
}

extern "C" int adapm_get_launch_times(adapm_ctx* c, float* ms, int32_t* kinds, int64_t capacity, int64_t* n_out) {
  if (!c || !n_out) return ADAPM_EINVAL;
  // the launches of the last profiled step (a step runs a subset of the program: see LaunchWhen)
  const size_t n = c->prof_valid ? c->prof_kinds.size() : c->program.size();
  *n_out = (int64_t)n;
  if (!ms && !kinds) return ADAPM_OK;
  if (capacity < (int64_t)n) return ADAPM_ERANGE;
  if (!c->prof_valid) return ADAPM_EINVAL;
  ADAPM_CUDA(cudaEventSynchronize(c->prof_events[n]));
  for (size_t i = 0; i < n; ++i) {
    if (ms) ADAPM_CUDA(cudaEventElapsedTime(&ms[i], c->prof_events[i], c->prof_events[i + 1]));
    if (kinds) kinds[i] = c->prof_kinds[i];
  }
  return ADAPM_OK;
}

extern "C" const char* adapm_launch_kind_name(int32_t kind) {
  switch (kind) {
    case LK_REDUCE_PARTIAL: return "reduce_partial";
    case LK_REDUCE_FINAL: return "reduce_final";
    case LK_REDUCE_ROWS: return "reduce_rows";
    case LK_GRADNORM: return "grad_norm";
    case LK_TC_COPY: return "tc_copy";
    case LK_TC_PAD: return "tc_pad";
    case LK_STREAM: return "stream_update";
    case LK_GEMM: return "gemm_simt";
    case LK_FP32_GRAM: return "fp32_gram";
    case LK_FP32_REFIT: return "fp32_refit";
    case LK_SPD_INVERSE: return "spd_inverse";
    case LK_APPLY_SIMT: return "apply_simt";
    case LK_COMMIT: return "commit_copy";
    case LK_TC_CONVERT: return "tc_convert";
    case LK_TC_CONVERT_WORK: return "tc_convert_work";
    case LK_TC_PANEL: return "tc_panel";
    case LK_TC_GRAM: return "tc_gram";
    case LK_TC_APPLY: return "tc_apply";
    default: return "unknown";
  }
}

extern "C" int adapm_get_status(adapm_ctx* c, adapm_stream stream, int32_t* status) {
  if (!c || !status) return ADAPM_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  int32_t h = 0;
  ADAPM_CUDA(cudaMemcpyAsync(&h, c->d_status, sizeof(h), cudaMemcpyDeviceToHost, s));
  ADAPM_CUDA(cudaStreamSynchronize(s));
  if (h != 0) {
    ADAPM_CUDA(cudaMemsetAsync(c->d_status, 0, sizeof(h), s));
    // steps issued while the word was set wrote nothing, so the bf16 copies of the factors no longer follow the
    // step numbers the host has counted: rebuild them from the state at the next step
    tensor_state_changed(c);
  }
  *status = h;
  return h == 0 ? ADAPM_OK : ADAPM_EDEVICE;
}

extern "C" size_t adapm_group_meansq_scratch_bytes(int64_t n_groups, int64_t group_elems) {
  if (n_groups <= 0 || group_elems <= 0) return 0;
  const int64_t cpg = (group_elems + kWarpUnitMax - 1) / kWarpUnitMax;
  return (size_t)round_up(n_groups * cpg, kStateAlign) * 4;
}

extern "C" int adapm_group_meansq(const void* g, int32_t grad_dtype, int64_t n_groups, int64_t group_elems, float* out,
                                  void* scratch, size_t scratch_bytes, adapm_stream stream) {
  if (!g || !out || !scratch || n_groups <= 0 || group_elems <= 0) return ADAPM_EINVAL;
  if (grad_dtype != ADAPM_GRAD_F32 && grad_dtype != ADAPM_GRAD_BF16) return ADAPM_EINVAL;
  if ((uintptr_t)g % 16 || (uintptr_t)scratch % 256) return ADAPM_EALIGN;
  if (scratch_bytes < adapm_group_meansq_scratch_bytes(n_groups, group_elems)) return ADAPM_ENOWORKSPACE;
  const int64_t cpg = (group_elems + kWarpUnitMax - 1) / kWarpUnitMax;
  if (cpg > INT32_MAX) return ADAPM_ERANGE;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = launch_meansq_partial(g, grad_dtype, n_groups, group_elems, (int)cpg, (float*)scratch, s);
  if (rc != ADAPM_OK) return rc;
  return launch_meansq_final((const float*)scratch, n_groups, group_elems, (int)cpg, out, s);
}

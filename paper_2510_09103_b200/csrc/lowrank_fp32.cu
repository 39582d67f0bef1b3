// Exact-fp32 refit and apply of the low-rank path on CUDA cores: fp32 gradients, ranks above what the
// tensor path takes, and every block of a caller who asks for it (ADAPM_PATH_SIMT).
//
// One pass of Algorithm 2 is two launches.  `gram` makes the r x r matrices
//   R R^T, R0 R^T, L^T L, L^T L0
// and `refit` the products with the gradient and, in the same CTA, the factor update
//   Q = g R^T,  L' = L - eta (L (R R^T) - b1 L0 (R0 R^T) - (1-b1) Q)      (and the same for R, column by column).
// Both cut long K loops into chunks when the set has too few tiles to fill the GPU; the CTA that comes
// last at a tile adds the partial products up, in the order of the chunks, and goes on with the tile.
// `apply` rebuilds m^c = cg g + c0 L0 R0 - c1 L R tile by tile and writes W.
//
// What bounds them: the FMA pipes (148 SMs x 128 lanes x 2 x 1.965 GHz = 74.4 TFLOP/s).  A thread holds
// RI x TN elements of a (16 RI) x (8 TN) tile and works on pairs along K with fma.rn.f32x2: both operands
// lie K-contiguous in shared memory, so a pair comes out of a 16-byte load ready for use, and 4 K cost a
// thread RI + TN loads for 2 RI TN packed FMAs.  TN is chosen so that a rank wastes at most seven columns.
#include "adapm_internal.h"
#include "device_math.cuh"

namespace adapm {

namespace {

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 fma_f32x2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 pack_f32x2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float sum_f32x2(f32x2 v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f.x + f.y;
}

// Four consecutive elements as fp32 (16- or 8-byte aligned), or one.
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const uint16_t* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}
__device__ __forceinline__ float load1(const float* p) { return *p; }
__device__ __forceinline__ float load1(const uint16_t* p) { return bf16_bits_to_float(*p); }

constexpr int kThreads = 128;            // 2 x 2 warps
constexpr int kAsyncStages = 3;          // of the loops that copy straight into shared memory
template <int RI_, int TN_, int BK_>
struct Tile {
  static constexpr int RI = RI_, TN = TN_, BK = BK_;
  static constexpr int kRows = 16 * RI, kCols = 8 * TN;
  // Row pitch in shared memory: BK + 4 makes the eight rows a warp reads at once start 4 banks apart, all different.
  static constexpr int P = BK + 4;
  static constexpr int kFloats = 2 * (kRows + kCols) * P;     // two stages, so that a stage costs one barrier
  static constexpr int kAsyncFloats = kAsyncStages * (kRows + kCols) * P;
};

// An operand: `n` rows (owners or columns of the tile, from i0) of K elements.  along_k: stored [n, K] with K
// contiguous, else [K, n].  A pitch that is a multiple of four elements means whole vectors (K or n is then a multiple
// of four too, whichever runs along memory).  ROWS: rows of the tile.
template <int ROWS, int BK, typename T>
struct Operand {
  const T* p;
  int64_t ld;
  int i0, n;
  bool along_k, vec;
  float scale;
  static constexpr int kVec = (ROWS * BK / 4 + kThreads - 1) / kThreads, kOne = (ROWS * BK + kThreads - 1) / kThreads;
  static constexpr int P = BK + 4;
  float v[kOne > 4 * kVec ? kOne : 4 * kVec];

  __device__ __forceinline__ void set(const T* p_, int64_t ld_, int i0_, int n_, bool along_k_, float scale_) {
    p = p_; ld = ld_; i0 = i0_; n = n_; along_k = along_k_; vec = (ld_ & 3) == 0; scale = scale_;
  }
  // (row, k) of this thread's q-th vector or element.  Along K, neighbouring lanes take neighbouring K.  Across K, the
  // lanes of a vector load take the K rows one by one (their scattered stores into shared memory then meet no bank
  // twice) and those of a scalar load neighbouring rows of the tile.
  __device__ __forceinline__ bool place(int q, int& row, int& k) const {
    const int id = threadIdx.x + kThreads * q;
    if (vec) {
      if (along_k) { row = id / (BK / 4); k = (id % (BK / 4)) * 4; } else { k = id % BK; row = (id / BK) * 4; }
      return (ROWS * BK / 4) % kThreads == 0 || id < ROWS * BK / 4;
    }
    if (along_k) { row = id / BK; k = id % BK; } else { row = id % ROWS; k = id / ROWS; }
    return (ROWS * BK) % kThreads == 0 || id < ROWS * BK;
  }
  __device__ __forceinline__ void fetch(int k0, int k_end) {
    int row, k;
    if (vec) {
#pragma unroll
      for (int q = 0; q < kVec; ++q) {
        const bool in = place(q, row, k);
        row += i0; k += k0;
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in && row < n && k < k_end) f = load4(p + (along_k ? (int64_t)row * ld + k : (int64_t)k * ld + row));
        v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < kOne; ++q) {
        const bool in = place(q, row, k);
        row += i0; k += k0;
        v[q] = (in && row < n && k < k_end) ? load1(p + (along_k ? (int64_t)row * ld + k : (int64_t)k * ld + row)) : 0.f;
      }
    }
  }
  __device__ __forceinline__ void store(float* s) const {
    int row, k;
    if (vec) {
#pragma unroll
      for (int q = 0; q < kVec; ++q) {
        if (!place(q, row, k)) continue;
        if (along_k) {
          *reinterpret_cast<float4*>(&s[row * P + k]) =
              make_float4(scale * v[4 * q], scale * v[4 * q + 1], scale * v[4 * q + 2], scale * v[4 * q + 3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) s[(row + e) * P + k] = scale * v[4 * q + e];
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < kOne; ++q)
        if (place(q, row, k)) s[row * P + k] = scale * v[q];
    }
  }
};

// 4 or 16 bytes from global into shared memory without a register in between; zeros if not `ok`.
__device__ __forceinline__ void copy4_async(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void copy16_async(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}

// The same operand, fp32 and unscaled, copied into the stages without registers in between.  A thread's elements of a stage
// are a fixed step apart, so that a stage costs it one address and one comparison each.
template <int ROWS, int BK>
struct AsyncOperand {
  static_assert(BK == 16 && kThreads == 128 && ROWS % 8 == 0, "places below");
  static constexpr int P = BK + 4;
  const float* p;             // of this thread's first element of the operand
  int64_t ld;
  int rows, k, dst;           // rows left from its first one, its first k of a stage, its place in a stage
  bool along_k, vec;

  __device__ __forceinline__ void set(const float* p_, int64_t ld_, int i0, int n, bool along_k_, int K) {
    const int tid = threadIdx.x;
    ld = ld_; along_k = along_k_; vec = along_k_ && (ld_ & 3) == 0;
    int row;
    if (vec) { row = tid / 4; k = tid % 4 * 4; }                     // whole vectors: rows 32 apart
    else if (along_k) { row = tid / 16; k = tid % 16; }              // rows 8 apart
    // across K, a warp takes eight rows, whole sectors, of four K (its words then lie in 32 banks); rows 8 apart
    else { row = tid % 8; k = tid / 8; }
    p = p_ + (along_k ? (int64_t)(i0 + row) * ld + k : (int64_t)k * ld + i0 + row);
    rows = n - i0 - row;
    if (rows <= 0 || k >= K) p = p_;            // (nothing is read, but the address stays inside the operand)
    dst = row * P + k;
  }
  __device__ __forceinline__ void copy(float* s, int k0, int k_end) const {
    const bool in = k0 + k < k_end;
    const float* const src = p + (along_k ? (int64_t)k0 : (int64_t)k0 * ld);
    if (vec) {
#pragma unroll
      for (int q = 0; q < (ROWS + 31) / 32; ++q) {
        if (ROWS % 32 != 0 && 32 * q + (int)threadIdx.x / 4 >= ROWS) continue;
        const bool ok = in && 32 * q < rows;
        copy16_async(s + dst + 32 * q * P, ok ? src + 32 * q * ld : p, ok);
      }
    } else {
      const int64_t step = along_k ? 8 * ld : 8;
#pragma unroll
      for (int q = 0; q < ROWS / 8; ++q) {
        const bool ok = in && 8 * q < rows;
        copy4_async(s + dst + 8 * q * P, ok ? src + q * step : p, ok);
      }
    }
  }
};

// Which elements of a tile this thread holds: rows row(i), columns col(c).
template <typename S>
struct Lane {
  int r0, c0;
  __device__ __forceinline__ Lane() {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    r0 = (warp >> 1) * 8 * S::RI + (lane & 7);
    c0 = (warp & 1) * 4 * S::TN + (lane >> 3);
  }
  __device__ __forceinline__ int row(int i) const { return r0 + 8 * i; }
  __device__ __forceinline__ int col(int c) const { return c0 + 4 * c; }
};

template <typename S>
using Acc = f32x2[S::RI][S::TN];        // each element as the sums over even and over odd K

template <typename S>
__device__ __forceinline__ void zero_acc(Acc<S>& acc) {
#pragma unroll
  for (int i = 0; i < S::RI; ++i)
#pragma unroll
    for (int c = 0; c < S::TN; ++c) acc[i][c] = 0ull;
}

// acc += X Y^T over one stage of K
template <typename S>
__device__ __forceinline__ void tile_stage(Acc<S>& acc, const float* xr, const float* yr) {
#pragma unroll
  for (int k = 0; k < S::BK; k += 4) {
    ulonglong2 y[S::TN];
#pragma unroll
    for (int c = 0; c < S::TN; ++c) y[c] = *reinterpret_cast<const ulonglong2*>(&yr[4 * c * S::P + k]);
#pragma unroll
    for (int i = 0; i < S::RI; ++i) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(&xr[8 * i * S::P + k]);
#pragma unroll
      for (int c = 0; c < S::TN; ++c) acc[i][c] = fma_f32x2(x.x, y[c].x, acc[i][c]);
#pragma unroll
      for (int c = 0; c < S::TN; ++c) acc[i][c] = fma_f32x2(x.y, y[c].y, acc[i][c]);
    }
  }
}

// acc += X Y^T over k in [k_begin, k_end), with kAsyncStages - 1 stages of copies in flight.
// Through registers, one stage ahead, the warps waited for their loads between bursts of FMAs (a third of their stalls) and held
// 21 to 24 registers for them.  Four refit launches of a step, us, registers -> copies: 6 layers of 768 x 3072 rank 8 769 -> 533,
// rank 38 1286 -> 977, rank 128 3581 -> 2884; rows of 2130 rank 38 1107 -> 834; the tiny set (rank 12) 107 -> 90.  Two CTAs of
// 248 registers per SM instead of three of 168: 569, 960, 3140.
template <typename S, typename X, typename Y>
__device__ __forceinline__ void tile_loop_async(Acc<S>& acc, const X& xop, const Y& yop, int k_begin, int k_end, float* sm) {
  const Lane<S> at;
  constexpr int kStage = (S::kRows + S::kCols) * S::P;
  const float* const xr = sm + at.r0 * S::P;
  const float* const yr = sm + (S::kRows + at.c0) * S::P;
  __syncthreads();                              // an earlier loop may still be reading the stages
  int fill = 0, use = 0, k_fill = k_begin;
  auto next = [&]() {
    if (k_fill < k_end) {
      xop.copy(sm + fill, k_fill, k_end);
      yop.copy(sm + fill + S::kRows * S::P, k_fill, k_end);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    k_fill += S::BK;
    fill = fill == (kAsyncStages - 1) * kStage ? 0 : fill + kStage;
  };
#pragma unroll
  for (int i = 0; i < kAsyncStages - 1; ++i) next();
#pragma unroll 1
  for (int k0 = k_begin; k0 < k_end; k0 += S::BK) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kAsyncStages - 2) : "memory");
    __syncthreads();                            // everyone's copies of this stage are here, and the one before it is free
    next();
    tile_stage<S>(acc, xr + use, yr + use);
    use = use == (kAsyncStages - 1) * kStage ? 0 : use + kStage;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// acc += X Y^T over k in [k_begin, k_end).
template <typename S, typename X, typename Y>
__device__ __forceinline__ void tile_loop(Acc<S>& acc, X& xop, Y& yop, int k_begin, int k_end, float* sm) {
  const Lane<S> at;
  constexpr int kStage = (S::kRows + S::kCols) * S::P;
  const float* const xr = sm + at.r0 * S::P;
  const float* const yr = sm + (S::kRows + at.c0) * S::P;
  int buf = 0;
  __syncthreads();                              // an earlier loop may still be reading the stages
  xop.fetch(k_begin, k_end);
  yop.fetch(k_begin, k_end);
#pragma unroll 1
  for (int k0 = k_begin; k0 < k_end; k0 += S::BK, buf ^= kStage) {
    xop.store(sm + buf);
    yop.store(sm + buf + S::kRows * S::P);
    __syncthreads();
    if (k0 + S::BK < k_end) {
      xop.fetch(k0 + S::BK, k_end);
      yop.fetch(k0 + S::BK, k_end);
    }
    tile_stage<S>(acc, xr + buf, yr + buf);
  }
}

// Leaves the tile's partial product in the workspace, [column][row] with row pitch S::kRows, and tells whether this
// CTA is the last of `splits` to do so.  The counter goes back to zero for the next launch.
template <typename S>
__device__ __forceinline__ bool put_partial(const Acc<S>& acc, float* part, int split, int splits, int32_t* counter) {
  __shared__ int last;
  const Lane<S> at;
  float* const p = part + (int64_t)split * (S::kRows * S::kCols);
#pragma unroll
  for (int c = 0; c < S::TN; ++c)
#pragma unroll
    for (int i = 0; i < S::RI; ++i) __stcg(p + at.col(c) * S::kRows + at.row(i), sum_f32x2(acc[i][c]));
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1) == splits - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  return true;
}

// acc = scale * the sum of the partial products, in the order of the chunks
template <typename S>
__device__ __forceinline__ void get_partials(Acc<S>& acc, const float* part, int splits, float scale) {
  const Lane<S> at;
  zero_acc<S>(acc);
#pragma unroll 1
  for (int s = 0; s < splits; ++s) {
    const float* const p = part + (int64_t)s * (S::kRows * S::kCols);
#pragma unroll
    for (int c = 0; c < S::TN; ++c)
#pragma unroll
      for (int i = 0; i < S::RI; ++i)
        acc[i][c] = pack_f32x2(sum_f32x2(acc[i][c]) + __ldcg(p + at.col(c) * S::kRows + at.row(i)), 0.f);
  }
#pragma unroll
  for (int c = 0; c < S::TN; ++c)
#pragma unroll
    for (int i = 0; i < S::RI; ++i) acc[i][c] = pack_f32x2(scale * sum_f32x2(acc[i][c]), 0.f);
}

// ---- r x r matrices --------------------------------------------------------------------------------------

template <typename S>
__device__ __forceinline__ void gram_tile(const Fp32Gram& G, int unit, const Bases& b, int32_t* counters, float* sm) {
  const int tile = unit / G.splits, split = unit - tile * G.splits;
  const int mt = tile / G.tiles_n, nt = tile - mt * G.tiles_n;
  const int k_begin = split * G.k_chunk, k_end = min(k_begin + G.k_chunk, G.K);
  Operand<S::kRows, S::BK, float> xop;
  Operand<S::kCols, S::BK, float> yop;
  xop.set(static_cast<const float*>(b.p[G.x_base]) + G.x_off, G.ld, mt * S::kRows, G.r, G.along_k, 1.f);
  yop.set(static_cast<const float*>(b.p[G.y_base]) + G.y_off, G.ld, nt * S::kCols, G.r, G.along_k, 1.f);
  Acc<S> acc;
  zero_acc<S>(acc);
  tile_loop<S>(acc, xop, yop, k_begin, k_end, sm);
  float* const work = static_cast<float*>(b.p[BASE_WORK]);
  if (G.splits > 1) {
    float* const part = work + G.part_off + (int64_t)tile * G.splits * (S::kRows * S::kCols);
    if (!put_partial<S>(acc, part, split, G.splits, counters + G.counter + tile)) return;
    get_partials<S>(acc, part, G.splits, 1.f);
  }
  const Lane<S> at;
#pragma unroll
  for (int c = 0; c < S::TN; ++c) {
    const int col = nt * S::kCols + at.col(c);
#pragma unroll
    for (int i = 0; i < S::RI; ++i) {
      const int row = mt * S::kRows + at.row(i);
      if (row < G.r && col < G.r) work[G.out_off + (int64_t)col * G.r + row] = sum_f32x2(acc[i][c]);
    }
  }
}

__global__ void __launch_bounds__(kThreads) fp32_gram_kernel(const Fp32Gram* __restrict__ tab,
                                                             const int32_t* __restrict__ unit_job, Bases b,
                                                             int32_t* __restrict__ counters) {
  __shared__ __align__(16) float sm[Tile<3, 5, 16>::kFloats];
  __shared__ Fp32Gram sG;
  if (threadIdx.x == 0) {
    sG = tab[unit_job[blockIdx.x]];
    if (*b.status != 0) sG.tn = 0;               // an earlier launch gave up: write nothing
  }
  __syncthreads();
  const int unit = (int)blockIdx.x - sG.first_unit;
  switch (sG.tn) {
    case 0: return;
    case 1: gram_tile<Tile<1, 1, 16>>(sG, unit, b, counters, sm); break;
    case 2: gram_tile<Tile<1, 2, 16>>(sG, unit, b, counters, sm); break;
    case 3: gram_tile<Tile<2, 3, 16>>(sG, unit, b, counters, sm); break;
    case 4: gram_tile<Tile<2, 4, 16>>(sG, unit, b, counters, sm); break;
    default: gram_tile<Tile<3, 5, 16>>(sG, unit, b, counters, sm); break;
  }
}

// ---- product with the gradient and factor update ---------------------------------------------------------

template <typename S, typename GT>
__device__ __forceinline__ void refit_tile(const Fp32Refit& U, int unit, const Bases& b, int32_t* counters, float* sm) {
  const int tile = unit / U.splits, split = unit - tile * U.splits;
  const int mt = tile / U.tiles_n, nt = tile - mt * U.tiles_n;
  const int k_begin = split * U.k_chunk, k_end = min(k_begin + U.k_chunk, U.K);
  const int r = U.r;
  const float* const work = static_cast<const float*>(b.p[BASE_WORK]);
  const float a1 = (1.f - U.b1) * (b.gscale ? __ldg(b.gscale) : 1.f);
  Acc<S> acc;
  zero_acc<S>(acc);
  Operand<S::kCols, S::BK, float> yop;
  if constexpr (sizeof(GT) == 4) {
    AsyncOperand<S::kRows, S::BK> xa;
    AsyncOperand<S::kCols, S::BK> ya;
    xa.set(static_cast<const float*>(b.p[BASE_GRADS]) + U.g_off, U.ldg, mt * S::kRows, U.owners, U.along_k, U.K);
    ya.set(static_cast<const float*>(b.p[U.y_base]) + U.y_off, U.along_k ? U.K : r, nt * S::kCols, r, U.along_k, U.K);
    tile_loop_async<S>(acc, xa, ya, k_begin, k_end, sm);
  } else {
    Operand<S::kRows, S::BK, GT> xop;
    xop.set(static_cast<const GT*>(b.p[BASE_GRADS]) + U.g_off, U.ldg, mt * S::kRows, U.owners, U.along_k, 1.f);
    yop.set(static_cast<const float*>(b.p[U.y_base]) + U.y_off, U.along_k ? U.K : r, nt * S::kCols, r, U.along_k, 1.f);
    tile_loop<S>(acc, xop, yop, k_begin, k_end, sm);
  }
  if (U.splits > 1) {
    float* const part = const_cast<float*>(work) + U.part_off + (int64_t)tile * U.splits * (S::kRows * S::kCols);
    if (!put_partial<S>(acc, part, split, U.splits, counters + U.counter + tile)) return;
    get_partials<S>(acc, part, U.splits, -a1);
  } else {
#pragma unroll
    for (int c = 0; c < S::TN; ++c)
#pragma unroll
      for (int i = 0; i < S::RI; ++i) acc[i][c] = pack_f32x2(-a1 * sum_f32x2(acc[i][c]), 0.f);
  }
  // acc = -(1-b1) Q; the derivative's other two terms on top of it.  In the first pass of a step the current factors
  // are the previous ones and one product does for both.
  const float* const cur = static_cast<const float*>(b.p[U.cur_base]) + U.cur_off;
  const int64_t ldf = U.along_k ? r : U.owners;
  Operand<S::kRows, S::BK, float> fop;
  fop.set(cur, ldf, mt * S::kRows, U.owners, U.along_k, U.gb_off >= 0 ? 1.f : 1.f - U.b1);
  yop.set(work + U.ga_off, r, nt * S::kCols, r, true, 1.f);
  tile_loop<S>(acc, fop, yop, 0, r, sm);
  if (U.gb_off >= 0) {
    fop.p = static_cast<const float*>(b.p[U.prev_base]) + U.prev_off;
    fop.scale = -U.b1;
    yop.p = work + U.gb_off;
    tile_loop<S>(acc, fop, yop, 0, r, sm);
  }
  const Lane<S> at;
  float* const out = static_cast<float*>(b.p[U.out_base]) + U.out_off;
  float* const save = U.save_off >= 0 ? static_cast<float*>(b.p[BASE_WORK]) + U.save_off : nullptr;
  const int64_t so = U.along_k ? r : 1, sk = U.along_k ? 1 : U.owners;     // strides over owners and over the rank
#pragma unroll
  for (int c = 0; c < S::TN; ++c) {
    const int col = nt * S::kCols + at.col(c);
#pragma unroll
    for (int i = 0; i < S::RI; ++i) {
      const int row = mt * S::kRows + at.row(i);
      if (row < U.owners && col < r) {
        const int64_t o = so * row + sk * col;
        const float old = __ldg(cur + o);
        out[o] = old - U.eta * sum_f32x2(acc[i][c]);
        if (save) save[o] = old;
      }
    }
  }
}

template <typename GT>
__global__ void __launch_bounds__(kThreads, 3) fp32_refit_kernel(const Fp32Refit* __restrict__ tab,
                                                                 const int32_t* __restrict__ unit_job, Bases b,
                                                                 int32_t* __restrict__ counters) {
  __shared__ __align__(16) float sm[sizeof(GT) == 4 ? Tile<8, 5, 16>::kAsyncFloats : Tile<8, 5, 16>::kFloats];
  __shared__ Fp32Refit sU;
  if (threadIdx.x == 0) {
    sU = tab[unit_job[blockIdx.x]];
    if (*b.status != 0) sU.tn = 0;               // an earlier launch gave up: write nothing
  }
  __syncthreads();
  const int unit = (int)blockIdx.x - sU.first_unit;
  switch (sU.tn) {
    case 0: return;
    case 1: refit_tile<Tile<8, 1, 16>, GT>(sU, unit, b, counters, sm); break;
    case 2: refit_tile<Tile<8, 2, 16>, GT>(sU, unit, b, counters, sm); break;
    case 3: refit_tile<Tile<8, 3, 16>, GT>(sU, unit, b, counters, sm); break;
    case 4: refit_tile<Tile<8, 4, 16>, GT>(sU, unit, b, counters, sm); break;
    default: refit_tile<Tile<8, 5, 16>, GT>(sU, unit, b, counters, sm); break;
  }
}

// ---- apply ----------------------------------------------------------------------------------------------------

// A 64 x 64 tile of D = c0 L0 R0 - c1 L R, put into shared memory (the stages' own room) so that the elementwise part
// runs along the rows of W: a warp takes a row at a time, two adjacent columns per lane where the pitch allows it,
// whatever the alignment of the rows.  What that part will read is asked into L2 before the products.
// Against a 4 x 4 tile per thread of 256 threads that writes from registers (59 M elements in blocks of 1024 x 2730, fp32
// gradients, us): rank 8 400|490 with row groups and 374|569 with a v per element, rank 51 842|785 and 828|846, rank 128
// 1399|1220 and 1381|1275, rank 290 3034|2448: ahead where the memory sets the pace, behind on the products of larger
// ranks (128 registers, issue slots half used, the FMA pipes busy 35 % of the time), and its sums, kept in two halves,
// are a little closer to 64 bits.
template <typename GT>
__global__ void __launch_bounds__(kThreads, 4) fp32_apply_kernel(const ApplyBlk* __restrict__ tab,
                                                                 const int32_t* __restrict__ tile_blk, Bases b,
                                                                 StepScalars sc) {
  using S = Tile<4, 8, 8>;
  static_assert(S::kRows == kApplyTile && S::kCols == kApplyTile, "apply tile");
  constexpr int DP = kApplyTile + 4;
  __shared__ __align__(16) union { float tile[S::kFloats]; float d[kApplyTile][DP]; } sm;
  __shared__ ApplyBlk sA;
  __shared__ int skip;
  if (threadIdx.x == 0) {
    sA = tab[tile_blk[blockIdx.x]];
    skip = *b.status != 0;
  }
  __syncthreads();
  if (skip) return;
  const ApplyBlk& A = sA;
  const int tile = (int)((int64_t)blockIdx.x - A.first_tile);
  const int i0 = (tile / A.tiles_n) * kApplyTile, j0 = (tile % A.tiles_n) * kApplyTile;
  const int m = A.rows, n = A.cols, r = A.rank;
  const bool grouped = A.v_mode == ADAPM_V_BLOCKMEAN;
  float* __restrict__ W = static_cast<float*>(b.p[BASE_PARAMS]) + A.off;
  const GT* __restrict__ G = static_cast<const GT*>(b.p[BASE_GRADS]) + A.off;
  float* __restrict__ V = static_cast<float*>(b.p[BASE_STATE]) + A.v_off;
  {
    const int i = i0 + ((int)threadIdx.x >> 1), c = j0 + 32 * ((int)threadIdx.x & 1);
    if (i < m && c < n) {
      const int64_t o = (int64_t)i * n + c;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(W + o));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(G + o));
      if (!grouped) asm volatile("prefetch.global.L2 [%0];" ::"l"(V + o));
    }
  }

  Acc<S> acc;
  zero_acc<S>(acc);
  {
    Operand<S::kRows, S::BK, float> xop;
    Operand<S::kCols, S::BK, float> yop;
    xop.set(static_cast<const float*>(b.p[A.l0_base]) + A.l0_off, r, i0, m, true, sc.c0);
    yop.set(static_cast<const float*>(b.p[A.r0_base]) + A.r0_off, n, j0, n, false, 1.f);
    tile_loop<S>(acc, xop, yop, 0, r, sm.tile);
    if (sc.c1 != 0.f) {
      xop.p = static_cast<const float*>(b.p[A.l1_base]) + A.l1_off; xop.scale = -sc.c1;
      yop.p = static_cast<const float*>(b.p[A.r1_base]) + A.r1_off;
      tile_loop<S>(acc, xop, yop, 0, r, sm.tile);
    }
  }
  __syncthreads();
  {
    const Lane<S> at;
#pragma unroll
    for (int i = 0; i < S::RI; ++i)
#pragma unroll
      for (int c = 0; c < S::TN; ++c) sm.d[at.row(i)][at.col(c)] = sum_f32x2(acc[i][c]);
  }
  __syncthreads();

  const float gs = b.gscale ? __ldg(b.gscale) : 1.f;
  const float lr_s = sc.lr * A.lr_scale;
  uint16_t* __restrict__ shadow = b.shadow ? b.shadow + A.off : nullptr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool pairs = (n & 1) == 0;
  constexpr int kInFlight = 8;                            // rows a warp has in flight
  // this lane's columns: 2 lane + {0, 1}, or lane + {0, 32} where rows start at odd elements
  const int c0 = pairs ? 2 * lane : lane, c1 = pairs ? 2 * lane + 1 : lane + 32;
  const bool ok0 = j0 + c0 < n, ok1 = j0 + c1 < n;
#pragma unroll 1
  for (int q0 = warp * kInFlight; q0 < kApplyTile; q0 += 4 * kInFlight) {
    float g[kInFlight][2], w[kInFlight][2], v[kInFlight][2];
#pragma unroll
    for (int e = 0; e < kInFlight; ++e) {
      const int i = i0 + q0 + e;
      const int64_t o = (int64_t)i * n + j0;
      g[e][0] = g[e][1] = w[e][0] = w[e][1] = v[e][0] = v[e][1] = 0.f;
      if (i >= m) continue;
      if (pairs) {
        if (ok0) {
          if (sizeof(GT) == 2) {
            const uint32_t x = *reinterpret_cast<const uint32_t*>(G + o + c0);
            g[e][0] = __uint_as_float(x << 16); g[e][1] = __uint_as_float(x & 0xffff0000u);
          } else {
            const float2 x = *reinterpret_cast<const float2*>(G + o + c0);
            g[e][0] = x.x; g[e][1] = x.y;
          }
          const float2 x = *reinterpret_cast<const float2*>(W + o + c0);
          w[e][0] = x.x; w[e][1] = x.y;
          if (!grouped) { const float2 y = *reinterpret_cast<const float2*>(V + o + c0); v[e][0] = y.x; v[e][1] = y.y; }
        }
      } else {
        if (ok0) { g[e][0] = load1(G + o + c0); w[e][0] = W[o + c0]; if (!grouped) v[e][0] = V[o + c0]; }
        if (ok1) { g[e][1] = load1(G + o + c1); w[e][1] = W[o + c1]; if (!grouped) v[e][1] = V[o + c1]; }
      }
      if (grouped) v[e][0] = v[e][1] = V[i / A.v_group_rows];
    }
#pragma unroll
    for (int e = 0; e < kInFlight; ++e) {
      const int i = i0 + q0 + e;
      if (i >= m) continue;
      const int64_t o = (int64_t)i * n + j0;
      float vn[2], wn[2];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const float gx = gs * g[e][x];
        const float mc = sc.cg * gx + sm.d[q0 + e][x ? c1 : c0];
        vn[x] = grouped ? v[e][x] : sc.beta2 * v[e][x] + (1.f - sc.beta2) * (gx * gx);
        wn[x] = adapm_param_update(w[e][x], mc, vn[x], sc, lr_s, A.wd);
      }
      if (pairs) {
        if (ok0) {
          *reinterpret_cast<float2*>(W + o + c0) = make_float2(wn[0], wn[1]);
          if (!grouped) *reinterpret_cast<float2*>(V + o + c0) = make_float2(vn[0], vn[1]);
          if (shadow) *reinterpret_cast<uint32_t*>(shadow + o + c0) = pack_bf16x2(wn[0], wn[1]);
        }
      } else {
        if (ok0) {
          W[o + c0] = wn[0];
          if (!grouped) V[o + c0] = vn[0];
          if (shadow) shadow[o + c0] = (uint16_t)(pack_bf16x2(wn[0], 0.f) & 0xffffu);
        }
        if (ok1) {
          W[o + c1] = wn[1];
          if (!grouped) V[o + c1] = vn[1];
          if (shadow) shadow[o + c1] = (uint16_t)(pack_bf16x2(wn[1], 0.f) & 0xffffu);
        }
      }
    }
  }
}

}  // namespace

#define ADAPM_LAUNCH_CHECK()                         \
  do {                                               \
    cudaError_t e__ = cudaGetLastError();            \
    if (e__ != cudaSuccess) {                        \
      set_cuda_error(e__, __func__);                 \
      return ADAPM_ECUDA;                            \
    }                                                \
  } while (0)

int launch_fp32_gram(const Fp32Gram* d_tab, const int32_t* d_unit_job, int64_t n_units, const Bases& b, int32_t* counters,
                     cudaStream_t s) {
  if (n_units <= 0) return ADAPM_OK;
  fp32_gram_kernel<<<(unsigned)n_units, kThreads, 0, s>>>(d_tab, d_unit_job, b, counters);
  ADAPM_LAUNCH_CHECK();
  return ADAPM_OK;
}

int launch_fp32_refit(const Fp32Refit* d_tab, const int32_t* d_unit_job, int64_t n_units, const Bases& b, int grad_dtype,
                      int32_t* counters, cudaStream_t s) {
  if (n_units <= 0) return ADAPM_OK;
  if (grad_dtype == ADAPM_GRAD_BF16)
    fp32_refit_kernel<uint16_t><<<(unsigned)n_units, kThreads, 0, s>>>(d_tab, d_unit_job, b, counters);
  else
    fp32_refit_kernel<float><<<(unsigned)n_units, kThreads, 0, s>>>(d_tab, d_unit_job, b, counters);
  ADAPM_LAUNCH_CHECK();
  return ADAPM_OK;
}

int launch_apply_simt(const ApplyBlk* d_tab, const int32_t* d_tile_blk, int64_t n_tiles, const Bases& b,
                      const StepScalars& sc, int grad_dtype, cudaStream_t s) {
  if (n_tiles <= 0) return ADAPM_OK;
  if (grad_dtype == ADAPM_GRAD_BF16)
    fp32_apply_kernel<uint16_t><<<(unsigned)n_tiles, kThreads, 0, s>>>(d_tab, d_tile_blk, b, sc);
  else
    fp32_apply_kernel<float><<<(unsigned)n_tiles, kThreads, 0, s>>>(d_tab, d_tile_blk, b, sc);
  ADAPM_LAUNCH_CHECK();
  return ADAPM_OK;
}

}  // namespace adapm

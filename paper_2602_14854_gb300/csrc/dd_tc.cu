// Tensor-core (tcgen05) form of the dense Galerkin contractions of the step, for the
// DD_TF32 and DD_BF16 precisions.
//
// The factors stay FP64 in memory.  Tiles are staged in shared memory by TMA
// (cp.async.bulk.tensor), split in shared memory into a high and a low part of the
// tensor-core type (x = hi + lo to ~2^-22 |x| in TF32, ~2^-17 in BF16), and multiplied as
// hi*hi + hi*lo + lo*hi with FP32 accumulation in tensor memory: the error-compensated
// splitting of Ootomo and Yokota (2022, "Recovering single precision accuracy from Tensor
// Cores while surpassing the FP32 theoretical peak performance") for TF32 and of Henry,
// Tang and Heinecke (2019, "Leveraging the bfloat16 artificial intelligence datatype for
// higher-precision computations") for BF16, so each product carries FP32-level error
// instead of the type's own 2^-11 / 2^-8.  Results are written back in FP64.
//
//   k_tc_tall  Y = alpha A M (or Y += alpha A M): A tall (rows x ni), M small (ni x nc),
//              per subdomain; 128-row tiles, M = 128 MMAs, double-buffered TMA loads.
//   k_tc_gram  partial Galerkin Grams D_p = A_p^T diag(w_p) B over a chunk of rows, two
//              A operands stacked along M = 128 per CTA, written to the chunk partials that
//              k_reduce sums in FP64 (the same layout as the FP64 Gram kernels).
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <climits>

#include "dd_internal.cuh"
#include "dd_launch.h"
#include "dd_tc.cuh"

namespace dd {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
// looked up once by tc_init; solvers may be created from several host threads
std::atomic<EncodeTiledFn> g_encode{nullptr};

// Tensor map of a row-major FP64 array (rows x ld) whose boxes are box_rows x ld
// (ld even: rows start on 16-byte boundaries).  Rows outside the array read as zero.
bool make_map(CUtensorMap* m, const double* ptr, int ld, long rows, int box_rows) {
  const EncodeTiledFn encode = g_encode.load(std::memory_order_acquire);
  if (!encode || (ld & 1) || ld > 256 || rows < 1) return false;
  cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 8};
  cuuint32_t box[2] = {(cuuint32_t)ld, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<double*>(ptr), dims, strides,
                box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

constexpr uint32_t kWait = 1u << 21;   // polls of a bounded mbarrier wait (about a second)

// Split f into the operand byte offset `off` of the hi (base) and lo (base + lo_off)
// planes.
template <int FMT>
__device__ __forceinline__ void put_split(uint8_t* base, uint32_t lo_off, uint32_t off, float f) {
  if (FMT == tc::FMT_TF32) {
    uint32_t h, l;
    tc::split_tf32(f, &h, &l);
    *reinterpret_cast<uint32_t*>(base + off) = h;
    *reinterpret_cast<uint32_t*>(base + lo_off + off) = l;
  } else {
    uint16_t h, l;
    tc::split_bf16(f, &h, &l);
    *reinterpret_cast<uint16_t*>(base + off) = h;
    *reinterpret_cast<uint16_t*>(base + lo_off + off) = l;
  }
}

// hi*hi + hi*lo + lo*hi over nslab K-slabs of 32 bytes (accumulating into d from `acc`)
template <int FMT>
__device__ __forceinline__ void mma_split(uint32_t d, uint32_t a_hi, uint32_t a_lo, uint32_t b_hi,
                                          uint32_t b_lo, int nslab, uint32_t sbo_a,
                                          uint32_t sbo_b, uint32_t id, uint32_t acc) {
  const uint32_t as[3] = {a_hi, a_lo, a_hi}, bs[3] = {b_lo, b_hi, b_hi};
#pragma unroll
  for (int p = 0; p < 3; ++p)
    for (int s = 0; s < nslab; ++s) {
      const uint64_t ad = tc::sdesc(as[p] + 256 * s, 128, sbo_a);
      const uint64_t bd = tc::sdesc(bs[p] + 256 * s, 128, sbo_b);
      if (FMT == tc::FMT_TF32) tc::mma_tf32(d, ad, bd, id, acc);
      else tc::mma_bf16(d, ad, bd, id, acc);
      acc = 1;
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------
// tall x small:  Y = alpha A M  (or Y += alpha A M)
// ---------------------------------------------------------------------------------------
struct TcTall {
  Geo g;
  int spatial;
  int lda;                          // leading dimension of A (its tensor map's box width)
  const int* ninner; int ninner_fix;
  const double* Bm; int bsmall;     // M: small slot bsmall of smbase, or Bm + k RC^2 (bsmall < 0)
  const double* smbase;
  const int* ncols; int ncols_fix;
  double* Y; int ldy;
  double alpha; int accumulate;     // accumulate: Y += alpha A M on columns < nc only
  int tps;                          // 128-row tiles per subdomain (of the largest)
  unsigned* status;
  const double* A;                  // A itself (the kernels that load it without a tensor map)
  long nrows;                       // rows of A (the Ozaki kernel's prefetch)
  int zfill;                        // columns nc .. ldy - 1 of Y set to zero (the Ozaki kernel; k_tc_*
                                    // load whole rows)
  int mtrans;                       // M read transposed (the Ozaki kernel)
  const double* rowscale;           // accumulate: Y_r += rowscale_r (A M)_r (the Ozaki kernel; null: 1)
};

#define TT_ROWS 128
#define TT_THREADS 256
#define TT_STAGE (TT_ROWS * DD_MAXC * 8)          // 64 KiB: FP64 tile, then its hi / lo planes
#define TT_BPLANE (DD_MAXC * DD_MAXC * 4)         // 16 KiB: one plane of M^T
size_t tc_tall_smem() { return 1024 + 2 * TT_STAGE + 2 * TT_BPLANE; }

// CTA b takes a contiguous range of the (subdomain, 128-row tile) pairs; the tile after
// the current one is loaded by TMA while the current one is split and multiplied.  Eight
// warps split; warp w reads TMEM lanes 32 (w % 4).. and the 16-column groups of parity w / 4.
template <int FMT>
__global__ void __launch_bounds__(TT_THREADS, 1) k_tc_tall(const __grid_constant__ CUtensorMap mapA,
                                                           TcTall a) {
  extern __shared__ uint8_t raw_tt[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_tt) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* stage[2] = {base, base + TT_STAGE};
  uint8_t* bop = base + 2 * TT_STAGE;
  __shared__ uint64_t bar_tma[2], bar_mma;
  __shared__ uint32_t tmem_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int RC = a.g.RC, es = FMT == tc::FMT_TF32 ? 4 : 2, kq = 32 / es;
  const long ntot = (long)a.g.nsub * a.tps;
  const long f0 = blockIdx.x * ntot / gridDim.x, f1 = (blockIdx.x + 1) * ntot / gridDim.x;
  auto rows_of = [&](int k) { return a.spatial ? a.g.N[k] : a.g.n; };
  auto valid = [&](long f) { return (int)(f % a.tps) * TT_ROWS < rows_of((int)(f / a.tps)); };
  auto next_valid = [&](long f) {
    while (f < f1 && !valid(f)) ++f;
    return f;
  };
  auto row0 = [&](long f) {
    const int k = (int)(f / a.tps);
    return (a.spatial ? (long)a.g.rowoff[k] : (long)k * a.g.n) + (long)(f % a.tps) * TT_ROWS;
  };
  long f = next_valid(f0);
  if (f >= f1) return;                                // nothing here (before any setup)
  if (tid == 0) {
    tc::mbar_init(&bar_tma[0], 1);
    tc::mbar_init(&bar_tma[1], 1);
    tc::mbar_init(&bar_mma, 1);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(&tmem_s, 64);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_s;
  const uint32_t box_bytes = (uint32_t)TT_ROWS * a.lda * 8;
  if (tid == 0) {
    tc::mbar_arrive_expect_tx(&bar_tma[0], box_bytes);
    tc::tma_load_2d(stage[0], &mapA, 0, (int)row0(f), &bar_tma[0]);
  }
  int kB = -1, it = 0;
  bool alive = true;
  for (; f < f1 && alive; f = next_valid(f + 1), ++it) {
    const int buf = it & 1;
    const long fn = next_valid(f + 1);
    if (tid == 0 && fn < f1) {                         // the other buffer's MMA completed
      tc::mbar_arrive_expect_tx(&bar_tma[buf ^ 1], box_bytes);
      tc::tma_load_2d(stage[buf ^ 1], &mapA, 0, (int)row0(fn), &bar_tma[buf ^ 1]);
    }
    const int k = (int)(f / a.tps), rows = rows_of(k);
    const int r0 = (int)(f % a.tps) * TT_ROWS;
    const int ni = a.ninner ? a.ninner[k] : a.ninner_fix;
    const int nc = a.ncols ? a.ncols[k] : a.ncols_fix;
    const int Kp = ni <= kq ? kq : (ni + kq - 1) / kq * kq;
    const int KB = Kp * es;
    const int N = nc <= 16 ? 16 : (nc + 15) / 16 * 16;
    count_work(a.g, KS_TC_TALL, 2.0 * min(TT_ROWS, rows - r0) * ni * nc);
    if (k != kB) {                                     // M^T as the B operand (N x Kp)
      const double* Mk = a.bsmall >= 0 ? a.smbase + ((long)k * NSMALL + a.bsmall) * RC * RC
                                       : a.Bm + (long)k * RC * RC;
      for (int e = tid; e < N * Kp; e += TT_THREADS) {
        const int n = e / Kp, kk = e - n * Kp;
        const float x = (n < nc && kk < ni) ? tc::f64_to_f32(Mk[kk * RC + n]) : 0.f;
        put_split<FMT>(bop, TT_BPLANE, tc::op_off(n, kk * es, KB), x);
      }
      kB = k;
    }
    const bool got = tc::mbar_wait(&bar_tma[buf], (it >> 1) & 1, kWait);
    // split the FP64 tile in place: every value read before any plane is written
    const double* st = reinterpret_cast<const double*>(stage[buf]);
    float v[DD_MAXC / 2];
#pragma unroll
    for (int j = 0; j < DD_MAXC / 2; ++j) {
      v[j] = 0.f;
      const int e = tid + TT_THREADS * j;
      if (e < TT_ROWS * Kp) {
        const int r = e / Kp, kk = e - r * Kp;
        if (got && kk < ni && r0 + r < rows) v[j] = tc::f64_to_f32(st[r * a.lda + kk]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < DD_MAXC / 2; ++j) {
      const int e = tid + TT_THREADS * j;
      if (e < TT_ROWS * Kp) {
        const int r = e / Kp, kk = e - r * Kp;
        put_split<FMT>(stage[buf], TT_STAGE / 2, tc::op_off(r, kk * es, KB), v[j]);
      }
    }
    tc::fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const uint32_t sa = tc::smem_u32(stage[buf]), sb = tc::smem_u32(bop);
      mma_split<FMT>(tmem, sa, sa + TT_STAGE / 2, sb, sb + TT_BPLANE, Kp / kq, 8 * KB, 8 * KB,
                     tc::idesc(FMT, 128, N), 0);
      tc::mma_commit(&bar_mma);
    }
    __syncwarp();
    const bool done = tc::mbar_wait(&bar_mma, it & 1, kWait);
    tc::fence_after_sync();
    const int r = r0 + (warp & 3) * 32 + lane;
    double* y = a.Y + (row0(f) - r0 + r) * a.ldy;
    for (int c0 = (warp >> 2) * 16; c0 < N; c0 += 32) {
      float d[16];
      tc::tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + c0, d);
      if (r < rows) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int c = c0 + j;
          const double x = tc::f32_to_f64(d[j]);
          if (c < nc) y[c] = a.accumulate ? y[c] + a.alpha * x : (a.alpha == 1.0 ? x : a.alpha * x);
          else if (!a.accumulate && c < a.ldy) y[c] = 0.0;
        }
      }
    }
    if (r < rows && !a.accumulate && warp < 4)
      for (int c = N; c < a.ldy; ++c) y[c] = 0.0;
    tc::fence_before_sync();
    alive = __syncthreads_and(got && done) != 0;        // block-uniform
    if (!alive && tid == 0) atomicOr(a.status, (unsigned)ST_TIMEOUT);
  }
  if (!alive && tid == 0) {                           // bounded waits for work in flight
    tc::mbar_wait(&bar_mma, (it - 1) & 1, kWait);
    if (f < f1) tc::mbar_wait(&bar_tma[it & 1], (it >> 1) & 1, kWait);
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 64);
}

// ---------------------------------------------------------------------------------------
// Galerkin Grams:  D_p = A_p^T diag(w_p) B  over a chunk of rows
// ---------------------------------------------------------------------------------------
#define TG_ROWS 32                                  // rows (the MMA's K) per stage
#define TG_THREADS 256
#define TG_STAGE (TG_ROWS * DD_MAXC * 8)            // 16 KiB FP64 tile
#define TG_APLANE (128 * TG_ROWS * 4)               // 16 KiB: one plane of the stacked A^T
#define TG_BPLANE (DD_MAXC * TG_ROWS * 4)           // 8 KiB: one plane of B^T
#define TG_OPS (2 * TG_APLANE + 2 * TG_BPLANE)      // one set of operands (hi and lo)
size_t tc_gram_smem() { return 1024 + 2 * 3 * TG_STAGE + 2 * TG_OPS; }

// One CTA per (row chunk, subdomain, source pair).  Stages of 32 rows: the FP64 tiles of
// the next stage load (TMA) while the current stage is split; the operands alternate
// between two buffers, each guarded by its own MMA barrier, so the split of stage s + 1
// overlaps the products of stage s.
template <int FMT>
__global__ void __launch_bounds__(TG_THREADS, 1) k_tc_gram(const __grid_constant__ CUtensorMap mapB,
                                                           const __grid_constant__ CUtensorMap mapA0,
                                                           const __grid_constant__ CUtensorMap mapA1,
                                                           TcGram a) {
  extern __shared__ uint8_t raw_tg[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_tg) + 1023) &
                                             ~uintptr_t(1023));
  // stage tiles: [buf][0] B, [buf][1] A0, [buf][2] A1; operands: [buf] A hi, A lo, B hi, B lo
  auto tile = [&](int b, int t) { return base + (b * 3 + t) * TG_STAGE; };
  auto ops = [&](int b) { return base + 6 * TG_STAGE + b * TG_OPS; };
  __shared__ uint64_t bar_tma[2], bar_mma[2];
  __shared__ uint32_t tmem_s;
  __shared__ float wgt[2][TG_ROWS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k = blockIdx.y, c = blockIdx.x, grp = blockIdx.z, RC = a.g.RC;
  const int rows = a.spatial ? a.g.N[k] : a.g.n;
  const long rb = a.spatial ? (long)a.g.rowoff[k] : (long)k * a.g.n;
  const int ch = (rows + a.nchunk - 1) / a.nchunk;
  const int i0 = min(rows, c * ch), i1 = min(rows, i0 + ch);
  const int nb = a.bcnt ? a.bcnt[k] : a.bfix;
  const int N = nb <= 16 ? 16 : (nb + 15) / 16 * 16;
  const int es = FMT == tc::FMT_TF32 ? 4 : 2, KB = TG_ROWS * es;
  // the two sources of this CTA: column counts, row bases (own or a neighbour's rows)
  int ma[2], src[2], sh[2];
  long arb[2];
  bool from_b[2];
  for (int h = 0; h < 2; ++h) {
    src[h] = 2 * grp + h;
    ma[h] = 0;
    arb[h] = 0;
    sh[h] = 0;
    from_b[h] = false;
    if (src[h] >= a.nsrc) continue;
    const TcGramSrc& s = a.src[src[h]];
    int kk = k;
    if (s.nbside >= 0) kk = a.g.nb[k * 4 + 2 * a.axis + s.nbside];
    if (kk < 0) continue;
    ma[h] = s.cnt ? s.cnt[kk] : s.fix;
    arb[h] = a.spatial ? (long)a.g.rowoff[kk] : (long)kk * a.g.n;
    from_b[h] = s.same_as_b;
    sh[h] = s.shift ? (a.axis == 0 ? 1 : a.g.nxk[k]) : 0;
  }
  // output: every source's RC x RC partial block, written whole (zeros outside the
  // product) so that k_reduce can sum the chunk partials
  auto out_of = [&](int p) {
    return a.part + (((long)k * a.nchunk + c) * a.nblk + a.src[p].blk) * RC * RC;
  };
  const bool any = (ma[0] > 0 || ma[1] > 0) && nb > 0 && i1 > i0;
  if (!any) {
    for (int h = 0; h < 2; ++h)
      if (src[h] < a.nsrc) {
        double* o = out_of(src[h]);
        for (int e = tid; e < RC * RC; e += blockDim.x) o[e] = 0.0;
      }
    return;
  }
  count_work(a.g, KS_TC_GRAM, 2.0 * (i1 - i0) * nb * (ma[0] + ma[1]));
  if (tid == 0) {
    tc::mbar_init(&bar_tma[0], 1);
    tc::mbar_init(&bar_tma[1], 1);
    tc::mbar_init(&bar_mma[0], 1);
    tc::mbar_init(&bar_mma[1], 1);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(&tmem_s, 128);        // two FP32 accumulators of 64 columns
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_s;
  const double* om = a.axis == 0 ? a.ox : a.oy;
  const int nst = (i1 - i0 + TG_ROWS - 1) / TG_ROWS;
  auto issue = [&](int s) {                            // thread 0: the tiles of stage s
    const int b = s & 1, r0 = i0 + s * TG_ROWS;
    uint32_t bytes = (uint32_t)TG_ROWS * a.ldb * 8;
    for (int h = 0; h < 2; ++h)
      if (ma[h] > 0 && !from_b[h]) bytes += (uint32_t)TG_ROWS * a.src[src[h]].ld * 8;
    tc::mbar_arrive_expect_tx(&bar_tma[b], bytes);
    tc::tma_load_2d(tile(b, 0), &mapB, 0, (int)(rb + r0), &bar_tma[b]);
    if (ma[0] > 0 && !from_b[0])                       // a shifted source reads rows earlier
      tc::tma_load_2d(tile(b, 1), &mapA0, 0, (int)(arb[0] + r0 - sh[0]), &bar_tma[b]);
    if (ma[1] > 0 && !from_b[1])
      tc::tma_load_2d(tile(b, 2), &mapA1, 0, (int)(arb[1] + r0 - sh[1]), &bar_tma[b]);
  };
  // Every stage's products go to a fresh FP32 accumulator in TMEM (two, alternating) and
  // are added into double-float sums (TwoSum) once the stage completes: the FP32 rounding
  // then spans one 32-row stage, not the whole chunk.  Thread: row m = 32 (w % 4) + lane of
  // D, the 16-column groups of parity w / 4.
  float2 acc[2][16];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[q][j] = make_float2(0.f, 0.f);
  bool ok = true;
  auto readout = [&](int j) {                          // stage j's products into acc
    const bool d = tc::mbar_wait(&bar_mma[j & 1], (j >> 1) & 1, kWait);
    ok = ok && d;
    tc::fence_after_sync();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c0 = (warp >> 2) * 16 + 32 * q;
      if (c0 < N) {
        float v[16];
        tc::tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((j & 1) * 64 + c0), v);
#pragma unroll
        for (int t = 0; t < 16; ++t) acc[q][t] = df_add(acc[q][t], make_float2(v[t], 0.f));
      }
    }
    tc::fence_before_sync();
  };
  if (tid == 0) issue(0);
  int s = 0;
  for (; s < nst && ok; ++s) {
    const int b = s & 1, r0 = i0 + s * TG_ROWS, nr = min(TG_ROWS, i1 - r0);
    if (tid == 0 && s + 1 < nst) issue(s + 1);         // its buffers' stage s - 1 is split
    // (the operands of buffer b were read by stage s - 2, read out in the last iteration)
    const bool got = tc::mbar_wait(&bar_tma[b], (s >> 1) & 1, kWait);
    // row weights of the two sources (FP32)
    if (tid < 2 * TG_ROWS) {
      const int h = tid / TG_ROWS, r = tid % TG_ROWS, row = r0 + r;
      float wv = 1.f;
      if (src[h] < a.nsrc && r < nr) {
        const TcGramSrc& so = a.src[src[h]];
        const long long ob = __double_as_longlong(om[min(row, a.g.n - 1)]);
        const bool ng = ob < 0 && ob != (long long)0x8000000000000000ull;
        switch (so.wsel) {
          case W_OMEGA: wv = tc::f64_to_f32(om[row]); break;
          case W_NEG: wv = ng ? 1.f : 0.f; break;
          case W_NONNEG: wv = ng ? 0.f : 1.f; break;
          case W_OMEGA_POS: wv = ng ? 0.f : tc::f64_to_f32(om[row]); break;
          case W_OMEGA_NEG: wv = ng ? tc::f64_to_f32(om[row]) : 0.f; break;
          case W_ROW: wv = tc::f64_to_f32(so.wrow[rb + row]); break;
          default: break;
        }
      }
      wgt[h][r] = wv;
    }
    __syncthreads();
    uint8_t* op = ops(b);
    // B^T (N x 32 rows) and the stacked, weighted A^T (128 x 32 rows)
    const double* sB = reinterpret_cast<const double*>(tile(b, 0));
    for (int e = tid; e < N * TG_ROWS; e += TG_THREADS) {
      const int n = e / TG_ROWS, r = e - n * TG_ROWS;
      const float x = (got && n < nb && r < nr) ? tc::f64_to_f32(sB[r * a.ldb + n]) : 0.f;
      put_split<FMT>(op + 2 * TG_APLANE, TG_BPLANE, tc::op_off(n, r * es, KB), x);
    }
    for (int e = tid; e < 128 * TG_ROWS; e += TG_THREADS) {
      const int m = e / TG_ROWS, r = e - m * TG_ROWS, h = m >> 6, i = m & 63;
      float x = 0.f;
      if (got && i < ma[h] && r < nr) {
        const double* sA = reinterpret_cast<const double*>(from_b[h] ? tile(b, 0) : tile(b, 1 + h));
        const int ld = from_b[h] ? a.ldb : a.src[src[h]].ld;
        if (sh[h]) {
          // the row minus the row one cell earlier along the axis (0 before a line start),
          // formed in FP64 before the split: the Gram is then the small difference E = I - T
          // itself, not T ~ I, whose FP32-level error would dominate I - T
          const int row = r0 + r;
          const int pos = a.axis == 0 ? row % a.g.nxk[k] : row / a.g.nxk[k];
          x = tc::f64_to_f32(sB[r * a.ldb + i] - (pos == 0 ? 0.0 : sA[r * ld + i]));
        } else {
          x = tc::f64_to_f32(sA[r * ld + i]);
        }
        x *= wgt[h][r];
      }
      put_split<FMT>(op, TG_APLANE, tc::op_off(m, r * es, KB), x);
    }
    tc::fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const uint32_t sa = tc::smem_u32(op), sb = sa + 2 * TG_APLANE;
      mma_split<FMT>(tmem + (uint32_t)(b * 64), sa, sa + TG_APLANE, sb, sb + TG_BPLANE,
                     TG_ROWS / (32 / es), 8 * KB, 8 * KB, tc::idesc(FMT, 128, N), 0u);
      tc::mma_commit(&bar_mma[b]);
    }
    if (s >= 1) readout(s - 1);                        // overlaps the products of stage s
    ok = __syncthreads_and(ok && got) != 0;            // block-uniform
  }
  if (s >= 1) readout(s - 1);
  ok = __syncthreads_and(ok) != 0;
  if (!ok) {
    if (tid == 0) {
      atomicOr(a.status, (unsigned)ST_TIMEOUT);
      if (s < nst) tc::mbar_wait(&bar_tma[s & 1], (s >> 1) & 1, kWait);   // load in flight
    }
  }
  // epilogue: the double-float sums of row m (source h = m / 64, column i = m % 64 of A_h)
  {
    const int m = (warp & 3) * 32 + lane, h = m >> 6, i = m & 63;
    double* o = src[h] < a.nsrc ? out_of(src[h]) : nullptr;
    const bool tr = o && a.src[src[h]].transpose;
    if (o && i < RC) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c0 = (warp >> 2) * 16 + 32 * q;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int cc = c0 + j;
          if (cc >= RC) continue;
          const double x = (ok && c0 < N && i < ma[h] && cc < nb)
                               ? tc::f32_to_f64(acc[q][j].x) + tc::f32_to_f64(acc[q][j].y)
                               : 0.0;
          if (tr) o[cc * RC + i] = x;
          else o[i * RC + cc] = x;
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 128);
}

// ---------------------------------------------------------------------------------------
// FP64-accurate tall x small products on the BF16 tensor cores (Ozaki scheme)
// ---------------------------------------------------------------------------------------
// Y = A M with the error-free splitting of Ozaki, Ogita, Oishi and Rump (2012, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication
// and its applications").  The rows of M are equalised by powers of two, M' = diag(2^-mu) M
// with mu_k the exponent of row k's largest entry, the inverse scale folded into the columns
// of A (A' = A diag(2^mu)); each row r of A' gets the power-of-two bound 2^e_r and each column
// n of M' the bound 2^f_n, and every value becomes a fixed-point integer with 56 fraction bits
// relative to its bound (truncated), split into 7 balanced base-256 digits (the top digit is at
// most 256, the others at most 128 in magnitude: exact in BF16).  Digit products of
// orders s, t go to the TMEM accumulator of g = s + t (pairs with g <= 6; 28 of 49): with at
// most 64 terms of at most 7 pairs every partial sum is an integer below 2^24, so the FP32
// accumulation is exact.  The epilogue combines the seven sums in 64-bit integers and builds
// the FP64 result from bits.  Error: a few units of 2^-56 of max_k |A'[r][k]| max_k
// |M'[k][n]| per entry (the FP64 rounding of each product is 2^-53 of the product).  No FP64
// arithmetic runs in the kernel.
//
#define OZ_DIG 7
#define OZ_NONE (-(1 << 20))                 // exponent of an all-zero row / column
#define OZ_BAD (1 << 21)                     // of one with a NaN or an infinity (above -OZ_NONE)

// biased FP64 exponent of x (0 for zero and subnormals)
__device__ __forceinline__ int f64_bexp(double x) {
  return (int)((unsigned)(__double_as_longlong(x) >> 52) & 0x7ffu);
}
// the BF16 digits of two values packed in one word (each digit has <= 8 significant bits:
// its BF16 is the top half of its FP32)
__device__ __forceinline__ uint32_t oz_pack(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
// ---- roles of a CTA of k_oz_tall --------------------------------------------------------
// One CTA per SM, its warps specialised, handing 128-row tiles over through mbarriers:
//   16 converter warps  8 rows of A each -> registers -> digit planes of A' in shared memory,
//                       M's digit planes once per subdomain;
//   1 MMA warp          one thread issues the digit products of a tile, 16 columns of Y at a
//                       time, into one of four TMEM buffers (7 accumulators of 16 columns);
//   8 epilogue warps    TMEM -> registers (the buffer is free again at once) -> FP64 -> Y.
// Conversion (integer and FP32 issue), the tensor cores and the epilogue (integer issue) of
// different tiles overlap; before, all 16 worker warps converted a tile's digits, then all of
// them ran the previous tile's epilogue, with CTA-wide barriers between, and issued on 40% of
// the cycles.  262144 x 40 x 40 (64 subdomains, lda 60), per launch: 166 us before, 106 now.
//
// Digit planes of A: rows of 2 KP bytes (KP = the inner dimension rounded up to 16), plane s
// of a stage at s APL; two stages while KP <= 48, one for KP = 64.  M: for column chunk c of
// 16, plane u: rows (7 c + u) 16 + n, so the planes a product needs are adjacent along N: A's
// plane s times M's planes 0 .. 6 - s is one MMA of N = 16 (7 - s) into the accumulators
// s .. 6 of the buffer.
#define OT_CONV 16
#define OT_EPI 8
#define OT_THREADS ((OT_CONV + OT_EPI + 1) * 32)
#define OT_NB 4                              // TMEM buffers of 128 columns (7 x 16 in use)
// tiles whose row and column exponents are kept: a converter is at most 5 tiles ahead of the
// epilogue (2 stages, and the MMAs of the tile before them wait for one of 4 TMEM buffers)
#define OT_RING 8
#define OT_AHEAD 3                           // tiles of A on their way into L2 ahead of the converters

static uint32_t ot_mpl(int KP) { return (uint32_t)OZ_DIG * DD_MAXC * 2 * KP; }
static uint32_t ot_apl(int KP) { return (uint32_t)OZ_DIG * TT_ROWS * 2 * KP; }
// dynamic shared memory for inner dimensions up to lda (<= 64): the largest plan among them
static size_t ot_smem(int lda) {
  size_t most = 0;
  for (int KP = 16; KP <= (lda + 15) / 16 * 16; KP += 16)
    most = std::max(most, (size_t)ot_mpl(KP) + (KP <= 48 ? 2 : 1) * (size_t)ot_apl(KP));
  return most + 128;
}

// Converter warps only: barrier, and barrier returning whether all of them pass true
__device__ __forceinline__ void ot_conv_sync() { asm volatile("bar.sync 2, %0;" ::"n"(OT_CONV * 32) : "memory"); }
__device__ __forceinline__ bool ot_conv_all(bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 2, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((int)p), "n"(OT_CONV * 32)
      : "memory");
  return r != 0;
}

// The 7 digits of T = trunc(x 2^(56 - e)) (|x| < 2^e, so |T| < 2^56), T = sum_s d_s 2^(48 - 8 s),
// of two values, packed: word s holds the BF16 digits s of x0 (low half) and x1.  By integer
// operations: with the mantissa left-aligned (implicit bit at bit 63) T is one right shift;
// adding 128 at each of the six low byte positions makes every low byte of
// V = T + 0x808080808080 equal to d_s + 128 with the borrows and carries of a balanced
// representation (d_s in [-128, 127] for s >= 1, and d_0 = V >> 48 in [-256, 256]).  Signed T
// needs nothing more: the identity is modular.  A low byte b = d + 128 becomes d in BF16 by two
// logic operations and one packed subtraction: 128 + (b & 127) is 0x4300 | (b & 127), and what
// has to come off it is 128 where bit 7 of b is set, else 256: 0x4300 | (~b & 128).
__device__ __forceinline__ void oz_digits2(double x0, int e0, double x1, int e1, uint32_t* w) {
  uint32_t vl[2], vh[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(i ? x1 : x0);
    const unsigned hi = (unsigned)(u >> 32);
    const int E = (int)((hi >> 20) & 0x7ffu);
    const int sh = 1030 + (i ? e1 : e0) - E;                 // >= 8
    const unsigned long long m = (u << 11) | 0x8000000000000000ull;
    long long T = (E != 0 && sh < 64) ? (long long)(m >> sh) : 0ll;
    if (hi >> 31) T = -T;
    const unsigned long long V = (unsigned long long)T + 0x808080808080ull;
    vl[i] = (unsigned)V;
    vh[i] = (unsigned)(V >> 32);
  }
#pragma unroll
  for (int s = 1; s < OZ_DIG; ++s) {
    const int b = (6 - s) & 3;                               // byte of the word
    const uint32_t sel = (uint32_t)(b | (b << 4) | ((4 + b) << 8) | ((4 + b) << 12));
    const uint32_t p = s <= 2 ? __byte_perm(vh[0], vh[1], sel) : __byte_perm(vl[0], vl[1], sel);
    const uint32_t X = (p & 0x007f007fu) | 0x43004300u, Y = (~p & 0x00800080u) | 0x43004300u;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(w[s]) : "r"(X), "r"(Y));
  }
  w[0] = oz_pack(__int_as_float(0x4B400000 + ((int)vh[0] >> 16)) - 12582912.0f,
                 __int_as_float(0x4B400000 + ((int)vh[1] >> 16)) - 12582912.0f);
}

// starts bringing rows [row, row + n) of the row-major A (rows x lda, lda even) into L2, none
// past the last; one thread
__device__ __forceinline__ void prefetch_rows(const double* A, long lda, long row, long n, long rows) {
  n = min(n, rows - row);
  if (n > 0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(A + row * lda),
                 "r"((unsigned)(n * lda * 8))
                 : "memory");
}

// 4 consecutive FP32 columns of this warp's 32 lanes, without the wait
__device__ __forceinline__ void oz_tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// The value sum_g D_g 2^(-8 g) of the seven accumulators (exact integers as FP32) as an
// integer in units of 2^-40.  |D_0|, |D_1| <= 2^22 for at most 64 terms (digit 0 is at most
// 256, the others 128 in magnitude): their integer is in the low bits of D + 1.5 2^23.  The
// others take the conversion instruction.
__device__ __forceinline__ long long oz_combine(const uint32_t* D, int stride) {
  auto f = [&](int g) { return __uint_as_float(D[g * stride]); };
  const int d0 = __float_as_int(f(0) + 12582912.0f) - 0x4B400000;
  const int d1 = __float_as_int(f(1) + 12582912.0f) - 0x4B400000;
  const int d2 = __float2int_rn(f(2)), d3 = __float2int_rn(f(3)), d4 = __float2int_rn(f(4));
  const int d5 = __float2int_rn(f(5)), d6 = __float2int_rn(f(6));
  long long J = (long long)(d5 + (d6 >> 8));
  J += (long long)d4 * 256;
  J += (long long)d3 * 65536;
  J += (long long)d2 * 16777216;
  J += (long long)((unsigned long long)(unsigned)(d1 + d0 * 256) << 32);
  return J;
}
// J 2^sc as an FP64 (rounded to nearest), by integer operations; |J| < 2^62
__device__ __forceinline__ double oz_round(long long J, int sc) {
  const unsigned sg = (unsigned)(J >> 63) & 0x80000000u;
  const unsigned long long u = (unsigned long long)(J < 0 ? -J : J);
  const int lz = __clzll((long long)u);
  // mantissa left-aligned at bit 62 (bit 63 free for the carry of the rounding)
  const unsigned long long n = (u << (lz & 63)) >> 1;
  const unsigned long long r = n + 0x1ffull + ((n >> 10) & 1ull);
  const int be = 1023 + 63 - lz + sc;                 // exponent of the leading bit
  unsigned long long b = (r >> 10) + ((unsigned long long)(unsigned)(be - 1) << 52);
  if (be <= 0) b = 0ull;
  if (be >= 2047) b = 0x7ff0000000000000ull;
  if (u == 0ull) return 0.0;
  return __longlong_as_double((long long)(b | ((unsigned long long)sg << 32)));
}

// 8 rows of a tile, KP = 8 C columns: lane (rho, q) loads row `row`, columns 8 c + 2 q and
// 8 c + 2 q + 1.  The loads are unconditional (columns past the array's read its last pair; what is
// not wanted is dropped where it is used): the compiler waits for a load under its own condition
// before the next one.
template <int C>
__device__ __forceinline__ void ot_load(double2 (&d)[8], const double* row, int q, int lda) {
#pragma unroll
  for (int c = 0; c < C; ++c)
    d[c] = __ldg(reinterpret_cast<const double2*>(row + min(8 * c + 2 * q, lda - 2)));
}
__device__ __forceinline__ void ot_load(double2 (&d)[8], const double* row, int q, int lda, int KP) {
  if (KP <= 16) ot_load<2>(d, row, q, lda);
  else if (KP <= 32) ot_load<4>(d, row, q, lda);
  else if (KP <= 48) ot_load<6>(d, row, q, lda);
  else ot_load<8>(d, row, q, lda);
}
// Their digit planes (row r of the stage asl, planes APL apart) and the row bound (lanes q = 0).
// A row with a NaN or an infinity has the bound OZ_BAD and no digits (as fixed-point numbers they
// would come out as large finite values); the epilogue makes its products NaN.
// One body per KP: with the column count a run-time bound every pair of values sat in a branch
// of its own and waited for the one before (7 clocks per instruction and warp; the converters
// took 12000 clocks per tile).
template <int C>
__device__ __forceinline__ void ot_convert(const double2 (&x)[8], const int* mexp, int ni, int q, int r,
                                           uint8_t* asl, uint32_t APL, int* rexp) {
  int2 me[C];
  int mx = OZ_NONE, top = 0;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int kk = 8 * c + 2 * q;
    me[c] = *reinterpret_cast<const int2*>(mexp + kk);   // OZ_NONE past ni and for zero rows of M
    const int E0 = kk < ni ? f64_bexp(x[c].x) : 0, E1 = kk + 1 < ni ? f64_bexp(x[c].y) : 0;
    top = max(top, max(E0, E1));
    mx = max(mx, E0 && me[c].x != OZ_NONE ? E0 - 1022 + me[c].x : OZ_NONE);
    mx = max(mx, E1 && me[c].y != OZ_NONE ? E1 - 1022 + me[c].y : OZ_NONE);
  }
  if (top == 0x7ff) mx = OZ_BAD;
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
  if (q == 0) rexp[r] = mx;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    uint32_t w[OZ_DIG];
    oz_digits2(me[c].x != OZ_NONE ? x[c].x : 0.0, mx - me[c].x, me[c].y != OZ_NONE ? x[c].y : 0.0,
               mx - me[c].y, w);
    uint8_t* p = asl + tc::op_off(r, (8 * c + 2 * q) * 2, 16 * C);
#pragma unroll
    for (int d = 0; d < OZ_DIG; ++d) *reinterpret_cast<uint32_t*>(p + d * APL) = w[d];
  }
}

struct OtShape {
  int rows, ni, nc, KP, nch;
  long row0;                        // first row of the subdomain
};

__global__ void __launch_bounds__(OT_THREADS, 1) k_oz_tall(TcTall a) {
  extern __shared__ uint8_t raw_oz[];
  uint8_t* msl = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_oz) + 127) &
                                            ~uintptr_t(127));
  __shared__ uint64_t full[2], empty[2], tfull[OT_NB], tempty[OT_NB], meta[OT_RING];
  __shared__ uint32_t tmem_s;
  __shared__ __align__(8) int mexp[DD_MAXC];
  __shared__ int fnow[DD_MAXC], red[OT_CONV / 2][DD_MAXC];
  __shared__ int rexp[OT_RING][TT_ROWS], fexp[OT_RING][DD_MAXC];
  __shared__ int part_w[32], range[4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int RC = a.g.RC, nsub = a.g.nsub;
  auto rows_of = [&](int k) { return a.spatial ? a.g.N[k] : a.g.n; };
  auto shape = [&](int k) {
    OtShape s;
    s.rows = rows_of(k);
    s.ni = a.ninner ? a.ninner[k] : a.ninner_fix;
    s.nc = a.ncols ? a.ncols[k] : a.ncols_fix;
    s.KP = max(16, (s.ni + 15) & ~15);
    s.nch = max(1, (s.nc + 15) >> 4);
    s.row0 = a.spatial ? (long)a.g.rowoff[k] : (long)k * a.g.n;
    return s;
  };
  // ---- this CTA's tiles: a contiguous range of (subdomain, tile) pairs of about equal cost,
  // the tiles of subdomain k costing about 2 + KP / 16 + column chunks each (a conversion, an
  // epilogue and the hand-over; subdomains of a batch differ in rank)
  auto cost = [&](const OtShape& s) { return 2 + (s.KP >> 4) + s.nch; };
  {
    const int per = (nsub + 511) / 512, ka = min(nsub, tid * per), kb = tid < 512 ? min(nsub, ka + per) : ka;
    int w = 0;
    for (int k = ka; k < kb; ++k) {
      const OtShape s = shape(k);
      w += ((s.rows + TT_ROWS - 1) / TT_ROWS) * cost(s);
    }
    int inc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) part_w[warp] = inc;
    if (tid < 4) range[tid] = tid & 1 ? 0 : nsub;
    __syncthreads();
    int total = 0, before = 0;
    for (int i = 0; i < 16; ++i) {
      if (i < warp) before += part_w[i];
      total += part_w[i];
    }
    const int lo = before + inc - w;                    // weight before subdomain ka
    for (int side = 0; side < 2; ++side) {
      // the first tile that starts at or after this side's share of the total
      const int x = (int)((long)(blockIdx.x + side) * total / gridDim.x);
      if (w > 0 && x >= lo && x < lo + w) {
        int at = lo;
        for (int k = ka; k < kb; ++k) {
          const OtShape s = shape(k);
          const int nt = (s.rows + TT_ROWS - 1) / TT_ROWS, wk = nt * cost(s);
          if (x < at + wk) {
            range[2 * side] = k;
            range[2 * side + 1] = (x - at + cost(s) - 1) / cost(s);
            break;
          }
          at += wk;
        }
      }
    }
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) { tc::mbar_init(&full[i], OT_CONV); tc::mbar_init(&empty[i], 1); }
    for (int i = 0; i < OT_NB; ++i) { tc::mbar_init(&tfull[i], 1); tc::mbar_init(&tempty[i], OT_EPI); }
    for (int i = 0; i < OT_RING; ++i) tc::mbar_init(&meta[i], OT_CONV);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(&tmem_s, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_s;
  const int k1 = range[2], j1 = range[3];
  // walk over this CTA's tiles: (k, j), normalised to an existing tile or the end
  auto settle = [&](int& k, int& j) {
    while (k < nsub && j * TT_ROWS >= rows_of(k)) { ++k; j = 0; }
    return k < k1 || (k == k1 && j < j1);
  };
  bool alive = true;

  if (warp < OT_CONV) {
    // ------------------------------------------------------------------ converters
    const int rho = lane & 7, q = lane >> 3;
    int k = range[0], j = range[1], kcur = -1, it = 0;
    unsigned used[2] = {0, 0};
    bool more = settle(k, j);
    OtShape s = shape(min(k, nsub - 1));
    const int r = 8 * warp + rho;                          // this lane's row of every tile
    double2 x[8];
    // (rows past the subdomain's read its last one; their results are not written)
    auto load = [&](const OtShape& t, int jt) {
      ot_load(x, a.A + (t.row0 + min(jt * TT_ROWS + r, t.rows - 1)) * a.lda, q, a.lda, t.KP);
    };
    if (more && tid == 0)
      prefetch_rows(a.A, a.lda, s.row0 + (long)j * TT_ROWS, OT_AHEAD * TT_ROWS, a.nrows);
    if (more) load(s, j);
    uint8_t* asl0 = msl;
    uint32_t APL = 0;
    while (more) {
      const int nst = s.KP <= 48 ? 2 : 1;
      if (k != kcur) {
        // ---- M's digit planes, once per subdomain.  The MMAs that read the old ones (and the
        // stages, used as scratch here) are complete first; all converters agree on going on.
        for (int b = 0; b < 2; ++b)
          if (used[b] && alive) alive = tc::mbar_wait(&empty[b], (used[b] - 1) & 1, kWait);
        alive = ot_conv_all(alive);
        if (!alive) break;
        kcur = k;
        APL = TT_ROWS * 2 * s.KP;
        asl0 = msl + (size_t)s.nch * 16 * OZ_DIG * 2 * s.KP;
        const double* Mk = a.bsmall >= 0 ? a.smbase + ((long)k * NSMALL + a.bsmall) * RC * RC
                                         : a.Bm + (long)k * RC * RC;
        double* Ms = reinterpret_cast<double*>(asl0);     // [kk][DD_MAXC]
#pragma unroll
        for (int i = 0; i < DD_MAXC * DD_MAXC / (OT_CONV * 32); ++i) {
          const int e = tid + OT_CONV * 32 * i, kk = e >> 6, n = e & (DD_MAXC - 1);
          if (kk < s.KP)
            Ms[e] = (kk < s.ni && n < s.nc)
                        ? __ldg(Mk + (a.mtrans ? (long)n * RC + kk : (long)kk * RC + n)) : 0.0;
        }
        ot_conv_sync();
        for (int kk = warp; kk < s.KP; kk += OT_CONV) {    // mu_k: warp per row
          const int E0 = f64_bexp(Ms[kk * DD_MAXC + lane]), E1 = f64_bexp(Ms[kk * DD_MAXC + lane + 32]);
          const int mx = __reduce_max_sync(0xffffffffu, max(E0 && E0 != 0x7ff ? E0 - 1022 : OZ_NONE,
                                                            E1 && E1 != 0x7ff ? E1 - 1022 : OZ_NONE));
          if (lane == 0) mexp[kk] = mx;
        }
        ot_conv_sync();
        {                                                  // f_n: OT_CONV / 2 threads per column
          const int n = tid & (DD_MAXC - 1), p = tid >> 6;
          int mx = OZ_NONE;
          for (int kk = p; kk < s.ni; kk += OT_CONV / 2) {
            const int E = f64_bexp(Ms[kk * DD_MAXC + n]);
            if (E) mx = max(mx, E != 0x7ff ? E - 1022 - mexp[kk] : OZ_BAD);
          }
          red[p][n] = mx;
        }
        ot_conv_sync();
        if (tid < DD_MAXC) {
          int mx = red[0][tid];
#pragma unroll
          for (int p = 1; p < OT_CONV / 2; ++p) mx = max(mx, red[p][tid]);
          fnow[tid] = mx;
        }
        ot_conv_sync();
        // digits of M'[kk][n] relative to 2^f_n, two adjacent kk per lane, 8 n x 4 pairs per warp
        const int kb = s.KP >> 3;
        for (int blk = warp; blk < s.nch * 2 * kb; blk += OT_CONV) {
          const int n = (blk / kb) * 8 + rho, kk = ((blk % kb) * 4 + q) * 2;
          uint32_t w[OZ_DIG];
          oz_digits2(Ms[kk * DD_MAXC + n], fnow[n] + mexp[kk], Ms[(kk + 1) * DD_MAXC + n],
                     fnow[n] + mexp[kk + 1], w);
          const int r0 = (n >> 4) * (16 * OZ_DIG) + (n & 15);
#pragma unroll
          for (int u = 0; u < OZ_DIG; ++u)
            *reinterpret_cast<uint32_t*>(msl + tc::op_off(r0 + 16 * u, kk * 2, 2 * s.KP)) = w[u];
        }
        tc::fence_async_smem();
        ot_conv_sync();                                    // Ms is read before the digits below
      }
      if (a.g.work) count_work(a.g, KS_OZ_TALL, 2.0 * min(TT_ROWS, s.rows - j * TT_ROWS) * s.ni * s.nc);
      const int b = nst == 2 ? it & 1 : 0, slot = it & (OT_RING - 1);
      // (the rows of consecutive tiles follow each other in memory, across subdomains too)
      if (tid == 0) prefetch_rows(a.A, a.lda, s.row0 + (long)(j + OT_AHEAD) * TT_ROWS, TT_ROWS, a.nrows);
      if (used[b] && alive) alive = tc::mbar_wait(&empty[b], (used[b] - 1) & 1, kWait);
      // the next tile
      int kn = k, jn = j + 1;
      more = settle(kn, jn);
      const OtShape sn = (more && kn != k) ? shape(kn) : s;
      uint8_t* asl = asl0 + (size_t)b * OZ_DIG * APL;
      if (tid < DD_MAXC) fexp[slot][tid] = fnow[tid];
      if (s.KP <= 16) ot_convert<2>(x, mexp, s.ni, q, r, asl, APL, rexp[slot]);
      else if (s.KP <= 32) ot_convert<4>(x, mexp, s.ni, q, r, asl, APL, rexp[slot]);
      else if (s.KP <= 48) ot_convert<6>(x, mexp, s.ni, q, r, asl, APL, rexp[slot]);
      else ot_convert<8>(x, mexp, s.ni, q, r, asl, APL, rexp[slot]);
      if (more) load(sn, jn);                              // under the fence and the next wait
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        tc::mbar_arrive(&meta[slot]);
        tc::mbar_arrive(&full[b]);
      }
      ++used[b];
      ++it;
      k = kn;
      j = jn;
      s = sn;
    }
  } else if (warp < OT_CONV + OT_EPI) {
    // ------------------------------------------------------------------ epilogue
    const int q4 = warp & 3, half = (warp - OT_CONV) >> 2, m = q4 * 32 + lane;
    int k = range[0], j = range[1], kcur = -1, it = 0, qc = 0;
    OtShape s{};
    const bool wide = (a.ldy & 3) == 0;
    while (alive && settle(k, j)) {
      if (k != kcur) { s = shape(k); kcur = k; }
      const int slot = it & (OT_RING - 1), r = j * TT_ROWS + m;
      const bool in = r < s.rows;
      double* yr = a.Y + (s.row0 + r) * a.ldy;
      alive = __all_sync(0xffffffffu, tc::mbar_wait(&meta[slot], (it / OT_RING) & 1, kWait));
      const int er = rexp[slot][m];
      const double rs = (a.accumulate && a.rowscale && in) ? a.rowscale[s.row0 + r] : 1.0;
      for (int c = 0; c < s.nch && alive; ++c, ++qc) {
        const int buf = qc & (OT_NB - 1);
        int c0 = 16 * c + 8 * half;
        alive = __all_sync(0xffffffffu, tc::mbar_wait(&tfull[buf], (qc / OT_NB) & 1, kWait));
        if (!alive) break;
        tc::fence_after_sync();
        const int lim = a.zfill ? a.ldy : s.nc;            // columns written
#pragma unroll 1
        for (int h = 0; h < 2; ++h, c0 += 4) {
          __syncwarp();                                    // (lanes past the last row came early)
          uint32_t D[OZ_DIG][4];
#pragma unroll
          for (int g = 0; g < OZ_DIG; ++g)
            oz_tmem_ld4(tmem + ((uint32_t)(q4 * 32) << 16) +
                            (uint32_t)(128 * buf + 16 * g + 8 * half + 4 * h), D[g]);
          double2 o[2];
          if (a.accumulate && in) {                        // Y's entries
#pragma unroll
            for (int i = 0; i < 2; ++i)
              o[i] = *reinterpret_cast<const double2*>(yr + min(c0 + 2 * i, a.ldy - 2));
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int g = 0; g < OZ_DIG; ++g)
#pragma unroll
            for (int i = 0; i < 4; ++i) asm volatile("" : "+r"(D[g][i]));
          if (h == 1) {                                    // the buffer is free again
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&tempty[buf]);
          }
          double v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int sc = er + fexp[slot][c0 + i] - 56;
            v[i] = oz_round(oz_combine(&D[0][i], 4), sc);
            if (sc > OZ_BAD / 4) v[i] = __longlong_as_double(0x7ff8000000000000ll);
            if (c0 + i >= s.nc) v[i] = 0.0;
          }
          if (!in) continue;
          double* yp = yr + c0;
          if (a.accumulate) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              v[2 * i] = fma(rs, v[2 * i], o[i].x);
              v[2 * i + 1] = fma(rs, v[2 * i + 1], o[i].y);
            }
          }
          if (c0 + 4 <= lim) {
            if (wide) {
              asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(yp), "d"(v[0]), "d"(v[1]),
                           "d"(v[2]), "d"(v[3])
                           : "memory");
            } else {
              *reinterpret_cast<double2*>(yp) = make_double2(v[0], v[1]);
              *reinterpret_cast<double2*>(yp + 2) = make_double2(v[2], v[3]);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (c0 + i < lim) yp[i] = v[i];
          }
        }
      }
      if (alive && a.zfill && in)                          // columns 16 nch .. ldy - 1
        for (int c = 16 * s.nch + 2 * half; c < a.ldy; c += 4)
          *reinterpret_cast<double2*>(yr + c) = make_double2(0.0, 0.0);
      ++it;
      ++j;
    }
  } else if (lane == 0) {
    // ------------------------------------------------------------------ MMA issue
    int k = range[0], j = range[1], kcur = -1, it = 0, qc = 0;
    unsigned used[2] = {0, 0};
    OtShape s{};
    while (alive && settle(k, j)) {
      if (k != kcur) { s = shape(k); kcur = k; }
      const int b = s.KP <= 48 ? it & 1 : 0;
      alive = tc::mbar_wait(&full[b], used[b] & 1, kWait);
      if (!alive) break;
      tc::fence_after_sync();
      const uint32_t APL = TT_ROWS * 2 * s.KP, MB = 16 * OZ_DIG * 2 * s.KP;
      const uint64_t ad0 = tc::sdesc(tc::smem_u32(msl + (size_t)s.nch * MB + (size_t)b * OZ_DIG * APL),
                                     128, 16 * s.KP);
      const uint64_t bd0 = tc::sdesc(tc::smem_u32(msl), 128, 16 * s.KP);
      const int nslab = s.KP >> 4;
      int c = 0;
      for (; c < s.nch; ++c, ++qc) {
        const int buf = qc & (OT_NB - 1);
        if (qc >= OT_NB) {
          alive = tc::mbar_wait(&tempty[buf], (qc / OT_NB - 1) & 1, kWait);
          if (!alive) break;
          tc::fence_after_sync();
        }
        for (int sl = 0; sl < nslab; ++sl)
#pragma unroll
          for (int d = 0; d < OZ_DIG; ++d)
            tc::mma_bf16(tmem + (uint32_t)(128 * buf + 16 * d), ad0 + ((d * APL + 256 * sl) >> 4),
                         bd0 + ((c * MB + 256 * sl) >> 4),
                         tc::idesc(tc::FMT_BF16, 128, 16 * (OZ_DIG - d)), (sl > 0 || d > 0) ? 1u : 0u);
        tc::mma_commit(&tfull[buf]);
      }
      if (c > 0) {                                     // (a tile cut short by a wait that ran out too)
        tc::mma_commit(&empty[b]);
        ++used[b];
      }
      if (!alive) break;
      ++it;
      ++j;
    }
    // nothing of this CTA's MMAs is in flight when its memory goes back: the last commit of
    // each stage has arrived
    for (int b = 0; b < 2; ++b)
      if (used[b]) alive = tc::mbar_wait(&empty[b], (used[b] - 1) & 1, kWait) && alive;
  }
  if (!alive && lane == 0) atomicOr(a.status, (unsigned)ST_TIMEOUT);
  __syncwarp();
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------------------
// FP64-accurate tall-skinny products A^T diag(w) B on the BF16 tensor cores (Ozaki scheme)
// ---------------------------------------------------------------------------------------
// One launch forms up to OG_PROD products per subdomain (the orthonormalisations' Grams, the
// Galerkin coefficients): each product's rows are cut into chunks of crows rows, and every
// (subdomain, product, chunk) item gives one partial, na x nb entries of an RC x RC block,
// summed by its consumer in chunk order.  With chunk exponents (symmetric Grams) the partial is
// the Gram of 2^-e A (e = the chunk's scale when it is far from 1; INT_MIN for a chunk below
// 2^-1000).
//
// A column's largest exponent over the chunk bounds it by 2^c; the values (weights multiplied
// in, in FP64) become 7 balanced base-256 digits relative to 2^(c + 1) (as for the tall
// products, one bit higher, so that every digit, the leading one included, is in
// [-128, 128]).  The rows are the K dimension of the MMAs: stages of 32 rows, digit planes
// P x 32 (P = the column count rounded up to 16) of both operands.  The M = 128 operand of an
// MMA starting at plane s1 covers h = 128 / P consecutive planes of A: lanes u P .. u P + P - 1
// ("band" u) hold plane s1 + u.  One MMA per s1 in {0, h, 2h, ..} with B's planes t = 0 .. 6 - s1
// stacked along N (accumulator column block s1 + t) serves every band at once: in band u, block
// c accumulates the digit pairs (s, t) of order s + t = c + u, at most 4 of them: over 256 rows
// their sums stay within 2^24, exact in FP32, and the accumulators are read out.  The read-out
// combines a band's blocks in 64-bit integers (< 2^63), shifts band u down by 8 u bits, adds the
// bands and converts to FP64.  Error: a few units of 2^-54 of the product of the two columns'
// largest entries per row (an FP64 dot product rounds every partial sum to 2^-53 of it).
//
// One CTA per SM, its warps specialised, each CTA walking a contiguous range of items of about
// equal cost:
//   8 converter warps  8 x 8 blocks of an operand -> registers (a stage ahead) -> digit planes
//                      (a warp's 32 stores of a plane are 128 consecutive bytes);
//   8 auxiliary warps  the column bounds of the item after the one being converted, then the
//                      read-out of the item before it;
//   1 MMA warp.
// The FP64 pipe does 2 operations per clock and SM, which made these products the largest part
// of a step with the rank at 20 (r_t = 40): spatial coefficients of 262144 x 40, per launch:
// 1700 us on the FP64 pipe, 470 now; the angular ones (131072 directions) 1300 -> 620; an
// orthonormalisation's Gram 271 on the FP64 pipe, 150 with this scheme but CTA-wide phases, 85
// (angular) to 140 (spatial) now.  Bound by instruction issue: 45% of the cycles, a third of the
// stalls for instructions (the roles' code together), the rest loads; 25 warps with the bounds
// and the read-out apart (72 registers, spills) were 25% slower, 16 converter warps 7%.
#define OG_KS 32                          // rows per stage (K of one stage's MMAs)
#define OG_GROUP 256                      // rows per read-out
#define OG_RING 4                         // items whose column exponents are kept
#define OG_XLD 17
#define OG_CONV 8                         // converter warps
#define OG_THREADS ((OG_CONV + 8 + 1) * 32)

// dynamic shared memory: stages, the space an M = 128 operand may read past the last plane,
// the read-out's exchange buffer
static __host__ __device__ __forceinline__ uint32_t og_stage(int RC) {
  return (uint32_t)OZ_DIG * 2 * ((RC + 15) / 16 * 16) * (2 * OG_KS);
}
static __host__ __device__ __forceinline__ int og_stages(int RC) { return og_stage(RC) * 4 <= 120 * 1024 ? 4 : 3; }
static size_t og_smem(int RC) {
  return 128 + (size_t)og_stages(RC) * og_stage(RC) + 128 * 2 * OG_KS + (size_t)128 * OG_XLD * 8;
}

__device__ __forceinline__ void og_aux_sync() { asm volatile("bar.sync 3, 256;" ::: "memory"); }

// rows of product p of subdomain k, columns of its operands
__device__ __forceinline__ void og_shape(const OzGram& a, int k, const OzProd& p, int* rows, int* na,
                                         int* nb) {
  *rows = p.rows == OG_CELLS ? a.g.N[k] : p.rows == OG_DIRS ? a.g.n : lines_of(a.g, k, a.axis).nlines;
  int ka = k;
  if (p.aside >= 0) {
    ka = a.g.nb[k * 4 + 2 * a.axis + p.aside];
    if (ka < 0) {                        // no neighbour: its physical inflow's column, or nothing
      const bool in = a.infl_on && a.infl_on[k * 4 + 2 * a.axis + p.aside];
      *na = in ? 1 : 0;
      *nb = p.bcnt ? p.bcnt[k] : p.bfix;
      if (!in) *rows = 0;
      return;
    }
  }
  *na = p.acnt ? p.acnt[ka] : p.afix;
  *nb = p.B ? (p.bcnt ? p.bcnt[k] : p.bfix) : *na;
}
__device__ __forceinline__ int og_chunks(const OzGram& a, int rows) {
  return rows > 0 ? (rows + a.crows - 1) / a.crows : 0;
}

// an item's operands: element (row, column) of A at A[row * astep + column]
struct OgItem {
  const double *A, *B, *w;              // w: row weights (null: none)
  long astep, bstep;
  int k, blk, c, r0, r1, na, nb, PA, PB, wsel, nx, shift;   // nx: row length for the line starts
  int rsafe;                            // a row of B that may be read in place of one left out
  bool sym, eok;
};
__device__ __forceinline__ OgItem og_item(const OzGram& a, int k, int pi, int c) {
  const OzProd& p = a.p[pi];
  OgItem t;
  int rows;
  og_shape(a, k, p, &rows, &t.na, &t.nb);
  t.k = k; t.c = c; t.blk = p.blk;
  t.r0 = c * a.crows;
  t.r1 = min(rows, t.r0 + a.crows);
  t.PA = t.na <= 16 ? 16 : (t.na + 15) & ~15;
  t.PB = t.nb <= 16 ? 16 : (t.nb + 15) & ~15;
  t.sym = p.B == nullptr;
  t.shift = p.shift;
  t.wsel = p.wsel;
  // (a shifted operand's rows start one cell early; row rsafe is inside)
  t.rsafe = p.shift ? (a.axis == 0 ? 1 : a.g.nxk[k]) : t.r0;
  t.w = nullptr;
  t.nx = p.shift ? (a.axis == 0 ? a.g.nxk[k] : 0) : 0;
  t.eok = a.cexp != nullptr;
  t.astep = p.lda;
  t.bstep = p.ldb;
  if (p.rows == OG_DIRS) {
    const int ka = p.aside >= 0 ? a.g.nb[k * 4 + 2 * a.axis + p.aside] : k;
    if (ka >= 0) {
      t.A = p.A + (long)ka * a.g.n * p.lda;
    } else {                            // physical inflow: one column, already masked
      t.A = a.infl_hw + ((long)k * 4 + 2 * a.axis + p.aside) * a.g.n;
      t.astep = 1;
    }
    t.B = t.sym ? t.A : p.B + (long)k * a.g.n * p.ldb;
    if (p.wsel != W_NONE) t.w = a.axis == 0 ? a.ox : a.oy;
  } else {
    const long row0 = a.g.rowoff[k];
    if (p.rows == OG_CELLS) {
      t.A = p.A + row0 * p.lda;
      t.B = t.sym ? t.A : p.B + row0 * p.ldb;
      if (p.shift) t.B = t.A - (long)(a.axis == 0 ? 1 : a.g.nxk[k]) * p.lda;
      if (p.shift) t.bstep = p.lda;
      if (p.wsel == W_ROW) t.w = p.wrow + row0;
    } else {
      const Lines L = lines_of(a.g, k, a.axis);
      const int side = p.rows == OG_FACE_HI;
      t.A = p.A + (row0 + cell_of(L, 0, side ? L.len - 1 : 0)) * p.lda;
      t.astep = (long)L.stride_line * p.lda;
      t.B = p.B + ((long)k * 2 + side) * a.maxlines * p.ldb;
    }
  }
  return t;
}
// whether a shift leaves row r of B inside its line
__device__ __forceinline__ bool og_inside(const OzGram& a, const OgItem& t, int r) {
  return !t.shift || (a.axis == 0 ? r % t.nx != 0 : r >= a.g.nxk[t.k]);
}
// whether a row of weight w is on the right side of a mask
__device__ __forceinline__ bool og_side(const OgItem& t, double w) {
  const long long ob = __double_as_longlong(w);
  const bool ng = ob < 0 && ob != (long long)0x8000000000000000ull;
  return !(t.wsel == W_NEG || t.wsel == W_NONNEG) || (t.wsel == W_NEG) == ng;
}
// the weight of a row (Omega+ and Omega- vanish on the other side)
__device__ __forceinline__ double og_weight(const OgItem& t, double w) {
  if (t.wsel == W_OMEGA_POS) return w > 0.0 ? w : 0.0;
  if (t.wsel == W_OMEGA_NEG) return w < 0.0 ? w : 0.0;
  return w;
}
__device__ __forceinline__ bool og_weighted(const OgItem& t) {
  return t.wsel == W_OMEGA || t.wsel == W_OMEGA_POS || t.wsel == W_OMEGA_NEG || t.wsel == W_ROW;
}

// Two rows (p0, p1) of an operand: column ci of the 8-column groups cg + 2 i, i < NB (columns past n
// read the last one)
template <int NB>
__device__ __forceinline__ void og_load(double (&d)[4][2], const double* p0, const double* p1, int cg,
                                        int ci, int n) {
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int col = max(0, min(8 * (cg + 2 * i) + ci, n - 1));
    d[i][0] = __ldg(p0 + col);
    d[i][1] = __ldg(p1 + col);
  }
}
__device__ __forceinline__ void og_load(double (&d)[4][2], const double* p0, const double* p1, int cg,
                                        int ci, int n, int P) {
  if (P <= 16) og_load<1>(d, p0, p1, cg, ci, n);                // warp-uniform; P a multiple of 16
  else if (P <= 32) og_load<2>(d, p0, p1, cg, ci, n);
  else if (P <= 48) og_load<3>(d, p0, p1, cg, ci, n);
  else og_load<4>(d, p0, p1, cg, ci, n);
}
// their digits (rows rp, rp + 1 of the stage; weights w multiplied in when mul; rows that are not
// ok count as zero; cs: column exponents) into the planes at base, PL apart
template <int NB>
__device__ __forceinline__ void og_convert(const double (&x)[4][2], const double (&w)[2], bool mul,
                                           const bool (&ok)[2], int cg, int ci, int rp, const int* cs,
                                           int n, uint8_t* base, uint32_t PL) {
  double v[NB][2];
#pragma unroll
  for (int i = 0; i < NB; ++i) { v[i][0] = x[i][0]; v[i][1] = x[i][1]; }
  if (mul)
#pragma unroll
    for (int i = 0; i < NB; ++i) { v[i][0] *= w[0]; v[i][1] *= w[1]; }
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int col = 8 * (cg + 2 * i) + ci, e1 = cs[col] + 1;
    uint32_t d[OZ_DIG];
    oz_digits2(ok[0] && col < n ? v[i][0] : 0.0, e1, ok[1] && col < n ? v[i][1] : 0.0, e1, d);
    uint8_t* pl = base + tc::op_off(col, rp * 2, 2 * OG_KS);
#pragma unroll
    for (int s = 0; s < OZ_DIG; ++s) *reinterpret_cast<uint32_t*>(pl + s * PL) = d[s];
  }
}
__device__ __forceinline__ void og_convert(const double (&x)[4][2], const double (&w)[2], bool mul,
                                           const bool (&ok)[2], int cg, int ci, int rp, const int* cs,
                                           int n, uint8_t* base, uint32_t PL, int P) {
  if (P <= 16) og_convert<1>(x, w, mul, ok, cg, ci, rp, cs, n, base, PL);
  else if (P <= 32) og_convert<2>(x, w, mul, ok, cg, ci, rp, cs, n, base, PL);
  else if (P <= 48) og_convert<3>(x, w, mul, ok, cg, ci, rp, cs, n, base, PL);
  else og_convert<4>(x, w, mul, ok, cg, ci, rp, cs, n, base, PL);
}

__global__ void __launch_bounds__(OG_THREADS, 1) k_oz_gram(const __grid_constant__ OzGram a) {
  extern __shared__ uint8_t raw_og[];
  uint8_t* buf0 = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_og) + 127) &
                                             ~uintptr_t(127));
  const int RC = a.g.RC, NST = og_stages(RC);
  const uint32_t SB = og_stage(RC);
  long long* X = reinterpret_cast<long long*>(buf0 + (size_t)NST * SB + 128 * 2 * OG_KS);
  __shared__ uint64_t full[4], empty[4], tfull[2], tempty[2], bnd[OG_RING];
  __shared__ uint32_t tmem_s;
  __shared__ int cs[OG_RING][2][DD_MAXC], exs[OG_RING], cred[8][2][DD_MAXC];
  __shared__ int part_w[32], range[4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int npair = a.g.nsub * a.nprod;
  // ---- this CTA's items: pairs (subdomain, product) in order, chunks within a pair; an item
  // costs its stages' conversions (and their MMAs) and a read-out
  auto pair_cost = [&](int u, int* nck) {
    int rows, na, nb;
    const OzProd& p = a.p[u % a.nprod];
    og_shape(a, u / a.nprod, p, &rows, &na, &nb);
    *nck = og_chunks(a, rows);
    const int st = (min(rows, a.crows) + OG_KS - 1) / OG_KS;
    return st * (2 + ((na + 15) >> 4) + (p.B ? (nb + 15) >> 4 : 1)) + 20;
  };
  {
    const int per = (npair + 511) / 512, ua = min(npair, tid * per), ub = tid < 512 ? min(npair, ua + per) : ua;
    int w = 0;
    for (int u = ua; u < ub; ++u) {
      int nck;
      const int c = pair_cost(u, &nck);
      w += nck * c;
    }
    int inc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) part_w[warp] = inc;
    if (tid < 4) range[tid] = tid & 1 ? 0 : npair;
    __syncthreads();
    int total = 0, before = 0;
    for (int i = 0; i < 16; ++i) {
      if (i < warp) before += part_w[i];
      total += part_w[i];
    }
    const int lo = before + inc - w;
    for (int side = 0; side < 2; ++side) {
      const int x = (int)((long)(blockIdx.x + side) * total / gridDim.x);
      if (w > 0 && x >= lo && x < lo + w) {
        int at = lo;
        for (int u = ua; u < ub; ++u) {
          int nck;
          const int c = pair_cost(u, &nck);
          if (x < at + nck * c) {
            range[2 * side] = u;
            range[2 * side + 1] = (x - at + c - 1) / c;
            break;
          }
          at += nck * c;
        }
      }
    }
  }
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) { tc::mbar_init(&full[i], OG_CONV); tc::mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { tc::mbar_init(&tfull[i], 1); tc::mbar_init(&tempty[i], 8); }
    for (int i = 0; i < OG_RING; ++i) tc::mbar_init(&bnd[i], 8);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(&tmem_s, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_s;
  const int u1 = range[2], c1 = range[3];
  // the next existing item at or after (u, c); false past this CTA's last
  auto settle = [&](int& u, int& c) {
    while (u < npair && (u < u1 || (u == u1 && c < c1))) {
      int rows, na, nb;
      og_shape(a, u / a.nprod, a.p[u % a.nprod], &rows, &na, &nb);
      if (c < og_chunks(a, rows)) return true;
      ++u;
      c = 0;
    }
    return false;
  };
  bool alive = true;

  if (warp < OG_CONV) {
    // ------------------------------------------------------------------ converters
    // A stage's 8 x 8 blocks: warp w takes row group w % 4 and the column groups w / 4 + 2 i of A,
    // then of B; an operand's loads are under way while the one before it converts
    int u = range[0], c = range[1], it = 0, st = 0;
    const int ci = lane & 7, rp = 8 * (warp & 3) + 2 * (lane >> 3), cg = warp >> 2;
    while (settle(u, c)) {
      const OgItem t = og_item(a, u / a.nprod, u % a.nprod, c);
      const int slot = it & (OG_RING - 1);
      const int nst = (t.r1 - t.r0 + OG_KS - 1) / OG_KS, nh = t.sym ? nst : 2 * nst;
      const bool wtd = og_weighted(t);
      double x[4][2], y[4][2], xw[2], yw[2];
      bool xo[2], yo[2];
      // half-stage hs: operand A or B of a stage (a symmetric product has A alone)
      auto load = [&](double(&d)[4][2], double(&w)[2], bool(&ok)[2], int hs) {
        const bool isB = !t.sym && (hs & 1);
        const int r = t.r0 + (t.sym ? hs : hs >> 1) * OG_KS + rp, n = isB ? t.nb : t.na;
        const double* p[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int rr = min(r + h, t.r1 - 1);
          ok[h] = r + h < t.r1;
          // (the row's weight or mask is looked at only when the row is converted: an address
          // that waited for it would hold up the conversion before)
          w[h] = 1.0;
          bool in = true;
          if (isB || t.sym) {
            in = og_inside(a, t, rr);
            ok[h] = ok[h] && in;
            if (t.w) w[h] = t.w[rr];
          }
          p[h] = (isB ? t.B : t.A) + (long)(in ? rr : t.rsafe) * (isB ? t.bstep : t.astep);
        }
        og_load(d, p[0], p[1], cg, ci, n, isB ? t.PB : t.PA);
      };
      load(x, xw, xo, 0);
      if (a.g.work)
        count_work(a.g, KS_OZ_GRAM, (t.sym ? 1.0 : 2.0) * (t.r1 - t.r0) * t.na * (t.sym ? t.na + 1 : t.nb));
      alive = tc::mbar_wait(&bnd[slot], (it / OG_RING) & 1, kWait) && alive;
      const uint32_t PLA = (uint32_t)t.PA * 2 * OG_KS, PLB = (uint32_t)t.PB * 2 * OG_KS;
#pragma unroll 1
      for (int hs = 0; hs < nh; ++hs) {
        if (hs + 1 < nh) load(y, yw, yo, hs + 1);
        const bool isB = !t.sym && (hs & 1), first = !isB, lasth = t.sym || isB;
        const int b4 = st % NST, use = st / NST;
        if (first && use > 0 && alive) alive = tc::mbar_wait(&empty[b4], (use - 1) & 1, kWait);
        uint8_t* base = buf0 + (size_t)b4 * SB + (isB ? OZ_DIG * PLA : 0u);
        const bool mul = wtd && (isB || t.sym);
        if (t.w && (isB || t.sym)) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            xo[h] = xo[h] && og_side(t, xw[h]);
            xw[h] = og_weight(t, xw[h]);
          }
        }
        og_convert(x, xw, mul, xo, cg, ci, rp, cs[slot][isB], isB ? t.nb : t.na, base, isB ? PLB : PLA,
                   isB ? t.PB : t.PA);
        if (lasth) {
          tc::fence_async_smem();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&full[b4]);
          ++st;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) { x[i][0] = y[i][0]; x[i][1] = y[i][1]; }
        xw[0] = yw[0]; xw[1] = yw[1];
        xo[0] = yo[0]; xo[1] = yo[1];
      }
      ++it;
      ++c;
    }
  } else if (warp < OG_CONV + 8) {
    // ------------------------------------------------------------------ bounds and read-out
    const int w8 = warp - OG_CONV, q4 = warp & 3, half = w8 >> 2, at = tid - 32 * OG_CONV;
    // column exponents of item number it: A (and B when it is another operand)
    auto bounds = [&](const OgItem& t, int it) {
      const int slot = it & (OG_RING - 1);
      const bool wtd = og_weighted(t);
#pragma unroll
      for (int op = 0; op < 2; ++op) {
        if (op == 1 && t.sym) break;
        const double* base = op ? t.B : t.A;
        const long step = op ? t.bstep : t.astep;
        const int n = op ? t.nb : t.na;
        const bool side = op == 1 || t.sym;
        int m0 = 0, m1 = 0;                              // biased exponents
        const int c0 = max(0, min(lane, n - 1)), c1 = max(0, min(lane + 32, n - 1));
        const bool plain = !side || !(wtd || t.shift || t.wsel == W_NEG || t.wsel == W_NONNEG);
        for (int rb = t.r0 + w8; rb < t.r1; rb += 128) {     // 16 rows at a time, all loads first
          int h0[16], h1[16], ew[16];
          if (plain) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int* hw = reinterpret_cast<const int*>(base + (long)min(rb + 8 * i, t.r1 - 1) * step) + 1;
              h0[i] = __ldg(hw + 2 * c0);
              h1[i] = __ldg(hw + 2 * c1);
              ew[i] = 0;
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int r = min(rb + 8 * i, t.r1 - 1);
              const bool in = og_inside(a, t, r);
              const double w = t.w ? t.w[r] : 1.0;
              const int* hw = reinterpret_cast<const int*>(base + (long)(in ? r : t.rsafe) * step) + 1;
              h0[i] = __ldg(hw + 2 * c0);
              h1[i] = __ldg(hw + 2 * c1);
              const int E = wtd ? f64_bexp(og_weight(t, w)) : 1022;
              ew[i] = in && og_side(t, w) && E ? E - 1022 : -4096;
            }
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int E0 = (h0[i] >> 20) & 0x7ff, E1 = (h1[i] >> 20) & 0x7ff;
            m0 = max(m0, E0 ? E0 + ew[i] : 0);
            m1 = max(m1, E1 ? E1 + ew[i] : 0);
          }
        }
        if (lane >= n) m0 = 0;
        if (lane + 32 >= n) m1 = 0;
        cred[w8][op][lane] = m0;
        cred[w8][op][lane + 32] = m1;
      }
      og_aux_sync();
      if (at < 2 * DD_MAXC) {
        const int op = at >> 6, col = at & 63;
        if (op == 0 || !t.sym) {
          int m = cred[0][op][col];
#pragma unroll
          for (int i = 1; i < 8; ++i) m = max(m, cred[i][op][col]);
          const int e = m > 0 ? m - 1022 : OZ_NONE;
          cs[slot][op][col] = e;
          if (t.sym) cs[slot][1][col] = e;
        }
      }
      if (t.eok && w8 == 0) {                            // the chunk's scale
        int m = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) m = max(m, max(cred[i][0][lane], cred[i][0][lane + 32]));
        m = __reduce_max_sync(0xffffffffu, m);
        const int e0 = m > 0 && m < 2047 ? m - 1023 : 0;
        const bool zero = m <= 0 || e0 < -1000;
        const int ex = (!zero && (e0 < -400 || e0 > 400)) ? e0 : 0;
        if (lane == 0) {
          exs[slot] = ex;
          a.cexp[(long)t.k * a.nchunk + t.c] = zero ? INT_MIN : ex;
        }
      }
      __syncwarp();
      og_aux_sync();                                     // cred is read; cs, exs are written
      if (lane == 0) tc::mbar_arrive(&bnd[slot]);
    };
    int grp = 0;                                         // read-out groups done
    auto readout = [&](const OgItem& t, int it) {
      const int slot = it & (OG_RING - 1), h = 128 / t.PA, nbd = min(h, OZ_DIG);
      const int tb = 14 * t.PB <= 512 ? 2 : 1;
      const int L = q4 * 32 + lane, u = L / t.PA;
      double* out = a.part + (((long)t.k * a.nchunk + t.c) * a.nblk + t.blk) * RC * RC;
      for (int r = t.r0; r < t.r1; r += OG_GROUP, ++grp) {
        // the group's TMEM half (all of it where 7 blocks do not fit twice)
        const int b2 = grp & 1;
        alive = __all_sync(0xffffffffu, tc::mbar_wait(&tfull[b2], (grp >> 1) & 1, kWait)) && alive;
        alive = __all_sync(0xffffffffu, alive);
        tc::fence_after_sync();
        for (int cg = 0; cg < t.PB; cg += 16) {
          if (alive) {
#pragma unroll 1
            for (int c4 = 8 * half; c4 < 8 * half + 8; c4 += 4) {
              uint32_t D[OZ_DIG][4];
#pragma unroll
              for (int g = 0; g < OZ_DIG; ++g)
                oz_tmem_ld4(tmem + ((uint32_t)(q4 * 32) << 16) +
                                (uint32_t)((tb == 2 ? 256 * b2 : 0) + g * t.PB + cg + c4), D[g]);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int g = 0; g < OZ_DIG; ++g)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  asm volatile("" : "+r"(D[g][i]));
                  if (g + u > OZ_DIG - 1) D[g][i] = 0u;  // orders past the last (junk planes among them)
                }
#pragma unroll
              for (int i = 0; i < 4; ++i)
                X[L * OG_XLD + c4 + i] = u < nbd ? oz_combine(&D[0][i], 4) >> (8 * u) : 0ll;
            }
          }
          if (cg + 16 >= t.PB) {                         // the accumulators are free again
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&tempty[b2]);
          }
          og_aux_sync();
          if (alive) {
            const int j = at & 15, col = cg + j;
            const int ex = t.eok ? 2 * exs[slot] : 0;
            if (col < t.nb)
              for (int i = at >> 4; i < t.na; i += 16) {
                long long J = 0;
                for (int v = 0; v < nbd; ++v) J += X[(v * t.PA + i) * OG_XLD + j];
                const double v = oz_round(J, cs[slot][0][i] + cs[slot][1][col] + 2 - 56 - ex);
                double* o = out + i * RC + col;
                *o = r == t.r0 ? v : *o + v;
              }
          }
          og_aux_sync();                                 // X is free
        }
      }
    };
    int u = range[0], c = range[1], it = 0;
    bool more = settle(u, c);
    OgItem prev{};
    bool have = false;
    while (more || have) {
      OgItem cur{};
      const bool now = more;
      if (now) {
        cur = og_item(a, u / a.nprod, u % a.nprod, c);
        ++c;
        more = settle(u, c);
        if (more && at == 0 && a.p[u % a.nprod].rows <= OG_DIRS) {   // the next item's rows into L2
          const OgItem nx = og_item(a, u / a.nprod, u % a.nprod, c);
          if (!(nx.astep & 1)) prefetch_rows(nx.A, nx.astep, nx.r0, nx.r1 - nx.r0, nx.r1);
          if (!nx.sym && !nx.shift && !(nx.bstep & 1))
            prefetch_rows(nx.B, nx.bstep, nx.r0, nx.r1 - nx.r0, nx.r1);
        }
        bounds(cur, it);
      }
      if (have) readout(prev, it - 1);
      prev = cur;
      have = now;
      ++it;
    }
  } else if (lane == 0) {
    // ------------------------------------------------------------------ MMA issue
    int u = range[0], c = range[1], st = 0, grp = 0, last = -1;
    bool dbl = true;                                     // the previous group left the other half free
    while (alive && settle(u, c)) {
      const OgItem t = og_item(a, u / a.nprod, u % a.nprod, c);
      const int h = 128 / t.PA, nper = 256 / t.PB, tb = 14 * t.PB <= 512 ? 2 : 1;
      const uint32_t PLA = (uint32_t)t.PA * 2 * OG_KS, PLB = (uint32_t)t.PB * 2 * OG_KS;
      for (int r = t.r0; r < t.r1 && alive; r += OG_GROUP, ++grp) {
        const int b2 = grp & 1;
        // this group's accumulators: the half's previous group is read out, and where either
        // this group or the one before it spans both halves, that one too
        if (grp >= 2) alive = tc::mbar_wait(&tempty[b2], ((grp >> 1) - 1) & 1, kWait);
        if (alive && grp >= 1 && (tb == 1 || !dbl))
          alive = tc::mbar_wait(&tempty[b2 ^ 1], ((grp - 1) >> 1) & 1, kWait);
        if (!alive) break;
        tc::fence_after_sync();
        dbl = tb == 2;
        const uint32_t d0 = tmem + (tb == 2 ? 256u * b2 : 0u);
        const int re = min(t.r1, r + OG_GROUP);
        for (int s0 = r; s0 < re; s0 += OG_KS, ++st) {
          const int b4 = st % NST;
          alive = tc::mbar_wait(&full[b4], (st / NST) & 1, kWait);
          if (!alive) break;
          tc::fence_after_sync();
          const uint32_t sa = tc::smem_u32(buf0 + (size_t)b4 * SB);
          const uint64_t ad = tc::sdesc(sa, 128, 16 * OG_KS);
          const uint64_t bd = t.sym ? ad : tc::sdesc(sa + OZ_DIG * PLA, 128, 16 * OG_KS);
          for (int j = 0; j < OG_KS / 16; ++j)
            for (int s1 = 0; s1 < OZ_DIG; s1 += h)
              for (int v0 = 0; v0 < OZ_DIG - s1; v0 += nper) {
                const int nu = min(nper, OZ_DIG - s1 - v0);
                tc::mma_bf16(d0 + (uint32_t)((s1 + v0) * t.PB), ad + ((s1 * PLA + 256 * j) >> 4),
                             bd + ((v0 * PLB + 256 * j) >> 4),
                             tc::idesc(tc::FMT_BF16, 128, nu * t.PB),
                             (s0 > r || j > 0 || s1 > 0) ? 1u : 0u);
              }
          tc::mma_commit(&empty[b4]);
          last = st;
        }
        if (!alive) break;
        tc::mma_commit(&tfull[b2]);
      }
      ++c;
    }
    // every MMA issued is complete before the memory goes back
    if (last >= 0) alive = tc::mbar_wait(&empty[last % NST], (last / NST) & 1, kWait) && alive;
  }
  if (!alive && lane == 0) atomicOr(a.status, (unsigned)ST_TIMEOUT);
  __syncwarp();
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// Sum of the chunk partials of every product, in chunk order, into the small matrices (slot
// dst[blk]), zero outside the product's na x nb entries.  Grid: (products x entries, subdomains): y
// ends at 65535, so that this kernel takes as many subdomains as every other one.  (The product in
// z, where its descriptor's index is uniform, took 14 us a launch instead of 11: one subdomain of
// 16384 cells, 64 chunks of 30 x 30.)
__global__ void __launch_bounds__(DD_THREADS) k_oz_reduce(const __grid_constant__ OzGram a, OzDst dst,
                                                          double* sm) {
  const int k = blockIdx.y, RC = a.g.RC;
  const int nbx = (RC * RC + DD_THREADS - 1) / DD_THREADS, pi = blockIdx.x / nbx;
  const OzProd& p = a.p[pi];
  int rows, na, nb;
  og_shape(a, k, p, &rows, &na, &nb);
  const int nck = og_chunks(a, rows);
  const double* part = a.part + ((long)k * a.nchunk * a.nblk + p.blk) * RC * RC;
  double* out = sm + ((long)k * NSMALL + dst.idx[p.blk]) * RC * RC;
  const int e = (blockIdx.x - pi * nbx) * DD_THREADS + threadIdx.x;
  if (e >= RC * RC) return;
  const int i = e / RC, j = e - i * RC;
  double s = 0.0;
  if (i < na && j < nb) {
#pragma unroll 8
    for (int c = 0; c < nck; ++c) s += part[(long)c * a.nblk * RC * RC + e];
  }
  out[e] = s;
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
// Failure-detection self-test of the bounded wait that every tensor-core kernel uses for its
// tile loads and MMAs: one thread initialises an mbarrier expecting one arrival that nothing
// makes and waits on its phase 0 for at most `polls` polls.  When the wait runs out it records
// ST_TIMEOUT in *status, as the production kernels do, then makes the arrival itself so that
// the barrier's phase is complete when the CTA exits.
__global__ void k_wait_selftest(unsigned* status, uint32_t polls) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  tc::mbar_init(&bar, 1);
  tc::mbar_init_fence();
  if (!tc::mbar_wait(&bar, 0, polls)) {
    atomicOr(status, (unsigned)ST_TIMEOUT);
    tc::mbar_arrive(&bar);
  }
}

cudaError_t wait_selftest(unsigned* status, unsigned polls, cudaStream_t st) {
  k_wait_selftest<<<1, 32, 0, st>>>(status, polls);
  return cudaGetLastError();
}

cudaError_t tc_init() {
  if (!g_encode.load(std::memory_order_acquire)) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    g_encode.store(reinterpret_cast<EncodeTiledFn>(fn), std::memory_order_release);
  }
  cudaError_t e;
  e = cudaFuncSetAttribute(k_tc_tall<tc::FMT_TF32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)tc_tall_smem());
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_tc_tall<tc::FMT_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)tc_tall_smem());
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_tc_gram<tc::FMT_TF32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)tc_gram_smem());
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_oz_tall, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)ot_smem(DD_MAXC));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_oz_gram, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)og_smem(DD_MAXC));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_tc_gram<tc::FMT_BF16>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_gram_smem());
}

bool tc_tall(const Problem& P, unsigned* status, cudaStream_t st, int spatial, const double* A,
             int lda, const int* ninner, int ninner_fix, const double* Bm, int bsmall,
             const double* smbase, const int* ncols, int ncols_fix, double* Y, int ldy,
             double alpha, int accumulate) {
  const long rows_all = spatial ? P.Ntot : (long)P.g.nsub * P.g.n;
  CUtensorMap map;
  if (!make_map(&map, A, lda, rows_all, TT_ROWS)) return false;
  TcTall a;
  a.g = P.g; a.spatial = spatial; a.lda = lda; a.ninner = ninner; a.ninner_fix = ninner_fix;
  a.Bm = Bm; a.bsmall = bsmall; a.smbase = smbase; a.ncols = ncols; a.ncols_fix = ncols_fix;
  a.Y = Y; a.ldy = ldy; a.alpha = alpha; a.accumulate = accumulate; a.status = status;
  a.A = A; a.mtrans = 0; a.rowscale = nullptr; a.nrows = 0; a.zfill = 1;
  a.tps = ((spatial ? P.maxN : P.g.n) + TT_ROWS - 1) / TT_ROWS;
  const long ntot = (long)P.g.nsub * a.tps;
  const int grid = (int)std::min<long>(ntot, P.nsm);
  pbeg(st, KS_TC_TALL);
  if (P.prec == PREC_BF16)
    k_tc_tall<tc::FMT_BF16><<<grid, TT_THREADS, tc_tall_smem(), st>>>(map, a);
  else
    k_tc_tall<tc::FMT_TF32><<<grid, TT_THREADS, tc_tall_smem(), st>>>(map, a);
  pend(st);
  return true;
}

bool oz_tall(const Problem& P, unsigned* status, cudaStream_t st, int spatial, const double* A,
             int lda, const int* ninner, int ninner_fix, const double* Bm, int bsmall,
             const double* smbase, const int* ncols, int ncols_fix, double* Y, int ldy,
             int mtrans, int accumulate, const double* rowscale) {
  if (lda > DD_MAXC || (lda & 1) || (ldy & 1)) return false;
  TcTall a;
  a.g = P.g; a.spatial = spatial; a.lda = lda; a.ninner = ninner; a.ninner_fix = ninner_fix;
  a.Bm = Bm; a.bsmall = bsmall; a.smbase = smbase; a.ncols = ncols; a.ncols_fix = ncols_fix;
  a.Y = Y; a.ldy = ldy; a.alpha = 1.0; a.accumulate = accumulate; a.status = status;
  a.A = A;
  a.nrows = spatial ? P.Ntot : (long)P.g.nsub * P.g.n;
  a.zfill = !accumulate && P.prec >= PREC_TF32;
  a.mtrans = mtrans;
  a.rowscale = rowscale;
  a.tps = ((spatial ? P.maxN : P.g.n) + TT_ROWS - 1) / TT_ROWS;
  const long ntot = (long)P.g.nsub * a.tps;
  const int grid = (int)std::min<long>(ntot, P.nsm);
  pbeg(st, KS_OZ_TALL);
  k_oz_tall<<<grid, OT_THREADS, ot_smem(lda), st>>>(a);
  pend(st);
  return true;
}

bool tc_gram(const Problem& P, cudaStream_t st, const TcGram& a0) {
  TcGram a = a0;
  a.g = P.g;
  a.ox = P.ox;
  a.oy = P.oy;
  const long rows_all = a.spatial ? P.Ntot : (long)P.g.nsub * P.g.n;
  CUtensorMap mb, ma[2];
  if (!make_map(&mb, a.B, a.ldb, rows_all, TG_ROWS)) return false;
  // one tensor map per source slot of a CTA (slot h holds sources h, h + 2, ...: the same
  // array is required across a slot's sources)
  for (int h = 0; h < 2; ++h) {
    const TcGramSrc* s = nullptr;                     // the slot's first loaded source
    for (int p = h; p < a.nsrc; p += 2) {
      if (a.src[p].same_as_b) continue;
      if (!s) s = &a.src[p];
      else if (a.src[p].ptr != s->ptr || a.src[p].ld != s->ld) return false;
    }
    if (!make_map(&ma[h], s ? s->ptr : a.B, s ? s->ld : a.ldb, rows_all, TG_ROWS)) return false;
  }
  dim3 grid(a.nchunk, P.g.nsub, (a.nsrc + 1) / 2);
  pbeg(st, KS_TC_GRAM);
  if (P.prec == PREC_BF16)
    k_tc_gram<tc::FMT_BF16><<<grid, TG_THREADS, tc_gram_smem(), st>>>(mb, ma[0], ma[1], a);
  else
    k_tc_gram<tc::FMT_TF32><<<grid, TG_THREADS, tc_gram_smem(), st>>>(mb, ma[0], ma[1], a);
  pend(st);
  return true;
}

bool oz_gram(const Problem& P, cudaStream_t st, OzGram& a, const OzDst* dst, double* sm) {
  if (P.g.RC > DD_MAXC || a.nprod < 1) return false;
  a.g = P.g;
  a.ox = P.ox; a.oy = P.oy;
  a.maxlines = P.maxlines;
  a.infl_on = P.infl_on; a.infl_hw = P.infl_hw;
  pbeg(st, KS_OZ_GRAM);
  k_oz_gram<<<P.nsm, OG_THREADS, og_smem(P.g.RC), st>>>(a);
  pend(st);
  if (dst) {
    pbeg(st, KS_REDUCE);
    const int nbx = (P.g.RC * P.g.RC + DD_THREADS - 1) / DD_THREADS;
    k_oz_reduce<<<dim3(nbx * a.nprod, P.g.nsub), DD_THREADS, 0, st>>>(a, *dst, sm);
    pend(st);
  }
  return true;
}

}  // namespace dd

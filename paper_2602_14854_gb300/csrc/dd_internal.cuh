// Internal declarations of the DD-DLRA CUDA library (not part of the ABI).
//
// Storage convention on the device (the factors of the paper, rescaled so that
// every orthonormality is Euclidean):
//   X = sqrt(hx*hy) * U        (N_k x r, row-major, X^T X = I)
//   Vt = diag(sqrt(w)) * V     (n x r,   row-major, Vt^T Vt = I)
//   S                          (r x r,   the paper's S)
// so f_{c,q} = X_c S Vt_q^T / (sqrt(hx*hy) sqrt(w_q)) and the singular values of S
// are the paper's weighted L2 singular values (Section 3.4 matrix form).
//
// Spatial tall arrays hold all subdomains back to back: row rowoff[k] + c for
// cell c (x-fastest inside subdomain k).  Angular tall arrays hold n rows per
// subdomain: row k*n + q.  Small per-subdomain matrices are RC x RC blocks.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#define DD_MAXC 64          // maximum columns of any tall or small matrix
#define DD_THREADS 256

namespace dd {

enum OrthMode { ORTH_QR = 0, ORTH_AUG = 1, ORTH_COMPLETE = 2 };
enum StatusBits { ST_NONFINITE = 1, ST_COMPLETION = 2, ST_RANKCAP = 4, ST_TIMEOUT = 8 };
// arithmetic of the step (dd_options.precision)
enum Prec { PREC_FP64 = 0, PREC_MIXED = 1, PREC_TF32 = 2, PREC_BF16 = 3 };

// Geometry of the tiling, device arrays (read-only inside kernels).
struct Geo {
  int nsub, n, RC, MC;
  const int* N;      // cells of subdomain k
  const int* nxk;    // width
  const int* nyk;    // height
  const int* rowoff; // first spatial row of subdomain k
  const int* nb;     // 4 per subdomain: x-lo, x-hi, y-lo, y-hi neighbour, -1 = physical boundary
  const int* cx0;    // x offset of the subdomain inside its problem's grid
  const int* cy0;    // y offset
  // per-subdomain problem parameters (a batch holds several independent problems
  // that share the direction table; every subdomain carries its problem's values)
  const double* hxk;  // cell widths
  const double* hyk;
  const double* dtk;  // time step
  const double* shk;  // sqrt(hx hy)
  const int* rlo;     // rank floor / lower truncation clamp (fixed mode: the rank)
  const int* rhi;     // upper truncation clamp (fixed mode: the rank)
  const int* raug;    // cap of the intermediate rank
  const int* fbase;   // first cell of the problem in the concatenated density output
  const int* fnx;     // width of the problem's grid
  // algorithmic flops per kernel slot, counted by the kernels while dd_dlra_profile_work
  // runs (null otherwise: nothing is counted)
  unsigned long long* work;
};

// Adds one CTA's algorithmic flops to the slot's counter (profiling only).
__device__ __forceinline__ void count_work(const Geo& g, int slot, double flops) {
  if (g.work && threadIdx.x == 0 && flops > 0.0)
    atomicAdd(&g.work[slot], (unsigned long long)flops);
}

// Line geometry along an axis (0 = x, 1 = y) for subdomain k.
struct Lines {
  int nlines, len, stride_line, stride_pos;
};
__device__ __forceinline__ Lines lines_of(const Geo& g, int k, int axis) {
  Lines L;
  int nx = g.nxk[k], ny = g.nyk[k];
  if (axis == 0) { L.nlines = ny; L.len = nx; L.stride_line = nx; L.stride_pos = 1; }
  else           { L.nlines = nx; L.len = ny; L.stride_line = 1; L.stride_pos = nx; }
  return L;
}
__device__ __forceinline__ int cell_of(const Lines& L, int line, int pos) {
  return line * L.stride_line + pos * L.stride_pos;
}

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Block-wide sum returned to every thread; red must hold >= 33 doubles.
__device__ __forceinline__ double block_sum(double v, double* red) {
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double t = (lane < nw) ? red[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) red[32] = t;
  }
  __syncthreads();
  return red[32];
}
// Three block-wide FP32 sums in one reduction, returned to every thread; red must hold
// >= 99 floats.
__device__ __forceinline__ void block_sum3f(float* a, float* b, float* c, float* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  float x = *a, y = *b, z = *c;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, o);
    y += __shfl_xor_sync(0xffffffffu, y, o);
    z += __shfl_xor_sync(0xffffffffu, z, o);
  }
  __syncthreads();
  if (lane == 0) { red[wid] = x; red[32 + wid] = y; red[64 + wid] = z; }
  __syncthreads();
  if (wid == 0) {
    x = lane < nw ? red[lane] : 0.f;
    y = lane < nw ? red[32 + lane] : 0.f;
    z = lane < nw ? red[64 + lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
      z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    if (lane == 0) { red[96] = x; red[97] = y; red[98] = z; }
  }
  __syncthreads();
  *a = red[96]; *b = red[97]; *c = red[98];
}

// The same order for non-negative, non-NaN values, compared by their bit patterns
// (which order as the values).
__device__ __forceinline__ void rank_sort_desc_nonneg(const double* v, int n, int* perm) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const long long x = __double_as_longlong(v[i]);
    int r = 0;
    for (int j = 0; j < n; ++j) {
      const long long y = __double_as_longlong(v[j]);
      r += (y > x) || (y == x && j < i);
    }
    perm[r] = i;
  }
}

// Spatial completion candidates (the cosine products of the completion family, by
// a + b, then a descending): at most kc_bmax(RC) of them are examined at once.
__host__ __device__ __forceinline__ int kc_bmax(int RC) { return RC + (4 * RC + 2) / 3 + 1; }
// doubles of scratch per subdomain: coefficients A (bmax x RC), B (RC x RC), then
// W = Q0^T C ((RC + 1) x bmax, the candidates' squared norms in row RC)
__host__ __device__ __forceinline__ size_t kc_region(int RC) {
  return (size_t)(kc_bmax(RC) + RC) * RC + (size_t)(RC + 1) * kc_bmax(RC);
}
// Length of the longest leading run of nc candidates that are mutually orthogonal to rel_tol
// in cosine and non-zero, from their Gram G (nc x nc, row-major, host memory): only those
// take the coefficient-space completion (a product quadrature makes the whole angular table
// so).
inline int orthogonal_prefix_gram(const double* G, int nc, double rel_tol) {
  int po = 0;
  for (; po < nc; ++po) {
    const double np = __builtin_sqrt(G[(size_t)po * nc + po]);
    bool ok = np > 0.0;
    for (int i = 0; i < po && ok; ++i)
      ok = __builtin_fabs(G[(size_t)i * nc + po]) <=
           rel_tol * __builtin_sqrt(G[(size_t)i * nc + i]) * np;
    if (!ok) break;
  }
  return po;
}

// Candidate j of an nxk x nyk subdomain: frequencies (a, b); false past the family.
__host__ __device__ __forceinline__ bool kc_cand(int j, int nxk, int nyk, int* ca, int* cb) {
  for (int d = 0; d <= nxk + nyk - 2; ++d) {
    const int ahi = d < nxk - 1 ? d : nxk - 1;
    const int alo = d - (nyk - 1) > 0 ? d - (nyk - 1) : 0;
    const int cnt = ahi - alo + 1;
    if (j < cnt) { *ca = ahi - j; *cb = d - *ca; return true; }
    j -= cnt;
  }
  return false;
}
// Candidates examined for cur0 columns done out of r_out: the missing ones plus 4 cur0 / 3
// for rejections.  The unit candidates are orthonormal, so their squared projections
// onto the span of the cur0 first columns sum to at most cur0, and a candidate rejected
// for that projection alone carries more than 3/4 of it; when the block still falls
// short, the sequential completion adds the rest.
__host__ __device__ __forceinline__ int kc_b(int nxk, int nyk, int cur0, int r_out, int RC) {
  const int need = r_out - cur0;
  if (need <= 0) return 0;
  int b = need + (4 * cur0 + 2) / 3 + 1;
  if (b > nxk * nyk) b = nxk * nyk;
  if (b > kc_bmax(RC)) b = kc_bmax(RC);
  return b;
}

// ---------------------------------------------------------------------------
// Double-float ("float-float") arithmetic: a value is the unevaluated sum hi + lo of
// two floats, |lo| <= ulp(hi)/2, about 48 significant bits.  Built from the exact
// error-free transformations of Knuth (TwoSum) and Dekker (Fast2Sum), with the product
// error taken by one FMA.  Explicit _rn intrinsics keep the compiler from contracting
// or reassociating the compensated sequences.  On this GPU FP32 issues at 64x the
// FP64 rate, so small sequential linear algebra runs several times faster this way
// than in FP64 while keeping ~1e-14 relative accuracy.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return make_float2(s, e);
}
__device__ __forceinline__ float2 df_fast_sum(float a, float b) {   // needs |a| >= |b| or a == 0
  const float s = __fadd_rn(a, b);
  return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
  const float2 s = df_two_sum(a.x, b.x);
  return df_fast_sum(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  return df_fast_sum(p, e);
}
__device__ __forceinline__ float2 df_mulf(float2 a, float b) {
  const float p = __fmul_rn(a.x, b);
  float e = __fmaf_rn(a.x, b, -p);
  e = __fmaf_rn(a.y, b, e);
  return df_fast_sum(p, e);
}
__device__ __forceinline__ float2 df_from_double(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - (double)h));
}
__device__ __forceinline__ double df_to_double(float2 a) { return (double)a.x + (double)a.y; }
__device__ __forceinline__ float2 df_shfl_xor(unsigned mask, float2 v, int o) {
  return make_float2(__shfl_xor_sync(mask, v.x, o), __shfl_xor_sync(mask, v.y, o));
}

}  // namespace dd

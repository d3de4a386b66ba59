// Small dense linear algebra of one CTA per subdomain (m <= 64): one-sided Jacobi sweeps, the
// singular value decomposition built on them, pivoted Cholesky, and the FP64 refinement of a
// symmetric eigendecomposition.
//
// These run on one SM per subdomain while the rest of the GPU waits, so what counts is latency:
// the barriers, shuffles and dependent operations of a Jacobi round, not its operations.  A
// round's m / 2 disjoint pairs of columns go to groups of 8 lanes (FP32; double-float with at most
// 32 columns) or 16 lanes (double-float beyond), a few rows per lane, columns in shared memory: two loads per row, one dot product (3 or 4
// shuffle steps), one rotation, two stores, one barrier among the warps that hold pairs.
// Measured per kernel launch with the sweeps laid out over whole warps (rows interleaved over
// the warps of the CTA, partners exchanged by shuffles, dot products summed through shared
// memory) and now, SM clocks: FP32 round 1200 -> 420 at m = 40; double-float round
// 2700 -> 900.
//
// Matrices are column-major with an odd leading dimension (lanes on consecutive rows or on
// consecutive columns both touch distinct banks).
#pragma once
#include "dd_internal.cuh"

namespace dd {

// threads of the small kernels: a pair of columns per 8 lanes up to 32 columns, per 16 beyond (the
// double-float sweeps; the FP32 ones keep 8)
__host__ __device__ __forceinline__ int small_threads(int RC) { return RC <= 32 ? 256 : 512; }
__host__ __device__ __forceinline__ int small_ld(int RC) { return RC | 1; }
// bytes of one RC-column region of 8-byte entries
__host__ __device__ __forceinline__ size_t small_region(int RC) {
  return sizeof(double) * (size_t)small_ld(RC) * RC;
}

// bytes of the region of the two FP32 matrices (columns padded to 32 or 64)
__host__ __device__ __forceinline__ size_t small_f32_region(int RC) {
  return RC <= 32 ? sizeof(float) * 2 * 36 * 32 : sizeof(float) * 2 * 68 * 64;
}

// barrier among the first n threads of the CTA (n a multiple of 32); _any also returns
// whether any of them passed a true predicate
__device__ __forceinline__ void part_sync(int n) {
  asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
}
__device__ __forceinline__ bool part_any(int n, bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
      "bar.red.or.pred q, 1, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((int)p), "r"(n)
      : "memory");
  return r != 0;
}

// Round-robin (circle method) pairing for parallel Jacobi sweeps over mm
// (even) indices: round r in [0, mm-1), pair i in [0, mm/2).  Both sums are below
// 2 (mm - 1), so each reduction modulo mm - 1 is one compare-and-subtract.
__device__ __forceinline__ void rr_pair(int mm, int r, int i, int* p, int* q) {
  const int M = mm - 1;
  if (i == 0) { *p = 0; *q = 1 + r; return; }
  int a = i + r, b = M - i + r;
  a = a >= M ? a - M : a;
  b = b >= M ? b - M : b;
  *p = 1 + a; *q = 1 + b;
}

// Rotation of a pair of columns (p, q) annihilating g = b_p . b_q, from d = |b_q|^2 - |b_p|^2:
// t = sgn(z) / (|z| + (1 + z^2)^1/2), z = d / (2g), c = (1 + t^2)^-1/2, s = c t, written
// without t: with D = |z| + (1 + z^2)^1/2, s = sgn(z) (1 + D^2)^-1/2 and c = D |s| (three
// dependent special-function operations); for |z| > 1e8, t = 1 / (2z) and c = 1.
__device__ __forceinline__ void jac_rotation(float d, float g, float* c, float* s, float* t) {
  const float z = __fdividef(d, 2.f * g);
  const float az = fabsf(z);
  const float w = __fmaf_rn(z, z, 1.f);
  const float D = az + w * rsqrtf(w);
  const float q = rsqrtf(__fmaf_rn(D, D, 1.f));
  const float iD = __fdividef(1.f, D);
  const bool huge = az > 1e8f;
  const float sg = z >= 0.f ? 1.f : -1.f;
  const float th = __fdividef(0.5f, z);
  *c = huge ? 1.f : D * q;
  *s = huge ? th : sg * q;
  *t = huge ? th : sg * iD;
}

// products below this against columns scaled to entries of order 1 are noise: rotating
// rounding noise never converges and cannot change the significant directions
#define JAC_ABS 1e-28f

// The FP32 matrices: leading dimension a multiple of 4 past 32 (64) rows, the rows past the
// matrix zero, so that a lane's four consecutive rows are one 16-byte access.
__host__ __device__ __forceinline__ int small_ldf(int RC) { return RC <= 32 ? 36 : 68; }

// FP32 sweeps of the columns of B (J, nc x nc, accumulates the rotations): a sweep rotates
// every pair with |b_p . b_q| > tol |b_p| |b_q|; the sweeps end after one in which every pair had
// |b_p . b_q| < stop |b_p| |b_q| (in the quadratic regime that leaves them at about stop^2).
// Eight lanes per pair, 4 rows (R4 = 1) or 2 x 4 rows per lane.  nrm: nc values (squared column
// norms, afresh at every sweep's start; a rotation maps them to |b_p|^2 - t g and |b_q|^2 + t g).
// Block-wide.
template <int R4>
__device__ __forceinline__ void jac_f32_t(float* B, float* J, int nc, int ld, float* nrm, float tol,
                                          float stop, int max_sweeps) {
  const int mm = nc + (nc & 1), np = mm >> 1, nt = (np * 8 + 31) & ~31;
  if (nc > 1 && (int)threadIdx.x < nt) {
    const int l = threadIdx.x & 7, pi = threadIdx.x >> 3;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
      for (int c0 = 0; c0 < nc; c0 += nt / 8) {
        const int c = c0 + pi;
        float a = 0.f;
        if (c < nc)
#pragma unroll
          for (int h = 0; h < R4; ++h) {
            const float4 x = *reinterpret_cast<const float4*>(B + c * ld + 4 * l + 32 * h);
            a = __fmaf_rn(x.x, x.x, a); a = __fmaf_rn(x.y, x.y, a);
            a = __fmaf_rn(x.z, x.z, a); a = __fmaf_rn(x.w, x.w, a);
          }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (l == 0 && c < nc) nrm[c] = a;
      }
      part_sync(nt);
      float lmax = 0.f;
      for (int r = 0; r < mm - 1; ++r) {
        int p, q;
        rr_pair(mm, r, min(pi, np - 1), &p, &q);
        const bool on = pi < np && p < nc && q < nc;
        p = min(p, nc - 1);
        q = min(q, nc - 1);
        float* bp = B + p * ld + 4 * l;
        float* bq = B + q * ld + 4 * l;
        float* jp = J + p * ld + 4 * l;
        float* jq = J + q * ld + 4 * l;
        float4 x[R4], y[R4], u[R4], v[R4];
        const float al = nrm[p], be = nrm[q];
        float g = 0.f;
#pragma unroll
        for (int h = 0; h < R4; ++h) {
          x[h] = *reinterpret_cast<const float4*>(bp + 32 * h);
          y[h] = *reinterpret_cast<const float4*>(bq + 32 * h);
        }
#pragma unroll
        for (int h = 0; h < R4; ++h) {
          u[h] = *reinterpret_cast<const float4*>(jp + 32 * h);
          v[h] = *reinterpret_cast<const float4*>(jq + 32 * h);
        }
#pragma unroll
        for (int h = 0; h < R4; ++h) {
          g = __fmaf_rn(x[h].x, y[h].x, g); g = __fmaf_rn(x[h].y, y[h].y, g);
          g = __fmaf_rn(x[h].z, y[h].z, g); g = __fmaf_rn(x[h].w, y[h].w, g);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        const float pr = al * be;
        const float rel = (on && fabsf(g) > JAC_ABS && pr > 0.f) ? fabsf(g) * rsqrtf(pr) : 0.f;
        lmax = fmaxf(lmax, rel);
        if (rel > tol) {
          float c, s, t;
          jac_rotation(be - al, g, &c, &s, &t);
          auto rot = [&](float4 a, float4 b, float* pa, float* pb) {
            *reinterpret_cast<float4*>(pa) = make_float4(c * a.x - s * b.x, c * a.y - s * b.y,
                                                         c * a.z - s * b.z, c * a.w - s * b.w);
            *reinterpret_cast<float4*>(pb) = make_float4(s * a.x + c * b.x, s * a.y + c * b.y,
                                                         s * a.z + c * b.z, s * a.w + c * b.w);
          };
#pragma unroll
          for (int h = 0; h < R4; ++h) rot(x[h], y[h], bp + 32 * h, bq + 32 * h);
#pragma unroll
          for (int h = 0; h < R4; ++h) rot(u[h], v[h], jp + 32 * h, jq + 32 * h);
          if (l == 0) {
            nrm[p] = al - t * g;
            nrm[q] = be + t * g;
          }
        }
        part_sync(nt);
      }
      if (!part_any(nt, lmax >= stop)) break;
    }
  }
  __syncthreads();
}
__device__ __forceinline__ void jac_f32(float* B, float* J, int nc, int ld, float* nrm, float tol,
                                        float stop, int max_sweeps) {
  if (ld <= 36) jac_f32_t<1>(B, J, nc, ld, nrm, tol, stop, max_sweeps);
  else jac_f32_t<2>(B, J, nc, ld, nrm, tol, stop, max_sweeps);
}

// ---- double-float accumulation ---------------------------------------------------------
// acc += a b with the product's and the sum's errors kept in acc.y (not normalised)
__device__ __forceinline__ void df_fma_acc(float2& acc, float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  const float2 s = df_two_sum(acc.x, p);
  acc.x = s.x;
  acc.y = __fadd_rn(acc.y, __fadd_rn(s.y, e));
}
__device__ __forceinline__ void df_fma_acc_f(float2& acc, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float e = __fmaf_rn(a, b, -p);
  const float2 s = df_two_sum(acc.x, p);
  acc.x = s.x;
  acc.y = __fadd_rn(acc.y, __fadd_rn(s.y, e));
}
// c x + s y
__device__ __forceinline__ float2 df_comb(float2 c, float2 x, float2 s, float2 y) {
  const float p = __fmul_rn(c.x, x.x);
  float e = __fmaf_rn(c.x, x.x, -p);
  e = __fmaf_rn(c.x, x.y, e);
  e = __fmaf_rn(c.y, x.x, e);
  const float q = __fmul_rn(s.x, y.x);
  float f = __fmaf_rn(s.x, y.x, -q);
  f = __fmaf_rn(s.x, y.y, f);
  f = __fmaf_rn(s.y, y.x, f);
  const float2 t = df_two_sum(p, q);
  return df_fast_sum(t.x, __fadd_rn(t.y, __fadd_rn(e, f)));
}
// sum over the LPP lanes of a group
template <int LPP>
__device__ __forceinline__ float2 df_group_sum(float2 v) {
#pragma unroll
  for (int o = LPP / 2; o > 0; o >>= 1) {
    const float2 w = df_shfl_xor(0xffffffffu, v, o);
    const float2 s = df_two_sum(v.x, w.x);
    v.x = s.x;
    v.y = __fadd_rn(s.y, __fadd_rn(v.y, w.y));
  }
  return df_fast_sum(v.x, v.y);
}

// Double-float sweeps (same iteration and contract): the tangent from FP32, c = (1 + t^2)^-1/2
// refined by one Newton step in double-float, so every rotation is orthogonal to double-float
// rounding.  nrm receives the squared column norms (afresh at every sweep's start and after
// the last; a rotation maps them to |b_p|^2 - t g and |b_q|^2 + t g).
template <int LPP, int R, bool WJ>
__device__ __forceinline__ void jac_df_t(float2* B, float2* J, int nr, int nc, int ld, float tol,
                                         float stop, int max_sweeps, float2* nrm) {
  const int mm = nc + (nc & 1), np = mm >> 1, nt = (np * LPP + 31) & ~31;
  const float2 z = make_float2(0.f, 0.f);
  if (nc > 0 && (int)threadIdx.x < nt) {
    const int l = threadIdx.x & (LPP - 1), pi = threadIdx.x / LPP;
    auto norms = [&] {
      for (int c0 = 0; c0 < nc; c0 += nt / LPP) {
        const int c = c0 + pi;
        float2 a = z;
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (c < nc && l + LPP * j < nr) {
            const float2 x = B[c * ld + l + LPP * j];
            df_fma_acc(a, x, x);
          }
        a = df_group_sum<LPP>(a);
        if (l == 0 && c < nc) nrm[c] = a;
      }
      part_sync(nt);
    };
    norms();
    for (int sweep = 0; sweep < max_sweeps && nc > 1; ++sweep) {
      float lmax = 0.f;
      for (int r = 0; r < mm - 1; ++r) {
        int p, q;
        rr_pair(mm, r, min(pi, np - 1), &p, &q);
        const bool on = pi < np && p < nc && q < nc;
        const float2 al = on ? nrm[p] : z, be = on ? nrm[q] : z;
        float2* bp = B + p * ld + l;
        float2* bq = B + q * ld + l;
        float2 x[R], y[R], g = z;
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const bool in = on && l + LPP * j < nr;
          x[j] = in ? bp[LPP * j] : z;
          y[j] = in ? bq[LPP * j] : z;
        }
#pragma unroll
        for (int j = 0; j < R; ++j) df_fma_acc(g, x[j], y[j]);
        g = df_group_sum<LPP>(g);
        const float pr = al.x * be.x;
        const float rel = (fabsf(g.x) > JAC_ABS && pr > 0.f) ? fabsf(g.x) * rsqrtf(pr) : 0.f;
        lmax = fmaxf(lmax, rel);
        if (on && rel > tol) {
          float c32, s32, t;
          jac_rotation(df_add(be, df_neg(al)).x, g.x, &c32, &s32, &t);
          const float2 w = df_add(make_float2(1.f, 0.f), df_mulf(make_float2(t, 0.f), t));
          const float y0 = rsqrtf(w.x);
          const float2 h = df_add(make_float2(1.f, 0.f), df_neg(df_mulf(df_mulf(w, y0), y0)));
          const float2 c = df_add(make_float2(y0, 0.f), df_mulf(h, 0.5f * y0));
          const float2 s = df_mulf(c, t), ns = df_neg(s);
#pragma unroll
          for (int j = 0; j < R; ++j)
            if (l + LPP * j < nr) {
              bp[LPP * j] = df_comb(c, x[j], ns, y[j]);
              bq[LPP * j] = df_comb(s, x[j], c, y[j]);
            }
          if (WJ) {
            float2* jp = J + p * ld + l;
            float2* jq = J + q * ld + l;
#pragma unroll
            for (int j = 0; j < R; ++j)
              if (l + LPP * j < nc) {
                const float2 u = jp[LPP * j], v = jq[LPP * j];
                jp[LPP * j] = df_comb(c, u, ns, v);
                jq[LPP * j] = df_comb(s, u, c, v);
              }
          }
          if (l == 0) {
            const float2 tg = df_mulf(g, t);
            nrm[p] = df_add(al, df_neg(tg));
            nrm[q] = df_add(be, tg);
          }
        }
        part_sync(nt);
      }
      const bool again = part_any(nt, lmax >= stop);
      norms();
      if (!again) break;
    }
  }
  __syncthreads();
}
template <bool WJ>
__device__ __forceinline__ void jac_df(float2* B, float2* J, int nr, int nc, int ld, float tol,
                                       float stop, int max_sweeps, float2* nrm) {
  const int m = max(nr, nc);
  if (m <= 16) jac_df_t<8, 2, WJ>(B, J, nr, nc, ld, tol, stop, max_sweeps, nrm);
  else if (m <= 32) jac_df_t<8, 4, WJ>(B, J, nr, nc, ld, tol, stop, max_sweeps, nrm);
  else if (m <= 48) jac_df_t<16, 3, WJ>(B, J, nr, nc, ld, tol, stop, max_sweeps, nrm);
  else jac_df_t<16, 4, WJ>(B, J, nr, nc, ld, tol, stop, max_sweeps, nrm);
}

// e -> (i <= j) of a dense enumeration of an upper triangle by columns
__device__ __forceinline__ void tri_index(int e, int* i, int* j) {
  int c = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
  c += (c + 1) * (c + 2) / 2 <= e;
  c -= c * (c + 1) / 2 > e;
  *j = c;
  *i = e - c * (c + 1) / 2;
}

// E = I - J^T J of the n x n FP32 J orthogonal to ~1e-6 (exact products, compensated sums: E
// to ~1e-14), in E (hi) and El (lo, may be null), leading dimension ld; J's is ldf
__device__ __forceinline__ void ortho_defect(const float* J, int ldf, float* E, float* El, int n, int ld) {
  for (int e = threadIdx.x; e < n * (n + 1) / 2; e += blockDim.x) {
    int i, j;
    tri_index(e, &i, &j);
    float2 x = make_float2(0.f, 0.f), y = x;
    for (int l = 0; l < n; l += 4) {
      const float4 a = *reinterpret_cast<const float4*>(J + i * ldf + l);
      const float4 b = *reinterpret_cast<const float4*>(J + j * ldf + l);
      df_fma_acc_f(x, a.x, b.x); df_fma_acc_f(y, a.y, b.y);
      df_fma_acc_f(x, a.z, b.z); df_fma_acc_f(y, a.w, b.w);
    }
    x = df_add(df_fast_sum(x.x, x.y), df_fast_sum(y.x, y.y));
    const float2 d = df_two_sum(i == j ? 1.f : 0.f, -x.x);
    const float2 v = df_fast_sum(d.x, d.y - x.y);
    E[i * ld + j] = v.x; E[j * ld + i] = v.x;
    if (El) { El[i * ld + j] = v.y; El[j * ld + i] = v.y; }
  }
  __syncthreads();
}

// Columns of W (nr x nc, double-float) orthogonal to ~1e-6 made orthogonal to double-float
// rounding, every pair at once: with g_pq = w_p . w_q and the angle t_pq that annihilates it,
// Q antisymmetric with q_pq = t_pq, W <- W (I + Q + Q^2 / 2), which is a rotation up to Q^4 / 4 (J,
// nc x nc, the same when WJ).  Cosines of 1e-6 and angles of 1e-4 leave cosines of ~1e-10 m^1/2,
// the second step those below rounding: two steps of n^2 m / 2 dot products and two small
// products take the place of two sweeps of n - 1 rounds (143000 against 281000 SM clocks at
// n = m = 60).  The angles are FP32 (an error delta in one leaves the cosine delta t), Q^2 too;
// W Q is summed in double-float.  Where two columns are so close in norm that an angle
// exceeds 2e-4 (Q^4 / 4 is then above rounding), nothing is changed and the caller's sweeps
// take over.  Q is kept exactly antisymmetric, apart from Q^2 / 2: rounding their sum in FP32
// would leave W's rotation 6e-14 off an orthogonal one.  nrm receives the squared
// column norms; Q, Q2: nc x nc FP32 scratch (leading dimension ld).  Block-wide; returns false
// where the sweeps have to finish.
template <bool WJ>
__device__ __forceinline__ bool jac_polish(float2* W, float2* J, int nr, int nc, int ld, float2* nrm,
                                           float* Q, float* Q2) {
  __shared__ unsigned pmax[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  bool more = true;
  for (int it = 0;; ++it) {
    if (threadIdx.x < 2) pmax[threadIdx.x] = 0u;
    // dot products (and norms) of all pairs; after the last step the norms alone
    const int ne = more ? nc * (nc + 1) / 2 : nc;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      int p = e, q = e;
      if (more) tri_index(e, &p, &q);
      float2 x = make_float2(0.f, 0.f), y = x;
      int l = 0;
      for (; l + 1 < nr; l += 2) {
        df_fma_acc(x, W[p * ld + l], W[q * ld + l]);
        df_fma_acc(y, W[p * ld + l + 1], W[q * ld + l + 1]);
      }
      if (l < nr) df_fma_acc(x, W[p * ld + l], W[q * ld + l]);
      x = df_add(df_fast_sum(x.x, x.y), df_fast_sum(y.x, y.y));
      if (p == q) nrm[p] = x;
      else Q[p * ld + q] = x.x;
    }
    __syncthreads();
    if (!more) return true;
    float cmax = 0.f, tmax = 0.f;
    for (int e = threadIdx.x; e < nc * (nc + 1) / 2; e += blockDim.x) {
      int p, q;
      tri_index(e, &p, &q);
      if (p == q) { Q[p * ld + p] = 0.f; continue; }
      const float g = Q[p * ld + q], pr = nrm[p].x * nrm[q].x;
      const float rel = (fabsf(g) > JAC_ABS && pr > 0.f) ? fabsf(g) * rsqrtf(pr) : 0.f;
      float t = 0.f;
      if (rel > 1e-13f) {
        float c, s;
        jac_rotation(df_add(nrm[q], df_neg(nrm[p])).x, g, &c, &s, &t);
        cmax = fmaxf(cmax, rel);
        tmax = fmaxf(tmax, fabsf(t));
      }
      Q[p * ld + q] = t;                           // row p, column q: w_q += t w_p
      Q[q * ld + p] = -t;                          // w_p -= t w_q
    }
    // (the maxima of non-negative floats by their bit patterns; NaN compares largest)
    atomicMax(&pmax[0], __float_as_uint(cmax));
    atomicMax(&pmax[1], __float_as_uint(tmax));
    __syncthreads();
    cmax = __uint_as_float(pmax[0]);
    tmax = __uint_as_float(pmax[1]);
    if (!(tmax <= 2e-4f) || it >= 6) return false;
    for (int r = warp; r < nc; r += nw)
      for (int c = lane; c < nc; c += 32) {
        float x = 0.f;
        for (int l = 0; l < nc; ++l) x = __fmaf_rn(Q[r * ld + l], Q[l * ld + c], x);
        Q2[r * ld + c] = 0.5f * x;
      }
    __syncthreads();
    // rows one by one (a warp per row: a row of the result needs only that row)
    for (int r = warp; r < nr + (WJ ? nc : 0); r += nw) {
      float2* A = r < nr ? W + r : J + (r - nr);
      float2 v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        float2 x = make_float2(0.f, 0.f), y = x;
        if (c < nc) {
          // (w + w') (q + q2): w q exactly, w' q and w q2 to FP32
          auto term = [&](float2& acc, int l) {
            const float2 w = A[l * ld];
            const float q = Q[l * ld + c];
            df_fma_acc_f(acc, w.x, q);
            acc.y = __fmaf_rn(w.y, q, __fmaf_rn(w.x, Q2[l * ld + c], acc.y));
          };
          int l = 0;
          for (; l + 1 < nc; l += 2) { term(x, l); term(y, l + 1); }
          if (l < nc) term(x, l);
          x = df_add(df_fast_sum(x.x, x.y), df_fast_sum(y.x, y.y));
          v[h] = df_add(A[c * ld], x);
        }
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (lane + 32 * h < nc) A[(lane + 32 * h) * ld] = v[h];
    }
    __syncthreads();
    more = cmax * fmaxf(4.f * tmax * sqrtf((float)nc), 2.4e-7f) > 1e-14f;
  }
}

// One-sided Jacobi of the nr x nc T (double-float, entries of order 1; its FP32 copy in B32, the
// identity in J32: leading dimension ldf, zero-padded): FP32 sweeps until the columns are
// orthogonal to ~1e-6; their rotation J made orthogonal to double-float rounding by
// J (I + E/2 + 3/8 E^2), E = I - J^T J; W = T J in double-float; jac_polish (or, where norms
// coincide, double-float sweeps) finishes.  T's entries are rounded pairs (df_from_double): split by
// integer operations, hi truncated, they carried two bits less, and a step's density was 5.9e-15 off
// 64 bits where it is 4.1e-15 off now (geometric mean over 64 smooth states of 31 x 29 cells,
// r = 5); the conversions cost 0.4% of a step.  W (nr x nc) in R2, J (nc x nc; as rotated by the last
// steps when WJ) in R3, squared column norms in nrm.  T, R2, R3: leading dimension ld.
template <bool WJ>
__device__ __forceinline__ void jacobi_core(const float2* T, float* B32, float* J32, double* R2,
                                            double* R3, int nr, int nc, int ld, int ldf, float2* nrm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float2* W = reinterpret_cast<float2*>(R2);
  float2* Jd = reinterpret_cast<float2*>(R3);
  jac_f32(B32, J32, nc, ldf, reinterpret_cast<float*>(nrm), 1e-6f, 1e-3f, 30);
  // F = E/2 + 3/8 E^2 as double-float in R2, E in R3
  float* E = reinterpret_cast<float*>(R3);
  float* El = E + (size_t)ld * nc;
  ortho_defect(J32, ldf, E, El, nc, ld);
  float2* F = W;
  for (int c = warp; c < nc; c += nw)
    for (int r = lane; r < nc; r += 32) {
      float x = 0.f;
#pragma unroll 4
      for (int l = 0; l < nc; ++l) x = __fmaf_rn(E[c * ld + l], E[l * ld + r], x);
      F[c * ld + r] = df_add(make_float2(0.5f * E[c * ld + r], 0.5f * El[c * ld + r]),
                             make_float2(0.375f * x, 0.f));
    }
  __syncthreads();
  for (int c = warp; c < nc; c += nw)                   // Jd = J + J F
    for (int r = lane; r < nc; r += 32) {
      float2 x = make_float2(0.f, 0.f), y = x;
      int l = 0;
      for (; l + 1 < nc; l += 2) {
        df_fma_acc(x, make_float2(J32[l * ldf + r], 0.f), F[c * ld + l]);
        df_fma_acc(y, make_float2(J32[(l + 1) * ldf + r], 0.f), F[c * ld + l + 1]);
      }
      if (l < nc) df_fma_acc(x, make_float2(J32[l * ldf + r], 0.f), F[c * ld + l]);
      x = df_add(df_fast_sum(x.x, x.y), df_fast_sum(y.x, y.y));
      Jd[c * ld + r] = df_add(make_float2(J32[c * ldf + r], 0.f), x);
    }
  __syncthreads();
  for (int c = warp; c < nc; c += nw)                   // W = T J
    for (int r = lane; r < nr; r += 32) {
      float2 x = make_float2(0.f, 0.f), y = x;
      int l = 0;
      for (; l + 1 < nc; l += 2) {
        df_fma_acc(x, T[l * ld + r], Jd[c * ld + l]);
        df_fma_acc(y, T[(l + 1) * ld + r], Jd[c * ld + l + 1]);
      }
      if (l < nc) df_fma_acc(x, T[l * ld + r], Jd[c * ld + l]);
      W[c * ld + r] = df_add(df_fast_sum(x.x, x.y), df_fast_sum(y.x, y.y));
    }
  __syncthreads();
  if (!jac_polish<WJ>(W, Jd, nr, nc, ld, nrm, B32, B32 + (size_t)ld * nc))
    jac_df<WJ>(W, Jd, nr, nc, ld, 1e-13f, 3e-7f, 10, nrm);
}

// SVD of the m x m column-major FP64 B (leading dimension ld, region R0) by one-sided Jacobi,
// accurate to about 1e-13 |B|, on a power-of-two scaled copy (jacobi_core).
// On return W = 2^-ex B J (orthogonal columns, squared norms in nrm) and J (orthogonal) are in
// R2 and R3 (float2) and B is overwritten; the function returns ex.  A zero or non-finite B
// returns J = I, W = B, ex = 0.  R0, R2, R3: regions of 8-byte entries; R1: the FP32 region.
// Block-wide.
static __device__ __noinline__ int svd_jacobi(double* R0, float* R1, double* R2, double* R3, int m,
                                              int ld, int ldf, float2* nrm) {
  __shared__ long long rbits[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float* B32 = R1;
  float* J32 = B32 + (size_t)ldf * (ldf - 4);
  float2* T = reinterpret_cast<float2*>(R0);
  float2* W = reinterpret_cast<float2*>(R2);
  float2* Jd = reinterpret_cast<float2*>(R3);
  long long mb = 0;                                     // largest |x| by its bit pattern
  for (int c = warp; c < m; c += nw)
    for (int r = lane; r < m; r += 32)
      mb = max(mb, __double_as_longlong(R0[c * ld + r]) & 0x7fffffffffffffffll);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  if (lane == 0) rbits[warp] = mb;
  __syncthreads();
  mb = 0;
  for (int w = 0; w < nw; ++w) mb = max(mb, rbits[w]);
  const bool ok = mb > 0 && mb < 0x7ff0000000000000ll;
  const int ex = ok ? ilogb(__longlong_as_double(mb)) : 0;
  for (int c = warp; c < m; c += nw)
    for (int r = lane; r < ldf - 4; r += 32) {
      float2 x = make_float2(0.f, 0.f);
      if (r < m) {
        x = df_from_double(scalbn(R0[c * ld + r], -ex));
        T[c * ld + r] = x;
      }
      B32[c * ldf + r] = x.x;
      J32[c * ldf + r] = c == r ? 1.f : 0.f;
    }
  __syncthreads();
  if (!ok) {
    for (int c = warp; c < m; c += nw) {
      for (int r = lane; r < m; r += 32) {
        W[c * ld + r] = T[c * ld + r];
        Jd[c * ld + r] = make_float2(c == r ? 1.f : 0.f, 0.f);
      }
      // the norm of a zero column, or a non-finite one for the caller's check
      if (lane == 0) nrm[c] = make_float2(mb > 0 ? __int_as_float(0x7f800000) : 0.f, 0.f);
    }
    __syncthreads();
    return 0;
  }
  jacobi_core<true>(T, B32, J32, R2, R3, m, m, ld, ldf, nrm);
  return ex;
}

// Pivoted Cholesky of the m x m (m <= 64) positive semidefinite A (lower triangle: entry
// (i, j), i >= j, at i * ld + j; overwritten by its Schur complements): A = X D^-1 X^T up to a
// remainder whose diagonal is <= thr_rel times the largest diagonal entry of A.  Column t of
// X (column-major, leading dimension ld, rows in the original order) is the pivot column of
// step t, dp[t] its pivot (the Cholesky factor's column is X_t / sqrt(dp[t])).  The pivot is
// the largest remaining positive normal diagonal entry, by the upper 32 bits of its pattern,
// lowest index on ties.  Block-wide; returns the number of columns.
//
// On this GPU one FP64 warp instruction holds the SM's FP64 pipe for ~16 cycles whatever the
// number of active lanes, and a dependent one waits longer still, so a step keeps its chain
// short: warp 0 holds the diagonal in registers and picks the next pivot and its reciprocal
// while the warps of the other three schedulers update the remaining pairs (i > j), enumerated
// densely.  2200-4500 clocks per step with a square root and two reductions in the chain
// before, 600-900 now up to 20 columns, 1900 at 60 (the update's pairs).  (The reciprocal is the
// division: Newton steps on an FP32 one gave the same densities, and steps 1.2% longer.)
__device__ __forceinline__ int pchol(double* A, double* X, int m, int ld, double thr_rel,
                                     double* dp) {
  __shared__ double cv[64], wv[64];
  __shared__ int perm[64], pos[64], piv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool lead = warp == 0;
  double d0 = 0.0, d1 = 0.0, inv = 0.0, thr = 0.0;     // warp 0: diagonal of rows lane, lane + 32
  bool o0 = lane < m, o1 = lane + 32 < m;              // not yet pivoted
  int b = -1;
  auto pick = [&](int k) {                             // warp 0: next pivot b, its reciprocal
    const int h0 = __double2hiint(d0), h1 = __double2hiint(d1);
    const unsigned k0 = (o0 && h0 >= 0x00100000 && h0 < 0x7ff00000) ? (unsigned)h0 : 0u;
    const unsigned k1 = (o1 && h1 >= 0x00100000 && h1 < 0x7ff00000) ? (unsigned)h1 : 0u;
    const unsigned best = __reduce_max_sync(0xffffffffu, max(k0, k1));
    const unsigned b0 = __ballot_sync(0xffffffffu, best && k0 == best);
    const unsigned b1 = __ballot_sync(0xffffffffu, best && k1 == best);
    b = b0 ? __ffs(b0) - 1 : (b1 ? 31 + __ffs(b1) : -1);
    const double dv0 = __shfl_sync(0xffffffffu, d0, b & 31), dv1 = __shfl_sync(0xffffffffu, d1, b & 31);
    const double d = b < 32 ? dv0 : dv1;
    if (k == 0) thr = b >= 0 ? thr_rel * d : 0.0;
    // (positive doubles order as their bits)
    if (b >= 0 && __double_as_longlong(d) <= __double_as_longlong(thr)) b = -1;
    if (b >= 0) {
      inv = 1.0 / d;
      if (lane == 0) dp[k] = d;
    }
    if (lane == 0) piv = b;
  };
  if (lead) {
    if (o0) { d0 = A[lane * ld + lane]; perm[lane] = lane; pos[lane] = lane; }
    if (o1) { d1 = A[(lane + 32) * ld + lane + 32]; perm[lane + 32] = lane + 32; pos[lane + 32] = lane + 32; }
    __syncwarp();
    pick(0);
  }
  int k = 0;
  __syncthreads();
  for (; k < m; ++k) {
    if (piv < 0) break;
    double w0 = 0.0, w1 = 0.0, c0 = 0.0, c1 = 0.0;
    if (lead) {                                        // the pivot column and its scaled copy
      if (o0) {
        c0 = lane == b ? d0 : A[max(lane, b) * ld + min(lane, b)];
        w0 = c0 * inv;
        cv[lane] = c0; wv[lane] = w0;
      }
      if (o1) {
        c1 = lane + 32 == b ? d1 : A[max(lane + 32, b) * ld + min(lane + 32, b)];
        w1 = c1 * inv;
        cv[lane + 32] = c1; wv[lane + 32] = w1;
      }
      if (lane < m) X[k * ld + lane] = c0;             // zero in the rows already pivoted
      if (lane + 32 < m) X[k * ld + lane + 32] = c1;
      if (lane == 0) {                                 // the pivot to place k of the order
        const int pb = pos[b], o = perm[k];
        perm[k] = b; perm[pb] = o;
        pos[o] = pb; pos[b] = k;
      }
      if (lane == b) o0 = false;
      if (lane + 32 == b) o1 = false;
    }
    __syncthreads();
    if (lead) {
      d0 = fma(-c0, w0, d0);
      d1 = fma(-c1, w1, d1);
      if (k + 1 < m) pick(k + 1);
    } else if (warp & 3) {                             // (the other scheduler is warp 0's alone)
      const int na = m - k - 1, ne = na * (na - 1) / 2, nu = (blockDim.x >> 7) * 96;
      for (int e = ((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane; e < ne; e += nu) {
        int a, c;
        tri_index(e, &a, &c);                          // a <= c: the pair (a, c + 1)
        const int i = perm[k + 1 + a], j = perm[k + 2 + c];
        const int hi = max(i, j), lo = min(i, j);
        A[hi * ld + lo] = fma(-cv[hi], wv[lo], A[hi * ld + lo]);
      }
    }
    __syncthreads();
  }
  return k;
}

// The smallest r whose tail (sum_{t >= r} sigma_t^2)^1/2 is within tol, for n <= 64 values by
// val(t), descending (one warp; every lane returns it).  A suffix sum over the lanes: 13
// dependent FP64 operations, where a sum per r afresh took n^2 / 2 and a square root each.
// (The root is compared, not the square with tol^2: a tolerance below zero cuts nothing.)
template <class F>
__device__ __forceinline__ int tail_rank(int n, double tol, F val) {
  const int lane = threadIdx.x & 31;
  double a = lane < n ? val(lane) : 0.0, b = lane + 32 < n ? val(lane + 32) : 0.0;
  a *= a;
  b *= b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_down_sync(0xffffffffu, a, o), v = __shfl_down_sync(0xffffffffu, b, o);
    if (lane + o < 32) { a += u; b += v; }
  }
  a += __shfl_sync(0xffffffffu, b, 0);
  const unsigned in0 = __ballot_sync(0xffffffffu, sqrt(a) <= tol || lane >= n);
  const unsigned in1 = __ballot_sync(0xffffffffu, sqrt(b) <= tol || lane + 32 >= n);
  if (in0) return min(n, __ffs(in0) - 1);
  if (in1) return min(n, 31 + __ffs(in1));
  return n;
}

// One FP64 refinement step of approximate eigenvectors of a symmetric matrix (Ogita and
// Aishima, 2018): with R = I - V^T V, S = V^T G V, lambda_i = s_ii / (1 - r_ii),
// V <- V (I + E), e_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i) for separated pairs,
// r_ij / 2 within clusters and on the diagonal; the error of V maps to about its square.
// G (symmetric) and V (V_ij = V[j * ld + i], refined in place): leading dimension ld; lam: the
// refined eigenvalues (not sorted).  S and R are symmetric (upper triangles computed,
// mirrored); the norms that set the cluster threshold, the quotients of E (a first-order
// correction) and the product V E are taken in FP32.  T, S, R: regions of scratch.  Block-wide.
static __device__ __noinline__ void refine_sym_eig(const double* G, double* V, double* lam, int m,
                                                   int ld, double* T, double* S, double* R) {
  __shared__ double rred[50];            // >= 99 floats for block_sum3f
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {            // T = G V
    const int j = e / m, i = e - j * m;
    double x = 0.0;
    for (int l = 0; l < m; ++l) x += G[l * ld + i] * V[j * ld + l];
    T[j * ld + i] = x;
  }
  __syncthreads();
  float offn = 0.f, rn = 0.f, gn = 0.f;
  const int ntri = m * (m + 1) / 2;
  for (int e = threadIdx.x; e < ntri; e += blockDim.x) {             // S = V^T T, R = I - V^T V
    int i, j;
    tri_index(e, &i, &j);
    double x = 0.0, y = 0.0;
    for (int l = 0; l < m; ++l) {
      const double v = V[i * ld + l];
      x += v * T[j * ld + l];
      y += v * V[j * ld + l];
    }
    const double rr = (i == j ? 1.0 : 0.0) - y;
    S[i * ld + j] = x; S[j * ld + i] = x;
    R[i * ld + j] = rr; R[j * ld + i] = rr;
    const float xf = (float)x, rf = (float)rr, gf = (float)G[i * ld + j];
    const float wgt = i == j ? 1.f : 2.f;
    if (i != j) offn += 2.f * xf * xf;
    rn += wgt * rf * rf;
    gn += wgt * gf * gf;
  }
  block_sum3f(&offn, &rn, &gn, reinterpret_cast<float*>(rred));
  const float delta = 2.f * (sqrtf(offn) + sqrtf(gn) * sqrtf(rn));   // cluster separation
  for (int i = threadIdx.x; i < m; i += blockDim.x) lam[i] = S[i * ld + i] / (1.0 - R[i * ld + i]);
  __syncthreads();
  float* Ef = reinterpret_cast<float*>(T);      // E in FP32 (T = G V is dead)
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const int j = e / m, i = e - j * m;
    float x = (float)(0.5 * R[i * ld + j]);
    if (i != j) {
      const float d = (float)(lam[j] - lam[i]);
      if (fabsf(d) > delta) x = __fdividef((float)(S[i * ld + j] + lam[j] * R[i * ld + j]), d);
    }
    Ef[j * ld + i] = x;
  }
  __syncthreads();
  float* Vf = reinterpret_cast<float*>(R);      // V in FP32 (R is dead)
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const int j = e / m, i = e - j * m;
    Vf[j * ld + i] = (float)V[j * ld + i];
  }
  __syncthreads();
  // V + V E with the correction V E in FP32 (E is itself a first-order FP32 quantity of the
  // size of V's error, so FP32 rounding of V E lies far below FP64 rounding of V)
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const int j = e / m, i = e - j * m;
    float x = 0.f;
    for (int l = 0; l < m; ++l) x = __fmaf_rn(Vf[l * ld + i], Ef[j * ld + l], x);
    V[j * ld + i] += (double)x;
  }
  __syncthreads();
}

}  // namespace dd

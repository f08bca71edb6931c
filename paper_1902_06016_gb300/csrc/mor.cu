// Model-order reduction of the MIMO system (Eqs. gfcclineqn and model) on the GPU, FP64.
//
// * Subspace: S holds orthonormalised solutions X_p(w_k). New columns lose their components along
//   the current S by block classical Gram-Schmidt (two passes), then within the block panel by panel:
//   Cholesky QR twice for well-conditioned panels, otherwise column by column (two passes); a column is
//   kept when its norm after the passes is >= drop_tol times its norm before, else dropped.
//   Orthonormality is in the complex inner product, so the projections written S^T in Eq. model are
//   applied as S^H.
// * Z = M S comes for free: every solved column satisfies M x = b - (w - i eta) x - r with the FP64
//   residual r of the solver, and every linear combination applied to S is applied to Z as well.
// * Reduced model: Hhat = S^H Z, bhat = S^H b, chat = c^T S, updated incrementally.
// * Evaluation at many frequencies: Hhat is reduced once to upper Hessenberg form by Householder
//   reflections (applied alongside to bhat, chat and the residual coefficients); each frequency is
//   then an O(m^2 np) shifted Hessenberg solve (partial pivoting between adjacent rows, then a blocked back
//   substitution). Ghat_pq = chat_q^T yhat_p for all frequencies is one complex GEMM, and A = -(1/pi) sum_p
//   Im Ghat_pp.
// * Residual estimate for refinement: the columns of [B, S, Z] are kept as coefficients in an
//   orthonormal basis Q of their span (extended with every new block), so that the residual
//   r = (w - i eta) S y + Z y - b has the coefficient vector (w - i eta) R_S y + R_Z y - R_B e_p and
//   ||r|| is its 2-norm, without the cancellation of a Gram-matrix formula; the coefficients of all
//   frequencies are two complex GEMMs.
#include "gfcc_internal.cuh"
#include "ozaki.cuh"

#include <algorithm>
#include <cmath>

namespace gfcc {
namespace {

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)std::min<long long>(std::max<long long>(g, 1), 152LL * 32);
}

__device__ __forceinline__ cplx cz() { return make_cuDoubleComplex(0.0, 0.0); }

// dst[nu][off + k] = src[nu][cols[k]]
__global__ void append_cols_kernel(const cplx* __restrict__ src, int lds, const int* __restrict__ cols, int nk,
                                   cplx* __restrict__ dst, int ldd, int off, long long D) {
  long long total = D * nk;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int k = (int)(t % nk);
    long long nu = t / nk;
    dst[nu * ldd + off + k] = src[nu * lds + cols[k]];
  }
}

// ---- Householder reduction to Hessenberg form (column-major matrices) ---------------------------
// v = x - alpha e1 with alpha = -e^{i arg x0} ||x||, tau = 2 / ||v||^2; stores v in vbuf[0..len), tau in *tau
__global__ void house_kernel(const cplx* __restrict__ x, int len, cplx* __restrict__ v, double* __restrict__ tau) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < len; i += blockDim.x) s = fma(x[i].x, x[i].x, fma(x[i].y, x[i].y, s));
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  double nx = sqrt(red[0]);
  cplx x0 = x[0];
  double a0 = cuCabs(x0);
  cplx ph = a0 > 0.0 ? make_cuDoubleComplex(x0.x / a0, x0.y / a0) : make_cuDoubleComplex(1.0, 0.0);
  cplx alpha = make_cuDoubleComplex(-ph.x * nx, -ph.y * nx);
  for (int i = threadIdx.x; i < len; i += blockDim.x) v[i] = x[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    v[0] = cuCsub(x0, alpha);
    double vn2 = red[0] - (x0.x * x0.x + x0.y * x0.y) + (v[0].x * v[0].x + v[0].y * v[0].y);
    *tau = (nx > 0.0 && vn2 > 0.0) ? 2.0 / vn2 : 0.0;
  }
}
// A reflection H = I - tau v v^H applied to several column-major matrices at once (one launch per side
// and Householder step):
//   left:  A[r0+i][col] -= tau v[i] (sum_k conj(v[k]) A[r0+k][col]) on the columns of A (from c0a) and B
//   right: w[row] = sum_k A[row][c0+k] v[k]; A[row][c0+k] -= tau w[row] conj(v[k]) on up to four matrices
struct RightMats {
  cplx* p[4];
  long long ld[4];
  int rows[4];
  int n;
};
__global__ void house_left2_kernel(cplx* __restrict__ A, long long lda, int c0a, int na, cplx* __restrict__ B,
                                   long long ldb, int nbc, int r0, int len, const cplx* __restrict__ v,
                                   const double* __restrict__ tau) {
  __shared__ cplx red[256];
  const bool inA = (int)blockIdx.x < na;
  cplx* a = inA ? A + (long long)(c0a + blockIdx.x) * lda + r0 : B + (long long)(blockIdx.x - na) * ldb + r0;
  (void)nbc;
  cplx sdot = cz();
  for (int i = threadIdx.x; i < len; i += blockDim.x) {
    const cplx vv = v[i], aa = a[i];
    sdot.x = fma(vv.x, aa.x, fma(vv.y, aa.y, sdot.x));
    sdot.y = fma(vv.x, aa.y, fma(-vv.y, aa.x, sdot.y));
  }
  red[threadIdx.x] = sdot;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) { red[threadIdx.x].x += red[threadIdx.x + w].x; red[threadIdx.x].y += red[threadIdx.x + w].y; }
    __syncthreads();
  }
  const cplx wsum = red[0];
  const double t = *tau;
  for (int i = threadIdx.x; i < len; i += blockDim.x) {
    const cplx d = cuCmul(v[i], wsum);
    a[i].x -= t * d.x;
    a[i].y -= t * d.y;
  }
}
// w[k][row] = sum_j A_k[row][c0 + j] v[j] for every matrix k and row (w rows stacked, matrix k at woff[k])
// w[row] = sum_j A[row][c0 + j] v[j] over the rows of all right-side matrices: a block takes a tile of 32
// rows (lanes, coalesced along the column-major rows) and its 8 warps split the reflector's length, so
// that short and long reflectors alike keep many warps in flight; the warps' sums meet in shared memory
__global__ void __launch_bounds__(256) house_right_w4_kernel(RightMats m, int c0, int len, const cplx* __restrict__ v,
                                                             cplx* __restrict__ w) {
  __shared__ cplx red[8][32];
  int t = blockIdx.x, k = 0, off = 0;
  while (k < m.n) {   // tile t -> matrix k (tiles do not cross matrices)
    const int nt = (m.rows[k] + 31) / 32;
    if (t < nt) break;
    t -= nt;
    off += m.rows[k];
    ++k;
  }
  if (k >= m.n) return;   // uniform for the whole block
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int row = t * 32 + lane;
  const bool ok = row < m.rows[k];
  const cplx* A = m.p[k];
  cplx sum = cz();
  if (ok)
    for (int j = wid; j < len; j += 8) sum = cuCadd(sum, cuCmul(A[(long long)(c0 + j) * m.ld[k] + row], v[j]));
  red[wid][lane] = sum;
  __syncthreads();
  if (wid == 0 && ok) {
    cplx r = red[0][lane];
    for (int q = 1; q < 8; ++q) r = cuCadd(r, red[q][lane]);
    w[off + row] = r;
  }
}
// A_k[row][c0 + j] -= tau w[k][row] conj(v[j])
__global__ void house_right_update4_kernel(RightMats m, int c0, int len, const cplx* __restrict__ v,
                                           const cplx* __restrict__ w, const double* __restrict__ tau, long long total) {
  const double t = *tau;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    long long r = q;
    int k = 0, off = 0;
    while (k < m.n && r >= (long long)m.rows[k] * len) { r -= (long long)m.rows[k] * len; off += m.rows[k]; ++k; }
    if (k >= m.n) return;
    const int row = (int)(r % m.rows[k]), j = (int)(r / m.rows[k]);
    const cplx d = cuCmul(w[off + row], cuConj(v[j]));
    cplx* p = m.p[k] + (long long)(c0 + j) * m.ld[k] + row;
    p->x -= t * d.x;
    p->y -= t * d.y;
  }
}

// Y[r0 + i][n] -= tau v[i] sum_k conj(v[k]) Y[r0 + k][n] for every column n < N (Y row-major, ld ldy)
__global__ void house_rows_kernel(cplx* __restrict__ Y, long long ldy, long long N, int r0, int len,
                                  const cplx* __restrict__ v, const double* __restrict__ tau) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= N) return;
  cplx sdot = cz();
  for (int k = 0; k < len; ++k) {
    const cplx vv = v[k], yy = Y[(long long)(r0 + k) * ldy + n];
    sdot.x = fma(vv.x, yy.x, fma(vv.y, yy.y, sdot.x));
    sdot.y = fma(vv.x, yy.y, fma(-vv.y, yy.x, sdot.y));
  }
  const double t = *tau;
  for (int k = 0; k < len; ++k) {
    const cplx d = cuCmul(v[k], sdot);
    Y[(long long)(r0 + k) * ldy + n].x -= t * d.x;
    Y[(long long)(r0 + k) * ldy + n].y -= t * d.y;
  }
}

// ---- per-frequency shifted Hessenberg solves -------------------------------------------------------
// (w - i eta + H) y_p = b_p for every frequency w and right-hand side p in two kernels: the elimination,
// one CTA per frequency, leaves U (double-float, in 32 x 32 tiles) and the transformed right-hand sides;
// the back substitution, one CTA per frequency and group of right-hand sides, is a blocked triangular solve.
struct EvalArgs {
  int m, np, nw;
  const cplx* H;      // m x m row-major, upper Hessenberg
  const cplx* b;      // m x np row-major; null: the right-hand sides are in Y (per frequency), solved in place
  const double* omegas;
  double eta;
  float4* U;          // per frequency: tiles (J, K), J <= K, of 32 x 32 entries at (K(K+1)/2 + J) * 1024
  cplx* dU;           // per frequency: the diagonal of U in FP64 (m)
  cplx* Y;            // solutions: Y[k * ldy + w * np + p] = yhat_p(w)[k]
  long long ldy;
  int* singular;
};
constexpr int ET = 32;   // tile edge of U
__host__ __device__ constexpr long long eval_tiles(int m) {
  return (long long)((m + ET - 1) / ET) * ((m + ET - 1) / ET + 1) / 2;
}

// ---- double-float arithmetic (value = h + l, two FP32 numbers) ------------------------------------
// GB300 issues FP32 operations at many times its FP64 rate, so the O(m^2 np) back substitution runs
// on pairs of floats (about 48 significant bits; Dekker 1971, Knuth's two-sum). The explicitly
// rounded intrinsics keep the compiler from contracting the error-free transformations.
struct df2 {
  float h, l;
};
__device__ __forceinline__ df2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ df2 fast_two_sum(float a, float b) {   // |a| >= |b| or a == 0
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df2 df_from(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_to(float h, float l) { return (double)h + (double)l; }
// c + a1 b1 + a2 b2 (all double-float): the leading products exactly (fma), the rest in FP32
__device__ __forceinline__ df2 df_dot2(df2 c, df2 a1, df2 b1, df2 a2, df2 b2) {
  const float p1 = __fmul_rn(a1.h, b1.h), p2 = __fmul_rn(a2.h, b2.h);
  const float e1 = __fmaf_rn(a1.h, b1.h, -p1), e2 = __fmaf_rn(a2.h, b2.h, -p2);
  float cross = __fmul_rn(a2.l, b2.h);
  cross = __fmaf_rn(a2.h, b2.l, cross);
  cross = __fmaf_rn(a1.l, b1.h, cross);
  cross = __fmaf_rn(a1.h, b1.l, cross);
  const df2 s1 = two_sum(c.h, p1);
  const df2 s2 = two_sum(s1.h, p2);
  float low = __fadd_rn(c.l, e1);
  low = __fadd_rn(low, e2);
  low = __fadd_rn(low, cross);
  low = __fadd_rn(low, s1.l);
  low = __fadd_rn(low, s2.l);
  return fast_two_sum(s2.h, low);
}
// complex double-float in a float4 (re.h, re.l, im.h, im.l)
__device__ __forceinline__ float4 dfc_from(cplx z) {
  const df2 r = df_from(z.x), i = df_from(z.y);
  return make_float4(r.h, r.l, i.h, i.l);
}
__device__ __forceinline__ cplx dfc_to(float4 v) { return make_cuDoubleComplex(df_to(v.x, v.y), df_to(v.z, v.w)); }
// c - u y
__device__ __forceinline__ float4 dfc_sub_mul(float4 c, float4 u, float4 y) {
  const df2 cr{c.x, c.y}, ci{c.z, c.w};
  const df2 nur{-u.x, -u.y}, ui{u.z, u.w}, nui{-u.z, -u.w};
  const df2 yr{y.x, y.y}, yi{y.z, y.w};
  const df2 r = df_dot2(cr, nur, yr, ui, yi);     // cr - ur yr + ui yi
  const df2 i = df_dot2(ci, nur, yi, nui, yr);    // ci - ur yi - ui yr
  return make_float4(r.h, r.l, i.h, i.l);
}

// df_from without FP64 arithmetic: h is x rounded to 24 bits (half up), l the rest rounded to 24 bits, both cut
// out of the bit pattern (the same split up to the direction of exact ties). Outside the range of normal
// FP32 numbers x is converted alone.
__device__ __forceinline__ df2 df_split(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFULL;
  const int e = (int)(b >> 52);
  if (e < 897 || e > 1149) return {(float)x, 0.f};
  const unsigned long long r = (b + 0x10000000ULL) & ~0x1FFFFFFFULL;   // rounded to 23 mantissa bits
  const int low = (int)(long long)(b - r);                             // in [-2^28, 2^28), times 2^(e - 1075)
  const unsigned sign = (unsigned)((unsigned long long)__double_as_longlong(x) >> 32) & 0x80000000u;
  const unsigned hb = (unsigned)(r >> 29) - (896u << 23);
  const int k = (e - 1075) >> 1;   // the scale in two factors, each a normal number
  const float l = (float)low * __uint_as_float((unsigned)(k + 127) << 23) *
                  __uint_as_float((unsigned)(e - 1075 - k + 127) << 23);
  return {__uint_as_float(hb | sign), __uint_as_float(__float_as_uint(l) ^ sign)};
}
__device__ __forceinline__ float4 dfc_split(cplx z) {
  const df2 r = df_split(z.x), i = df_split(z.y);
  return make_float4(r.h, r.l, i.h, i.l);
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool on) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gmem), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// bits of max(|re|, |im|): non-negative doubles order like their bit patterns
__device__ __forceinline__ unsigned long long max_bits(cplx z) {
  const unsigned long long a = (unsigned long long)__double_as_longlong(z.x) & 0x7FFFFFFFFFFFFFFFULL;
  const unsigned long long b = (unsigned long long)__double_as_longlong(z.y) & 0x7FFFFFFFFFFFFFFFULL;
  return a > b ? a : b;
}
// x / p for the elimination: x conj(p) / |p|^2 with p scaled to order one by a power of two and the reciprocal by
// two Newton steps from an FP32 seed. 15 FP64 operations in a chain of 10, where the library's complex division
// is two FP64 divisions one after the other: an FP64 instruction holds a scheduler for 75 clocks on this
// GPU (measured 1.7 lanes per clock and SM) and the division is the serial part of every elimination step.
__device__ __forceinline__ cplx cdiv_newton(cplx x, cplx p) {
  const int e = (int)(max_bits(p) >> 52);
  if (e < 100 || e > 1946) return cuCdiv(x, p);   // near the ends of the exponent range
  const double s = __longlong_as_double((long long)(2046 - e) << 52);   // 2^(1023 - e)
  const double a = p.x * s, b = p.y * s;
  const double d = fma(a, a, b * b);   // in [1, 8)
  double r = (double)(1.0f / (float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  r = fma(r, fma(-d, r, 1.0), r);
  r *= s;
  return make_cuDoubleComplex(fma(x.x, a, x.y * b) * r, fma(x.y, a, -(x.x * b)) * r);
}

// Elimination, one CTA per frequency: LU of (w - i eta + H) with partial pivoting between adjacent rows
// (the only pivots a Hessenberg matrix needs), in FP64, the np right-hand sides carried along as np more
// columns. Only one row is carried from step to step (in shared memory, every thread owning the columns
// it alone reads and writes), and the rows still to come arrive by cp.async EF_RING - 1 steps ahead. The
// chain of a step is the pivot of its owner thread (an FP64 division) and one barrier; everything else
// (two FP64 multiply-adds per column, the split to double-float) is in its shadow. RING = false (rows too
// long for shared memory) reads each row when it is needed and carries the row in global memory (m + np
// entries per frequency of EvalScratch::rows).
constexpr int EF_T = 128, EF_RING = 4;
template <bool RING>
__global__ void __launch_bounds__(EF_T) eval_factor_kernel(EvalArgs a, int w0, cplx* __restrict__ rows) {
  extern __shared__ float4 ef_sm[];
  __shared__ cplx s_l[2];
  __shared__ int s_swap[2];
  const int m = a.m, np = a.np, n = m + np, f = blockIdx.x, w = w0 + f, tid = threadIdx.x;
  const cplx sig = make_cuDoubleComplex(a.omegas[w], -a.eta);
  cplx* cur = RING ? reinterpret_cast<cplx*>(ef_sm) : rows + (long long)f * n;
  cplx* ring = reinterpret_cast<cplx*>(ef_sm) + n;
  cplx* R = a.Y + (long long)w * np;   // row k at R[k * ldy]
  float4* U = a.U + (long long)f * eval_tiles(m) * (ET * ET);
  cplx* dU = a.dU + (long long)f * m;
  auto src = [&](int r, int col) -> const cplx* {
    if (col < m) return a.H + (long long)r * m + col;
    return a.b ? a.b + (long long)r * np + (col - m) : R + (long long)r * a.ldy + (col - m);
  };
  // the thread's own columns of row r (columns before r - 1 are zero and never read)
  auto issue = [&](int r) {
    if (RING && r < m) {
      cplx* d = ring + (long long)(r % EF_RING) * n;
      for (int col = tid; col < n; col += EF_T)
        if (col >= r - 1) cp_async16(d + col, src(r, col), true);
    }
    cp_async_commit();
  };
  auto next = [&](int r, int col) { return RING ? ring[(long long)(r % EF_RING) * n + col] : *src(r, col); };
  // pivot of step j from the carried row's entry c: swap and multiplier (owner of column j)
  auto pivot = [&](int j, cplx c) {
    cplx l = cz();
    int swap = 0;
    if (j + 1 < m) {
      const cplx x = next(j + 1, j);
      swap = max_bits(x) > max_bits(c);
      const cplx piv = swap ? x : c;
      if (piv.x == 0.0 && piv.y == 0.0) atomicExch(a.singular, 1);
      else l = cdiv_newton(swap ? c : x, piv);
    }
    s_l[j & 1] = l;
    s_swap[j & 1] = swap;
  };
  for (int r = 1; r < EF_RING; ++r) issue(r);   // rows 1 .. EF_RING - 1
  for (int col = tid; col < n; col += EF_T) {
    cplx h = *src(0, col);
    if (col == 0) h = cuCadd(h, sig);
    cur[col] = h;
  }
  cp_async_wait<EF_RING - 2>();   // row 1
  if (tid == 0) pivot(0, cur[0]);
  for (int j = 0; j < m; ++j) {
    __syncthreads();
    const cplx l = s_l[j & 1];
    const int swap = s_swap[j & 1];
    const bool last = j + 1 == m;
    cp_async_wait<EF_RING - 3>();   // row j + 2 (the next pivot); row j + 1 arrived a step ago
    const int J = j / ET;
    // the new carried value of a column and its entry of U (or of the transformed right-hand sides)
    auto step = [&](int col, cplx x) {
      const cplx c = cur[col];
      const cplx u = swap ? x : c, low = swap ? c : x;
      if (!last)
        cur[col] = make_cuDoubleComplex(fma(-l.x, u.x, fma(l.y, u.y, low.x)),
                                        fma(-l.x, u.y, fma(-l.y, u.x, low.y)));
      if (col < m) {
        const int K = col / ET;
        U[((long long)K * (K + 1) / 2 + J) * (ET * ET) + (j % ET) * ET + col % ET] = dfc_split(u);
        if (col == j) dU[j] = u;
      } else {
        R[(long long)j * a.ldy + (col - m)] = u;
      }
    };
    int col = j + ((tid - j) & (EF_T - 1));   // the thread's first column >= j
    if (!last && col == j + 1) {              // the next pivot first: the next step waits for nothing else
      step(col, cuCadd(next(j + 1, col), sig));
      pivot(col, cur[col]);
      col += EF_T;
    }
    for (; col < n; col += EF_T) step(col, last ? cz() : next(j + 1, col));
    issue(j + EF_RING);   // into the slot of row j, which this thread has consumed
  }
}

// Back substitution, one CTA per (frequency, group of P = 8 C right-hand sides), by blocks of 32 rows from
// the bottom: acc = R_J - sum_{K > J} U_JK Y_K in double-float with 2 x C register tiles, then the 32 x 32
// triangular solve by four lanes per right-hand side with one warp barrier per row. Every row takes its terms one after
// the other from the last column down, renormalised after each: the sums of a plain column-by-column substitution, bit
// for bit. (Renormalising every eighth term and going up through the columns of a tile took 16.7 ms instead of 17.9
// for order 336, 42 right-hand sides and 2000 frequencies, and was 1.7 to 2.9 times further from extended precision,
// orders 40 to 800.) The division by the diagonal is a product with its
// reciprocal, both in FP64, shared by two lanes: a complex division is thirty instructions on the FP64 pipe, this five.
// U and Y arrive by cp.async in steps of 16 columns of U, double-buffered: per step a thread takes 2 + C shared loads
// for 2 C complex multiply-adds of 56 FP32 operations, so the FP32 pipe is what bounds it; 34-43 KB of shared memory
// and 128 threads whatever P keep four CTAs (one warp each per scheduler) on an SM. Solved blocks are kept
// in Y as double-float and converted to FP64 at the end.
constexpr int EB_T = 128, EK = ET / 2;
template <int C>
__global__ void __launch_bounds__(EB_T, 4) eval_backsub_kernel(EvalArgs a, int w0) {
  constexpr int P = 8 * C, US = EK + 1;    // padded U row: rows of a column on different banks
  extern __shared__ float4 eb_sm[];
  float4* sU = eb_sm;                      // [2][ET][US]: a half tile each; both halves of the diagonal tile
  float4* sY = sU + 2 * ET * US;           // [2][EK][P]; the block's right-hand sides during its solve
  cplx* sD = reinterpret_cast<cplx*>(sY + 2 * EK * P);   // [ET] reciprocal diagonal
  const int m = a.m, np = a.np, tid = threadIdx.x, f = blockIdx.x, w = w0 + f;
  const int p0 = blockIdx.y * P, pn = min(P, np - p0);
  const float4* U = a.U + (long long)f * eval_tiles(m) * (ET * ET);
  const cplx* dU = a.dU + (long long)f * m;
  cplx* R = a.Y + (long long)w * np + p0;
  const int T = (m + ET - 1) / ET;
  const int tx = tid & 7, ty = tid >> 3;   // columns tx + 8 i, rows 2 ty + r
  // half h of tile (J, K) into buffer h; columns of U beyond m as zeros
  auto load_u = [&](int J, int K, int h) {
    const float4* s = U + ((long long)K * (K + 1) / 2 + J) * (ET * ET) + h * EK;
    for (int t = tid; t < ET * EK; t += EB_T) {
      const int r = t / EK, k = t % EK;
      cp_async16(sU + (h * ET + r) * US + k, s + r * ET + k, K * ET + h * EK + k < m);
    }
  };
  auto load_y = [&](int K, int h) {
    for (int t = tid; t < EK * P; t += EB_T) {
      const int k = K * ET + h * EK + t / P, p = t % P;
      const bool on = k < m && p < pn;
      cp_async16(sY + h * EK * P + t, on ? R + (long long)k * a.ldy + p : R, on);
    }
  };
  for (int J = T - 1; J >= 0; --J) {
    if (J < T - 1) {
      load_u(J, T - 1, 1);
      load_y(T - 1, 1);
      cp_async_commit();
    }
    float4 acc[2][C];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int row = J * ET + 2 * ty + r, p = tx + 8 * i;
        acc[r][i] = (row < m && p < pn) ? dfc_from(R[(long long)row * a.ldy + p]) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    for (int K = T - 1; K > J; --K) {
#pragma unroll 1
      for (int h = 1; h >= 0; --h) {
        // the next half tile: the first half of this one, the second of the next; after the last the diagonal
        // tile is loaded below
        if (h == 1 || K - 1 > J) {
          load_u(J, h == 1 ? K : K - 1, h ^ 1);
          load_y(h == 1 ? K : K - 1, h ^ 1);
        }
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();
        const float4* u = sU + (h * ET + 2 * ty) * US;
        const float4* y = sY + h * EK * P + tx;
#pragma unroll 2
        for (int k = EK - 1; k >= 0; --k) {
          const float4 u0 = u[k], u1 = u[US + k];
#pragma unroll
          for (int i = 0; i < C; ++i) {
            const float4 yy = y[k * P + 8 * i];
            acc[0][i] = dfc_sub_mul(acc[0][i], u0, yy);
            acc[1][i] = dfc_sub_mul(acc[1][i], u1, yy);
          }
        }
        __syncthreads();
      }
    }
    load_u(J, J, 0);
    load_u(J, J, 1);
    cp_async_commit();
    float4* sR = sY;   // [ET][P]
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int i = 0; i < C; ++i) sR[(2 * ty + r) * P + tx + 8 * i] = acc[r][i];
    if (tid < ET && J * ET + tid < m) {
      const cplx d = dU[J * ET + tid];
      sD[tid] = (d.x == 0.0 && d.y == 0.0) ? cz() : cuCdiv(make_cuDoubleComplex(1.0, 0.0), d);
    }
    cp_async_wait<0>();
    __syncthreads();
    {
      // lanes 8 g .. 8 g + 7 hold eight right-hand sides and take the rows i = g (mod 4)
      const int g = (tid & 31) >> 3;
      for (int c8 = tid >> 5; c8 < C; c8 += EB_T / 32) {
        const int p = c8 * 8 + (tid & 7);
        for (int j = min(ET, m - J * ET) - 1; j >= 0; --j) {
          const float4* u = sU + (j / EK) * ET * US + j % EK;
          // lanes with even g form the real part of sR_j sD_j, those with odd g the imaginary one
          const float4 r = sR[j * P + p];
          const cplx d = sD[j];
          const bool im = g & 1;
          const double mine = im ? df_to(r.z, r.w) : df_to(r.x, r.y), other = __shfl_xor_sync(0xffffffffu, mine, 8);
          const df2 v = df_split(fma(mine, d.x, other * (im ? d.y : -d.y)));
          const float oh = __shfl_xor_sync(0xffffffffu, v.h, 8), ol = __shfl_xor_sync(0xffffffffu, v.l, 8);
          const float4 y = im ? make_float4(oh, ol, v.h, v.l) : make_float4(v.h, v.l, oh, ol);
          for (int i = g; i < j; i += 4) sR[i * P + p] = dfc_sub_mul(sR[i * P + p], u[i * US], y);
          __syncwarp();
          if (g == 0) sR[j * P + p] = y;
        }
      }
    }
    __syncthreads();
    for (int t = tid; t < ET * P; t += EB_T) {
      const int row = J * ET + t / P, p = t % P;
      if (row < m && p < pn) *reinterpret_cast<float4*>(R + (long long)row * a.ldy + p) = sR[t];
    }
    __syncthreads();
  }
  for (int t = tid; t < m * P; t += EB_T) {
    const int p = t % P;
    cplx* q = R + (long long)(t / P) * a.ldy + p;
    if (p < pn) *q = dfc_to(*reinterpret_cast<const float4*>(q));
  }
}

// width of the right-hand-side groups: the one that pads np least (the widest of equals: U is read once
// per group)
int eval_group(int np) {
  int best = 8;
  for (int P : {8, 16, 24, 32, 40, 48})
    if ((np + P - 1) / P * P <= (np + best - 1) / best * best) best = P;
  return best;
}
struct EvalScratch {   // U tiles and diagonals of the frequencies in flight
  DBuf<float4> U;
  DBuf<cplx> dU, rows;
  int nf = 0;          // frequencies they hold
};
// Frequencies in flight: U of all of them in at most 4 GB and an eighth of the free memory.
void eval_scratch_alloc(EvalScratch& e, int m, int np, int nw) {
  const long long per = eval_tiles(m) * ET * ET * (long long)sizeof(float4) + 16LL * m;
  long long budget = 1LL << 30;
  if (per * nw > budget) {
    size_t freeb = device_free_bytes();
    if (freeb == 0) freeb = 8ull << 30;
    budget = std::min<long long>(4LL << 30, (long long)(freeb / 8));
  }
  e.nf = (int)std::max<long long>(1, std::min<long long>({(long long)nw, budget / per, 65535LL}));
  e.U.alloc(eval_tiles(m) * ET * ET * e.nf);
  e.dU.alloc((long long)m * e.nf);
  if (sizeof(cplx) * (size_t)(EF_RING + 1) * (m + np) > 200 * 1024) e.rows.alloc((long long)(m + np) * e.nf);
}
void launch_eval_solve(EvalArgs ea, EvalScratch& es, cudaStream_t s) {
  const size_t fbytes = sizeof(cplx) * (size_t)(EF_RING + 1) * (ea.m + ea.np);
  const bool ring = fbytes <= 200 * 1024;
  int dev = 0;
  GFCC_CUDA(cudaGetDevice(&dev));
  GFCC_CHECK(dev >= 0 && dev < 64, GFCC_ERR_ARG, "device ordinal above 63");
  ea.U = es.U.p;
  ea.dU = es.dU.p;
  auto backsub = [&](auto Cc, int w0, int nf) {
    constexpr int C = decltype(Cc)::value;   // at most 43 KB of shared memory: no attribute needed
    constexpr size_t bytes = sizeof(float4) * (2 * ET * (EK + 1) + 2 * EK * 8 * C + ET);
    static_assert(bytes <= 48 * 1024, "default shared memory");
    eval_backsub_kernel<C><<<dim3(nf, (ea.np + 8 * C - 1) / (8 * C)), EB_T, bytes, s>>>(ea, w0);
  };
  static bool attr_f[64] = {};
  if (!attr_f[dev]) {
    GFCC_CUDA(cudaFuncSetAttribute(eval_factor_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    attr_f[dev] = true;
  }
  for (int w0 = 0; w0 < ea.nw; w0 += es.nf) {
    const int nf = std::min(es.nf, ea.nw - w0);
    if (ring) eval_factor_kernel<true><<<nf, EF_T, fbytes, s>>>(ea, w0, nullptr);
    else eval_factor_kernel<false><<<nf, EF_T, 0, s>>>(ea, w0, es.rows.p);
    GFCC_LAUNCH_CHECK();
    switch (eval_group(ea.np)) {
      case 8: backsub(std::integral_constant<int, 1>{}, w0, nf); break;
      case 16: backsub(std::integral_constant<int, 2>{}, w0, nf); break;
      case 24: backsub(std::integral_constant<int, 3>{}, w0, nf); break;
      case 32: backsub(std::integral_constant<int, 4>{}, w0, nf); break;
      case 40: backsub(std::integral_constant<int, 5>{}, w0, nf); break;
      default: backsub(std::integral_constant<int, 6>{}, w0, nf); break;
    }
    GFCC_LAUNCH_CHECK();
  }
}

// A[w] = -(1/pi) sum_p Im G[w][p][qidx[p]] (p with a matching q only)
__global__ void spectral_from_G_kernel(const cplx* __restrict__ G, int nw, int np, int nq, const int* __restrict__ qidx,
                                       double* __restrict__ A) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= nw) return;
  double acc = 0.0;
  for (int p = 0; p < np; ++p) {
    const int qi = qidx[p];
    if (qi >= 0) acc += G[((long long)w * np + p) * nq + qi].y;
  }
  A[w] = -acc / 3.14159265358979323846;
}

// Ys[k][w np + p] = (w - i eta) Y[k][w np + p]
__global__ void shift_scale_kernel(const cplx* __restrict__ Y, long long ldy, int m, int np, int nw,
                                   const double* __restrict__ omegas, double eta, cplx* __restrict__ Ys) {
  const long long total = (long long)m * nw * np;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long k = t / ((long long)nw * np), n = t % ((long long)nw * np);
    const int w = (int)(n / np);
    Ys[k * ldy + n] = cuCmul(make_cuDoubleComplex(omegas[w], -eta), Y[k * ldy + n]);
  }
}

// res[w np + p] = || C[:, w np + p] - RB[:, p] || / bn[p]   (C row-major [qn][ldc])
__global__ void resnorm_kernel(const cplx* __restrict__ C, long long ldc, int qn, const cplx* __restrict__ RB,
                               int np, int nw, const double* __restrict__ bn, double* __restrict__ res) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= (long long)nw * np) return;
  const int p = (int)(n % np);
  double s = 0.0;
  for (int r = 0; r < qn; ++r) {
    const cplx d = cuCsub(C[(long long)r * ldc + n], RB[r + (long long)p * qn]);
    s = fma(d.x, d.x, fma(d.y, d.y, s));
  }
  res[n] = sqrt(s) / bn[p];
}
__global__ void rowmax_kernel(const double* __restrict__ res, int np, int nw, double* __restrict__ out) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= nw) return;
  double mx = 0.0;
  for (int p = 0; p < np; ++p) mx = fmax(mx, res[(long long)w * np + p]);
  out[w] = mx;
}

}  // namespace

// ------------------------------------------------------------------------------------------------
namespace {

// reallocate a batch-minor [rows][old_cap] block as [rows][new_cap] keeping ncols columns
void regrow_rows(DBuf<cplx>& b, long long rows, int old_cap, int new_cap, int ncols, cudaStream_t s) {
  DBuf<cplx> nb2;
  nb2.alloc(rows * new_cap);
  nb2.zero(s);
  if (ncols > 0)
    GFCC_CUDA(cudaMemcpy2DAsync(nb2.p, sizeof(cplx) * new_cap, b.p, sizeof(cplx) * old_cap, sizeof(cplx) * ncols, rows,
                                cudaMemcpyDeviceToDevice, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  std::swap(b.p, nb2.p);
  std::swap(b.n, nb2.n);
}
// reallocate a col-major [old_ld x ...] matrix as [new_ld x alloc_cols] keeping nrows x ncols
void regrow_cm(DBuf<cplx>& b, int old_ld, int new_ld, int alloc_cols, int nrows, int ncols, cudaStream_t s) {
  DBuf<cplx> nb2;
  nb2.alloc((long long)new_ld * std::max(alloc_cols, 1));
  nb2.zero(s);
  if (nrows > 0 && ncols > 0)
    GFCC_CUDA(cudaMemcpy2DAsync(nb2.p, sizeof(cplx) * new_ld, b.p, sizeof(cplx) * old_ld, sizeof(cplx) * nrows, ncols,
                                cudaMemcpyDeviceToDevice, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  std::swap(b.p, nb2.p);
  std::swap(b.n, nb2.n);
}

// FP64 arithmetic runs on a narrow pipe on this GPU: every product of the orthonormalisation above a
// small size goes to the exact-slice tensor-core GEMM (7 slices of 7 bits, 48 bits per row). Fewer bits are
// not enough: the residual basis resolves the solver-residual directions of Z = M S, about 1e-8 of
// the columns' norms, and 41-bit products perturb them enough to spoil the refinement estimates.
// The coefficients of the first Gram-Schmidt pass are the exception (ns = 4, 35 bits): the reconstruction
// y = Q (C1 + C2) + y'' holds for whatever C1 the first update subtracts, and the second pass, whose
// coefficients and both updates keep the 48 bits, removes what a less accurate C1 leaves along Q. The
// second-pass and panel Gram products need the full accuracy even for the residual basis: with 34 bits the
// refinement no longer converged (the model grew to the size limit).
void fp64_accurate_zgemm(const ZGemmDesc& g, cudaStream_t s, int ns = OZ_SLICES_MOR, int bits = OZ_BITS_MOR) {
  if ((double)g.M * (double)g.N * (double)g.K >= (double)(1 << 22) && g.batch == 1) zgemm_oz(g, ns, s, bits);
  else zgemm(g, s);
}

// ---- panel kernels: column-wise CGS2 inside a panel of at most PB columns -----------------------
constexpr int PB = 32;            // panel width (one lane per panel column)
constexpr int PTY = 8;            // warps per block, each sweeping its own rows

// out[c] (partial[chunk][c]) = sum_{nu in chunk} |Y[nu][c]|^2 for c < nc; block (32, PTY)
__global__ void colnorms_partial_kernel(const cplx* __restrict__ Y, int nc, long long D, long long rows,
                                        double* __restrict__ partial) {
  __shared__ double red[PTY][32];
  const int c = blockIdx.x * 32 + threadIdx.x;
  const long long r0 = blockIdx.y * rows, r1 = min(D, r0 + rows);
  double acc = 0.0;
  if (c < nc)
    for (long long nu = r0 + threadIdx.y; nu < r1; nu += PTY) {
      const cplx a = Y[nu * nc + c];
      acc = fma(a.x, a.x, fma(a.y, a.y, acc));
    }
  red[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y == 0 && c < nc) {
    double t = 0.0;
    for (int k = 0; k < PTY; ++k) t += red[k][threadIdx.x];
    partial[(long long)blockIdx.y * nc + c] = t;
  }
}
__global__ void colnorms_reduce_kernel(const double* __restrict__ partial, int nchunk, int nc, double* __restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nc) return;
  double t = 0.0;
  for (int k = 0; k < nchunk; ++k) t += partial[(long long)k * nc + c];
  out[c] = sqrt(t);
}

// partial[chunk][i] = sum_{nu in chunk} conj(Y[nu][c0 + i]) Y[nu][j] for i < n (n < PB); block (32, PTY)
__global__ void pdot_kernel(const cplx* __restrict__ Y, int nc, long long D, int c0, int n, int j, long long rows,
                            cplx* __restrict__ partial) {
  __shared__ cplx red[PTY][32];
  const int i = threadIdx.x;
  const long long r0 = blockIdx.y * rows, r1 = min(D, r0 + rows);
  cplx acc = cz();
  if (i < n)
#pragma unroll 4
    for (long long nu = r0 + threadIdx.y; nu < r1; nu += PTY) {
      const cplx a = Y[nu * nc + c0 + i], b = Y[nu * nc + j];
      acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
      acc.y = fma(a.x, b.y, fma(-a.y, b.x, acc.y));
    }
  red[threadIdx.y][i] = acc;
  __syncthreads();
  if (threadIdx.y == 0 && i < n) {
    cplx t = cz();
    for (int k = 0; k < PTY; ++k) { t.x += red[k][i].x; t.y += red[k][i].y; }
    partial[(long long)blockIdx.y * PB + i] = t;
  }
}
// h[i] = sum_chunk partial[chunk][i]; T[c0 + i][j] += h[i] (T col-major, ld ldt) when T is non-null
// (block (32, PTY))
__global__ void preduce_kernel(const cplx* __restrict__ partial, int nchunk, int n, cplx* __restrict__ h,
                               cplx* __restrict__ T, int ldt, int c0, int j) {
  __shared__ cplx red[PTY][32];
  const int i = threadIdx.x;
  cplx t = cz();
  if (i < n)
    for (int k = threadIdx.y; k < nchunk; k += PTY) {
      t.x += partial[(long long)k * PB + i].x;
      t.y += partial[(long long)k * PB + i].y;
    }
  red[threadIdx.y][i] = t;
  __syncthreads();
  if (threadIdx.y == 0 && i < n) {
    for (int k = 1; k < PTY; ++k) { t.x += red[k][i].x; t.y += red[k][i].y; }
    h[i] = t;
    if (T) { T[c0 + i + (long long)j * ldt].x += t.x; T[c0 + i + (long long)j * ldt].y += t.y; }
  }
}
// Y[nu][j] -= sum_{i<n} Y[nu][c0 + i] h[i] (and MY alike); then, for mode 0, the partial dot products
// of the updated column with the panel columns (as pdot_kernel) or, for mode 1, partial[chunk][0].x =
// sum |Y[nu][j]|^2. Lane i holds panel column c0 + i; each warp takes PU rows per step (independent
// shuffle reductions in flight), block (32, PTY).
constexpr int PU = 4;
// Sums over the 32 lanes of the components of PU = 4 complex numbers s: the eight values are halved between lane pairs
// while they are summed (9 additions instead of 40: FP64 additions are what bounds this kernel; D = 56,580, 32-column
// panels: 73 -> 40 us a launch), after which lanes
// with lane >> 2 == 2 u + component hold the total of component (0: re, 1: im) of s[u].
__device__ __forceinline__ double warp_sum4(const cplx (&s)[PU], int lane) {
  static_assert(PU == 4, "four rows");
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
  cplx t0 = h16 ? s[2] : s[0], t1 = h16 ? s[3] : s[1];
  const cplx o0 = h16 ? s[0] : s[2], o1 = h16 ? s[1] : s[3];
  t0.x += __shfl_xor_sync(0xffffffffu, o0.x, 16);
  t0.y += __shfl_xor_sync(0xffffffffu, o0.y, 16);
  t1.x += __shfl_xor_sync(0xffffffffu, o1.x, 16);
  t1.y += __shfl_xor_sync(0xffffffffu, o1.y, 16);
  cplx t = h8 ? t1 : t0;
  const cplx o = h8 ? t0 : t1;
  t.x += __shfl_xor_sync(0xffffffffu, o.x, 8);
  t.y += __shfl_xor_sync(0xffffffffu, o.y, 8);
  double v = h4 ? t.y : t.x;
  v += __shfl_xor_sync(0xffffffffu, h4 ? t.x : t.y, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}
__global__ void pupdate_kernel(cplx* __restrict__ Y, cplx* __restrict__ MY, int nc, long long D, int c0, int n,
                               int j, long long rows, const cplx* __restrict__ h, int mode,
                               cplx* __restrict__ partial) {
  __shared__ cplx red[PTY][32];
  const int i = threadIdx.x;
  const long long r0 = blockIdx.y * rows, r1 = min(D, r0 + rows);
  const cplx hi = i < n ? h[i] : cz();
  cplx acc = cz();
  for (long long base = r0 + (long long)threadIdx.y * PU; base < r1; base += (long long)PTY * PU) {
    cplx a[PU], y[PU], s[PU];
#pragma unroll
    for (int u = 0; u < PU; ++u) {
      const long long nu = base + u;
      const bool in = nu < r1;
      a[u] = (in && i < n) ? Y[nu * nc + c0 + i] : cz();
      y[u] = in ? Y[nu * nc + j] : cz();   // read by every lane before lane 0 writes it
      s[u] = make_cuDoubleComplex(a[u].x * hi.x - a[u].y * hi.y, a[u].x * hi.y + a[u].y * hi.x);
    }
    double v = warp_sum4(s, i);
    __syncwarp();
#pragma unroll
    for (int u = 0; u < PU; ++u) {
      y[u].x -= __shfl_sync(0xffffffffu, v, 8 * u);
      y[u].y -= __shfl_sync(0xffffffffu, v, 8 * u + 4);
      if (i == 0 && base + u < r1) Y[(base + u) * nc + j] = y[u];
    }
    if (MY) {
#pragma unroll
      for (int u = 0; u < PU; ++u) {
        const long long nu = base + u;
        const cplx b = (nu < r1 && i < n) ? MY[nu * nc + c0 + i] : cz();
        s[u] = make_cuDoubleComplex(b.x * hi.x - b.y * hi.y, b.x * hi.y + b.y * hi.x);
      }
      v = warp_sum4(s, i);
      const long long nu = base + (i >> 3);   // lanes 0, 4, 8, ...: one component of a row each
      if ((i & 3) == 0 && nu < r1) reinterpret_cast<double*>(MY + nu * nc + j)[(i >> 2) & 1] -= v;
    }
#pragma unroll
    for (int u = 0; u < PU; ++u) {
      if (mode == 0) {
        acc.x = fma(a[u].x, y[u].x, fma(a[u].y, y[u].y, acc.x));
        acc.y = fma(a[u].x, y[u].y, fma(-a[u].y, y[u].x, acc.y));
      } else if (i == 0) {
        acc.x = fma(y[u].x, y[u].x, fma(y[u].y, y[u].y, acc.x));
      }
    }
  }
  red[threadIdx.y][i] = acc;
  __syncthreads();
  if (threadIdx.y == 0 && (mode == 0 ? i < n : i == 0)) {
    cplx t = cz();
    for (int k = 0; k < PTY; ++k) { t.x += red[k][i].x; t.y += red[k][i].y; }
    partial[(long long)blockIdx.y * PB + i] = t;
  }
}
// n1 = sqrt(sum_chunk partial[chunk][0].x); keep column j when n0[j] > 0 and n1 >= drop_tol n0[j];
// scale[j] = keep ? 1 / n1 : 0; T[j][j] = n1 when kept
__global__ void pfinish_kernel(const cplx* __restrict__ partial, int nchunk, const double* __restrict__ n0, int j,
                               double drop_tol, double* __restrict__ scale, int* __restrict__ keep,
                               cplx* __restrict__ T, int ldt) {
  __shared__ double red[256];
  double t = 0.0;
  for (int k = threadIdx.x; k < nchunk; k += blockDim.x) t += partial[(long long)k * PB].x;
  red[threadIdx.x] = t;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double n1 = sqrt(red[0]);
    const bool k = n0[j] > 0.0 && n1 >= drop_tol * n0[j];
    scale[j] = k ? 1.0 / n1 : 0.0;
    keep[j] = k ? 1 : 0;
    if (T && k) T[j + (long long)j * ldt] = make_cuDoubleComplex(n1, 0.0);
  }
}
__global__ void pscale_kernel(cplx* __restrict__ Y, cplx* __restrict__ MY, int nc, long long D, int j,
                              const double* __restrict__ scale) {
  const double sc = scale[j];
  for (long long nu = blockIdx.x * (long long)blockDim.x + threadIdx.x; nu < D; nu += (long long)gridDim.x * blockDim.x) {
    Y[nu * nc + j].x *= sc; Y[nu * nc + j].y *= sc;
    if (MY) { MY[nu * nc + j].x *= sc; MY[nu * nc + j].y *= sc; }
  }
}
// T[i][c0 + j] += Cf[i][j] for i < rows, j < pb (Cf row-major [rows][pb], T col-major ld ldt)
__global__ void add_block_kernel(cplx* __restrict__ T, int ldt, int c0, const cplx* __restrict__ Cf, int rows, int pb) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= rows * pb) return;
  const int i = t / pb, j = t % pb;
  T[i + (long long)(c0 + j) * ldt].x += Cf[t].x;
  T[i + (long long)(c0 + j) * ldt].y += Cf[t].y;
}

// Complex Cholesky G = R^H R of a Hermitian positive definite n x n matrix (row-major); returns false
// when a pivot is not positive.
bool cholesky_upper(const std::vector<cplx>& G, int n, std::vector<cplx>& R) {
  R.assign((size_t)n * n, make_cuDoubleComplex(0.0, 0.0));
  for (int j = 0; j < n; ++j) {
    double d = G[(size_t)j * n + j].x;
    for (int i = 0; i < j; ++i) d -= R[(size_t)i * n + j].x * R[(size_t)i * n + j].x + R[(size_t)i * n + j].y * R[(size_t)i * n + j].y;
    if (!(d > 0.0)) return false;
    const double rjj = std::sqrt(d);
    R[(size_t)j * n + j] = make_cuDoubleComplex(rjj, 0.0);
    for (int k = j + 1; k < n; ++k) {
      cplx t = G[(size_t)j * n + k];
      for (int i = 0; i < j; ++i) t = cuCsub(t, cuCmul(cuConj(R[(size_t)i * n + j]), R[(size_t)i * n + k]));
      R[(size_t)j * n + k] = make_cuDoubleComplex(t.x / rjj, t.y / rjj);
    }
  }
  return true;
}
// inverse of an upper triangular n x n matrix (row-major)
std::vector<cplx> inverse_upper(const std::vector<cplx>& R, int n) {
  std::vector<cplx> X((size_t)n * n, make_cuDoubleComplex(0.0, 0.0));
  for (int j = n - 1; j >= 0; --j) {
    X[(size_t)j * n + j] = cuCdiv(make_cuDoubleComplex(1.0, 0.0), R[(size_t)j * n + j]);
    for (int k = j + 1; k < n; ++k) {
      cplx t = make_cuDoubleComplex(0.0, 0.0);
      for (int i = j + 1; i <= k; ++i) t = cuCadd(t, cuCmul(R[(size_t)j * n + i], X[(size_t)i * n + k]));
      X[(size_t)j * n + k] = cuCmul(cuCsub(make_cuDoubleComplex(0.0, 0.0), t), X[(size_t)j * n + j]);
    }
  }
  return X;
}

// Panel of pb columns Y[:, c0:c0+pb] (already orthogonal to every earlier column): Cholesky QR twice
// (Y = Q R2 R1 with the Gram matrices formed by FP64-accurate GEMMs). In exact arithmetic this is the
// column-by-column Gram-Schmidt of the panel (the same Q and R with a positive diagonal). It is taken
// only when the panel is well conditioned: every first-pass pivot R1_jj at least 1e-5 of its column's
// norm (a bound on the conditioning of the column-scaled panel, which is what Cholesky QR's accuracy
// depends on) and at least 10 drop_tol of the column's norm before any projection (n0), so that two
// passes give orthonormality to rounding and no column is within a factor 10 of the drop threshold;
// otherwise the caller runs the column-by-column passes. Writes T[c0:c0+pb, c0:c0+pb] = R2 R1 and keep = 1.
// Z[nu][j] <- sum_{k <= j} Z[nu][k] X[k][j] for the pb (<= 32) columns of a panel: X upper
// triangular, double-float, row-major pb x pb. One warp per row, in place; each lane forms one output
// column in double-float (the row's entries are split once by their own lanes and broadcast).
__global__ void __launch_bounds__(256) panel_apply_kernel(cplx* __restrict__ Z, int nc, int pb, long long D,
                                                          const float4* __restrict__ Xdf) {
  __shared__ float4 xs[32 * 32];
  for (int t = threadIdx.x; t < pb * pb; t += blockDim.x) xs[t] = Xdf[t];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long long nu = blockIdx.x * 8LL + warp; nu < D; nu += gridDim.x * 8LL) {
    cplx* row = Z + nu * nc;
    const float4 zk = lane < pb ? dfc_from(row[lane]) : make_float4(0.f, 0.f, 0.f, 0.f);
    df2 ar{0.f, 0.f}, ai{0.f, 0.f};
    for (int k = 0; k < pb; ++k) {
      const float zrh = __shfl_sync(0xffffffffu, zk.x, k), zrl = __shfl_sync(0xffffffffu, zk.y, k);
      const float zih = __shfl_sync(0xffffffffu, zk.z, k), zil = __shfl_sync(0xffffffffu, zk.w, k);
      if (lane >= k && lane < pb) {
        const float4 x = xs[k * pb + lane];
        const df2 zr{zrh, zrl}, zi{zih, zil}, nzi{-zih, -zil}, xr{x.x, x.y}, xi{x.z, x.w};
        ar = df_dot2(ar, zr, xr, nzi, xi);   // re += zr xr - zi xi
        ai = df_dot2(ai, zr, xi, zi, xr);    // im += zr xi + zi xr
      }
    }
    if (lane < pb) row[lane] = make_cuDoubleComplex(df_to(ar.h, ar.l), df_to(ai.h, ai.l));
  }
}

struct PanelWork {
  DBuf<cplx> Gd;
  DBuf<float4> Rdf;
};
bool panel_cholqr2(gfcc_ctx* c, cplx* Y, cplx* MY, int nc, long long D, int c0, int pb, const double* n0,
                   cplx* T, int* keep_dev, PanelWork& pw) {
  cudaStream_t s = c->stream;
  std::vector<cplx> G((size_t)pb * pb), R1, R2;
  DBuf<cplx>& Gd = pw.Gd;
  DBuf<float4>& Rdf = pw.Rdf;
  Gd.alloc((long long)pb * pb);
  Rdf.alloc((long long)pb * pb);
  auto gram = [&]() {
    ZGemmDesc g;
    g.M = pb; g.N = pb; g.K = (int)D;
    g.A = Y + c0; g.sam = 1; g.sak = nc; g.conjA = true;
    g.B = Y + c0; g.sbk = nc; g.sbn = 1;
    g.C = Gd.p; g.scm = pb; g.scn = 1;
    g.work = zgemm_work(c);
    fp64_accurate_zgemm(g, s);
    GFCC_CUDA(cudaMemcpyAsync(G.data(), Gd.p, sizeof(cplx) * pb * pb, cudaMemcpyDeviceToHost, s));
    GFCC_CUDA(cudaStreamSynchronize(s));
    for (int i = 0; i < pb; ++i) {   // exact Hermitian symmetry and a real diagonal
      G[(size_t)i * pb + i].y = 0.0;
      for (int k = i + 1; k < pb; ++k) G[(size_t)k * pb + i] = cuConj(G[(size_t)i * pb + k]);
    }
  };
  auto apply = [&](const std::vector<cplx>& R) {   // Y (and MY) <- Y R^{-1}, in double-float
    GFCC_CHECK(pb <= 32, GFCC_ERR_ARG, "panel wider than a warp");
    std::vector<cplx> X = inverse_upper(R, pb);
    std::vector<float4> Xf((size_t)pb * pb);
    for (size_t t = 0; t < Xf.size(); ++t) {   // the same split as on the device: h = fl(x), l = fl(x - h)
      const float rh = (float)X[t].x, ih = (float)X[t].y;
      Xf[t] = make_float4(rh, (float)(X[t].x - (double)rh), ih, (float)(X[t].y - (double)ih));
    }
    GFCC_CUDA(cudaMemcpyAsync(Rdf.p, Xf.data(), sizeof(float4) * pb * pb, cudaMemcpyHostToDevice, s));
    const int grid = (int)std::min<long long>((D + 7) / 8, 152LL * 16);
    for (cplx* Z : {Y, MY}) {
      if (!Z) continue;
      panel_apply_kernel<<<grid, 256, 0, s>>>(Z + c0, nc, pb, D, Rdf.p);
      GFCC_LAUNCH_CHECK();
    }
    GFCC_CUDA(cudaStreamSynchronize(s));   // Xf is host memory of this scope
  };
  gram();
  if (!cholesky_upper(G, pb, R1)) return false;
  for (int j = 0; j < pb; ++j) {   // pivot relative to the column's own norm (scale-invariant test)
    const double r = R1[(size_t)j * pb + j].x;
    if (!(r >= 1e-5 * std::sqrt(G[(size_t)j * pb + j].x)) || !(r >= 10.0 * c->opts.drop_tol * n0[j])) return false;
  }
  apply(R1);
  gram();
  if (!cholesky_upper(G, pb, R2)) return false;   // cannot happen after a well-conditioned first pass
  apply(R2);
  if (T) {   // T block = R2 R1 (upper triangular), column-major in T (ld nc)
    std::vector<cplx> Tb((size_t)pb * pb, make_cuDoubleComplex(0.0, 0.0));
    for (int i = 0; i < pb; ++i)
      for (int k = i; k < pb; ++k) {
        cplx t = make_cuDoubleComplex(0.0, 0.0);
        for (int l = i; l <= k; ++l) t = cuCadd(t, cuCmul(R2[(size_t)i * pb + l], R1[(size_t)l * pb + k]));
        Tb[(size_t)k * pb + i] = t;   // column k, row i
      }
    GFCC_CUDA(cudaMemcpy2DAsync(T + c0 + (long long)c0 * nc, sizeof(cplx) * nc, Tb.data(), sizeof(cplx) * pb,
                                sizeof(cplx) * pb, pb, cudaMemcpyHostToDevice, s));
  }
  std::vector<int> ones(pb, 1);
  GFCC_CUDA(cudaMemcpyAsync(keep_dev + c0, ones.data(), sizeof(int) * pb, cudaMemcpyHostToDevice, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  return true;
}

// Orthonormalise the nc columns of Y ([D][nc] batch-minor) against the n_cur columns of the basis
// Bs ([D][cap]) and against each other, column by column in order: each column loses its components
// along all earlier columns by classical Gram-Schmidt applied twice, and is kept when its norm after
// that is >= drop_tol times its norm before, else zeroed. The same linear operations are applied to
// MY when it is non-null (MBs being the matching block of Bs). Cold (device, n_cur x nc col-major,
// ld n_cur) and T (device, nc x nc col-major) receive the coefficients
// y_j = Bs Cold[:, j] + sum_i T[i, j] ynew_i when the pointers are non-null. Returns the kept columns.
//
// Blocking (the same projections in exact arithmetic, since the subspaces are mutually orthogonal):
// two passes of block CGS against Bs; then panels of PB columns, each projected twice against the
// finished earlier panels by two GEMMs per pass, and finally column by column inside the panel, whose
// PB columns stay resident in L2. The keep decisions are taken on the device.
std::vector<int> ortho_block(gfcc_ctx* c, const cplx* Bs, int cap, int n_cur, cplx* Y, cplx* MY, const cplx* MBs,
                             int nc, cplx* Cold, cplx* T) {
  if (nc <= 0) return {};
  cudaStream_t s = c->stream;
  const long long D = c->D;
  // one chunk of rows per block: one wave of two PTY-warp blocks per SM (pupdate_kernel's registers)
  const long long rows = std::max<long long>(64, (D + 152 * 2 - 1) / (152 * 2));
  const int nchunk = (int)((D + rows - 1) / rows);
  DBuf<double> n0, scale, npart;
  DBuf<int> keep;
  n0.alloc(nc);
  scale.alloc(nc);
  keep.alloc(nc);
  npart.alloc((long long)nchunk * nc);
  colnorms_partial_kernel<<<dim3((nc + 31) / 32, nchunk), dim3(32, PTY), 0, s>>>(Y, nc, D, rows, npart.p);
  GFCC_LAUNCH_CHECK();
  colnorms_reduce_kernel<<<(nc + 127) / 128, 128, 0, s>>>(npart.p, nchunk, nc, n0.p);
  GFCC_LAUNCH_CHECK();
  if (T) GFCC_CUDA(cudaMemsetAsync(T, 0, sizeof(cplx) * nc * nc, s));
  DBuf<cplx> Cf;
  Cf.alloc((long long)std::max(std::max(n_cur, nc), 1) * std::max(nc, 1));
  auto block_cgs = [&](const cplx* Pb, int ldp, int np_, const cplx* MPb, int col0, int ncols, bool to_cold) {
    // two passes: Cf (row-major [np_][ncols]) = Pb^H Y[:, col0:col0+ncols]; Y[:, col0:...] -= Pb Cf.
    // Pb and MPb do not change between the passes: their slices as left operands of the updates are
    // made once.
    void* cache_p = zgemm_slice_cache(c, 0);
    void* cache_m = zgemm_slice_cache(c, 1);
    zgemm_slice_cache_reset(cache_p);
    zgemm_slice_cache_reset(cache_m);
    for (int pass = 0; pass < 2; ++pass) {
      ZGemmDesc g;
      g.M = np_; g.N = ncols; g.K = (int)D;
      g.A = Pb; g.sam = 1; g.sak = ldp; g.conjA = true;
      g.B = Y + col0; g.sbk = nc; g.sbn = 1;
      g.C = Cf.p; g.scm = ncols; g.scn = 1;
      g.work = zgemm_work(c);
      {
        ProfScope pg(PROF_ORTHO_GRAM, 0.0, s);
        if (pass == 0) fp64_accurate_zgemm(g, s, 4, OZ_BITS);
        else fp64_accurate_zgemm(g, s);
      }
      ZGemmDesc u;
      u.M = (int)D; u.N = ncols; u.K = np_;
      u.A = Pb; u.sam = ldp; u.sak = 1;
      u.B = Cf.p; u.sbk = ncols; u.sbn = 1;
      u.C = Y + col0; u.scm = nc; u.scn = 1;
      u.alpha = make_cuDoubleComplex(-1.0, 0.0); u.beta = make_cuDoubleComplex(1.0, 0.0);
      u.work = zgemm_work(c);
      u.a_cache = cache_p;
      {
        ProfScope pu(PROF_ORTHO_UPDATE, 0.0, s);
        fp64_accurate_zgemm(u, s);
        if (MY) { u.A = MPb; u.C = MY + col0; u.a_cache = cache_m; fp64_accurate_zgemm(u, s); }
      }
      if (to_cold) {
        if (Cold) {   // Cold (col-major, ld n_cur) += Cf (row-major [n_cur][nc])
          int dims[3] = {np_, ncols, 2};
          int pm[3] = {1, 0, 2};
          permute(reinterpret_cast<const double*>(Cf.p), dims, 3, pm, reinterpret_cast<double*>(Cold), 1.0, 1.0, s);
        }
      } else if (T) {
        add_block_kernel<<<(np_ * ncols + 255) / 256, 256, 0, s>>>(T, nc, col0, Cf.p, np_, ncols);
        GFCC_LAUNCH_CHECK();
      }
    }
  };
  if (n_cur > 0) {
    if (Cold) GFCC_CUDA(cudaMemsetAsync(Cold, 0, sizeof(cplx) * n_cur * nc, s));
    block_cgs(Bs, cap, n_cur, MBs, 0, nc, true);
  }
  DBuf<cplx> partial, h;
  partial.alloc((long long)nchunk * PB);
  h.alloc(PB);
  const dim3 pgrid(1, nchunk), pblock(32, PTY);
  PanelWork pwork;
  std::vector<double> hn0(nc);
  GFCC_CUDA(cudaMemcpyAsync(hn0.data(), n0.p, sizeof(double) * nc, cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  for (int c0 = 0; c0 < nc; c0 += PB) {
    const int pb = std::min(PB, nc - c0);
    if (c0 > 0) block_cgs(Y, nc, c0, MY, c0, pb, false);
    ProfScope pp(PROF_MOR_PANEL, 0.0, s);
    bool done;
    {
      ProfScope pq(PROF_ORTHO_CHOLQR, 0.0, s);
      done = panel_cholqr2(c, Y, MY, nc, D, c0, pb, hn0.data() + c0, T, keep.p, pwork);
    }
    if (done) continue;
    for (int j = c0; j < c0 + pb; ++j) {
      const int n = j - c0;
      if (n > 0) {
        pdot_kernel<<<pgrid, pblock, 0, s>>>(Y, nc, D, c0, n, j, rows, partial.p);
        GFCC_LAUNCH_CHECK();
        preduce_kernel<<<1, pblock, 0, s>>>(partial.p, nchunk, n, h.p, T, nc, c0, j);
        GFCC_LAUNCH_CHECK();
        pupdate_kernel<<<pgrid, pblock, 0, s>>>(Y, MY, nc, D, c0, n, j, rows, h.p, 0, partial.p);
        GFCC_LAUNCH_CHECK();
        preduce_kernel<<<1, pblock, 0, s>>>(partial.p, nchunk, n, h.p, T, nc, c0, j);
        GFCC_LAUNCH_CHECK();
      }
      pupdate_kernel<<<pgrid, pblock, 0, s>>>(Y, MY, nc, D, c0, n, j, rows, h.p, 1, partial.p);
      GFCC_LAUNCH_CHECK();
      pfinish_kernel<<<1, 256, 0, s>>>(partial.p, nchunk, n0.p, j, c->opts.drop_tol, scale.p, keep.p, T, nc);
      GFCC_LAUNCH_CHECK();
      pscale_kernel<<<grid_for(D), 256, 0, s>>>(Y, MY, nc, D, j, scale.p);
      GFCC_LAUNCH_CHECK();
    }
  }
  zgemm_work_check(c);
  std::vector<int> hk(nc);
  GFCC_CUDA(cudaMemcpyAsync(hk.data(), keep.p, sizeof(int) * nc, cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  std::vector<int> kept;
  for (int j = 0; j < nc; ++j)
    if (hk[j]) kept.push_back(j);
  return kept;
}

}  // namespace

// New column capacity of a model buffer that must hold `need` columns: doubling (few regrowths), unless the
// doubled buffers (bytes_per_col per column) would take more than half of the free device memory, in
// which case it grows to what is needed, rounded up to `quantum` (the old buffer is still held while the
// columns are copied, and large models at the biggest sizes are limited by memory, not by regrowths).
static int grown_capacity(gfcc_ctx* c, int cap_now, int need, int quantum, double bytes_per_col) {
  int cap = std::max(need, std::max(quantum, 2 * cap_now));
  size_t freeb = device_free_bytes();
  if (freeb == 0) return cap;
  if ((double)cap * bytes_per_col > 0.5 * (double)freeb) {
    // memory is short: give back the scratch buffers first (they regrow on demand), then size exactly
    release_scratch(c);
    freeb = device_free_bytes();
    if ((double)cap * bytes_per_col > 0.5 * (double)freeb)
      cap = std::max(need, ((need + quantum - 1) / quantum) * quantum);
  }
  return cap;
}

void release_scratch(gfcc_ctx* c) {
  GFCC_CUDA(cudaStreamSynchronize(c->stream));
  release_sigma_batch_buffers(c);
  c->ws.ut.release();
  c->ws.ct.release();
  c->ws.xe.release();
  c->ws.nb_cap = 0;
  zgemm_work_check(c);
  zgemm_work_free(c);
  GFCC_CUDA(cudaStreamSynchronize(c->stream));   // the frees have reached the pool before memory is measured
}

static void grow_model(gfcc_ctx* c, int need) {
  MorState& ms = c->mor;
  if (need <= ms.m_cap) return;
  const int np = (int)ms.porb.size(), nq = (int)ms.qorb.size();
  const int cap = grown_capacity(c, ms.m_cap, need, 64, 2.0 * (double)c->D * sizeof(cplx));   // S and Z
  cudaStream_t s = c->stream;
  regrow_rows(ms.S, c->D, ms.m_cap, cap, ms.m, s);
  regrow_rows(ms.Z, c->D, ms.m_cap, cap, ms.m, s);
  regrow_cm(ms.Hh, ms.m_cap, cap, cap, ms.m, ms.m, s);
  regrow_cm(ms.bh, ms.m_cap, cap, np, ms.m, np, s);
  regrow_cm(ms.ch, nq, nq, cap, nq, ms.m, s);
  regrow_cm(ms.RS, ms.q_cap, ms.q_cap, cap, ms.qn, ms.m, s);
  regrow_cm(ms.RZ, ms.q_cap, ms.q_cap, cap, ms.qn, ms.m, s);
  ms.m_cap = cap;
}

static void grow_basis(gfcc_ctx* c, int need) {
  MorState& ms = c->mor;
  if (need <= ms.q_cap) return;
  const int np = (int)ms.porb.size();
  const int cap = grown_capacity(c, ms.q_cap, need, 128, (double)c->D * sizeof(cplx));
  cudaStream_t s = c->stream;
  regrow_rows(ms.Q, c->D, ms.q_cap, cap, ms.qn, s);
  regrow_cm(ms.RS, ms.q_cap, cap, std::max(ms.m_cap, 1), ms.qn, ms.m, s);
  regrow_cm(ms.RZ, ms.q_cap, cap, std::max(ms.m_cap, 1), ms.qn, ms.m, s);
  regrow_cm(ms.RB, ms.q_cap, cap, np, ms.qn, np, s);
  ms.q_cap = cap;
}

// Append the kept columns of Ynew ([D][nc], destroyed) to Q and return, col-major [qn_new x nc], the
// coefficients of the ORIGINAL columns of Ynew in the enlarged basis (host memory).
static std::vector<cplx> basis_append(gfcc_ctx* c, cplx* Ynew, int nc) {
  MorState& ms = c->mor;
  cudaStream_t s = c->stream;
  ProfScope prof(PROF_MOR_BASIS, 0.0, s);
  const long long D = c->D;
  const int qn0 = ms.qn;
  DBuf<cplx> Cold, T;
  Cold.alloc((long long)std::max(qn0, 1) * nc);
  T.alloc((long long)nc * nc);
  std::vector<int> kept = ortho_block(c, ms.Q.p, ms.q_cap, qn0, Ynew, nullptr, nullptr, nc,
                                      qn0 > 0 ? Cold.p : nullptr, T.p);
  const int acc = (int)kept.size();
  grow_basis(c, qn0 + acc);
  if (acc > 0) {
    DBuf<int> dk;
    dk.alloc(acc);
    GFCC_CUDA(cudaMemcpyAsync(dk.p, kept.data(), sizeof(int) * acc, cudaMemcpyHostToDevice, s));
    append_cols_kernel<<<grid_for(D * acc), 256, 0, s>>>(Ynew, nc, dk.p, acc, ms.Q.p, ms.q_cap, qn0, D);
    GFCC_LAUNCH_CHECK();
    GFCC_CUDA(cudaStreamSynchronize(s));
  }
  const int qn1 = qn0 + acc;
  ms.qn = qn1;
  std::vector<cplx> hC((size_t)std::max(qn0, 1) * nc), hT((size_t)nc * nc);
  if (qn0 > 0) GFCC_CUDA(cudaMemcpyAsync(hC.data(), Cold.p, sizeof(cplx) * qn0 * nc, cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaMemcpyAsync(hT.data(), T.p, sizeof(cplx) * nc * nc, cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  std::vector<cplx> out((size_t)qn1 * nc, make_cuDoubleComplex(0.0, 0.0));
  for (int j = 0; j < nc; ++j) {
    for (int i = 0; i < qn0; ++i) out[(size_t)j * qn1 + i] = hC[(size_t)j * qn0 + i];
    for (int r = 0; r < acc; ++r) out[(size_t)j * qn1 + qn0 + r] = hT[(size_t)j * nc + kept[r]];
  }
  return out;
}

// write coefficient columns (host, col-major [rows x ncols]) into a device col-major matrix
static void put_cols(DBuf<cplx>& R, int ld, int col0, const std::vector<cplx>& h, int rows, int hcol0, int ncols,
                     cudaStream_t s) {
  if (ncols <= 0 || rows <= 0) return;
  GFCC_CUDA(cudaMemcpy2DAsync(R.p + (long long)col0 * ld, sizeof(cplx) * ld, h.data() + (size_t)hcol0 * rows,
                              sizeof(cplx) * rows, sizeof(cplx) * rows, ncols, cudaMemcpyHostToDevice, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
}

void mor_init_basis(gfcc_ctx* c) {
  MorState& ms = c->mor;
  ++ms.version;
  cudaStream_t s = c->stream;
  const long long D = c->D;
  const int np = (int)ms.porb.size();
  DBuf<cplx> Bc;
  DBuf<int> rows;
  Bc.alloc(D * np);
  rows.alloc(np);
  GFCC_CUDA(cudaMemcpyAsync(rows.p, ms.porb.data(), sizeof(int) * np, cudaMemcpyHostToDevice, s));
  gather_rows_real_to_cplx(c->bvec.p, (int)D, rows.p, np, (int)D, Bc.p, np, s);
  GFCC_CUDA(cudaStreamSynchronize(s));
  std::vector<cplx> coef = basis_append(c, Bc.p, np);
  grow_basis(c, ms.qn);
  put_cols(ms.RB, ms.q_cap, 0, coef, ms.qn, 0, np, s);
}

void mor_append(gfcc_ctx* c, const cplx* Xin, const cplx* MXin, int nc) {
  MorState& ms = c->mor;
  ++ms.version;   // the model changes: its cached Hessenberg form is stale
  cudaStream_t s = c->stream;
  ProfScope prof(PROF_MOR_ORTHO, 0.0, s);
  const long long D = c->D;
  const int np = (int)ms.porb.size(), nq = (int)ms.qorb.size();
  if (nc == 0) return;
  DBuf<cplx> Y, MY;
  Y.alloc(D * nc);
  MY.alloc(D * nc);
  GFCC_CUDA(cudaMemcpyAsync(Y.p, Xin, sizeof(cplx) * D * nc, cudaMemcpyDeviceToDevice, s));
  GFCC_CUDA(cudaMemcpyAsync(MY.p, MXin, sizeof(cplx) * D * nc, cudaMemcpyDeviceToDevice, s));
  std::vector<int> kept = ortho_block(c, ms.S.p, ms.m_cap, ms.m, Y.p, MY.p, ms.Z.p, nc, nullptr, nullptr);
  const int acc = (int)kept.size();
  if (acc == 0) return;
  const int m0 = ms.m, m1 = ms.m + acc;
  grow_model(c, m1);
  const int cap = ms.m_cap;
  DBuf<cplx> SZ;   // [S_new | Z_new] for the residual basis
  SZ.alloc(D * 2 * acc);
  {
    DBuf<int> dk, di;
    dk.alloc(acc);
    di.alloc(acc);
    std::vector<int> iota(acc);
    for (int k = 0; k < acc; ++k) iota[k] = k;
    GFCC_CUDA(cudaMemcpyAsync(dk.p, kept.data(), sizeof(int) * acc, cudaMemcpyHostToDevice, s));
    append_cols_kernel<<<grid_for(D * acc), 256, 0, s>>>(Y.p, nc, dk.p, acc, ms.S.p, cap, m0, D);
    GFCC_LAUNCH_CHECK();
    append_cols_kernel<<<grid_for(D * acc), 256, 0, s>>>(MY.p, nc, dk.p, acc, ms.Z.p, cap, m0, D);
    GFCC_LAUNCH_CHECK();
    append_cols_kernel<<<grid_for(D * acc), 256, 0, s>>>(Y.p, nc, dk.p, acc, SZ.p, 2 * acc, 0, D);
    GFCC_LAUNCH_CHECK();
    append_cols_kernel<<<grid_for(D * acc), 256, 0, s>>>(MY.p, nc, dk.p, acc, SZ.p, 2 * acc, acc, D);
    GFCC_LAUNCH_CHECK();
    GFCC_CUDA(cudaStreamSynchronize(s));
  }
  auto proj = [&](const cplx* Lp, int l0, int nl, const cplx* Rp, int r0, int nr, long long ldr_rows,
                  cplx* Cp, long long scm, long long scn) {
    // C(i, j) = sum_nu conj(L[nu][l0+i]) R[nu][r0+j]
    ZGemmDesc g;
    g.M = nl; g.N = nr; g.K = (int)D;
    g.A = Lp + l0; g.sam = 1; g.sak = cap; g.conjA = true;
    g.B = Rp + r0; g.sbk = ldr_rows; g.sbn = 1;
    g.C = Cp; g.scm = scm; g.scn = scn;
    g.work = zgemm_work(c);
    zgemm(g, s);
  };
  // Hhat[0:m1, m0:m1] = S^H Z_new ; Hhat[m0:m1, 0:m0] = S_new^H Z_old
  proj(ms.S.p, 0, m1, ms.Z.p, m0, acc, cap, ms.Hh.p + (long long)m0 * cap, 1, cap);
  if (m0 > 0) proj(ms.S.p, m0, acc, ms.Z.p, 0, m0, cap, ms.Hh.p + m0, 1, cap);
  DBuf<cplx> Bc, Cc;
  Bc.alloc(D * np);
  Cc.alloc(D * nq);
  {
    DBuf<int> rows_p, rows_q;
    rows_p.alloc(np); rows_q.alloc(nq);
    GFCC_CUDA(cudaMemcpyAsync(rows_p.p, ms.porb.data(), sizeof(int) * np, cudaMemcpyHostToDevice, s));
    GFCC_CUDA(cudaMemcpyAsync(rows_q.p, ms.qorb.data(), sizeof(int) * nq, cudaMemcpyHostToDevice, s));
    gather_rows_real_to_cplx(c->bvec.p, (int)D, rows_p.p, np, (int)D, Bc.p, np, s);
    gather_rows_real_to_cplx(c->cvec.p, (int)D, rows_q.p, nq, (int)D, Cc.p, nq, s);
    GFCC_CUDA(cudaStreamSynchronize(s));
  }
  proj(ms.S.p, m0, acc, Bc.p, 0, np, np, ms.bh.p + m0, 1, cap);
  {  // chat[q][m0+i] = sum_nu Cc[nu][q] S[nu][m0+i]
    ZGemmDesc g;
    g.M = nq; g.N = acc; g.K = (int)D;
    g.A = Cc.p; g.sam = 1; g.sak = nq;
    g.B = ms.S.p + m0; g.sbk = cap; g.sbn = 1;
    g.C = ms.ch.p + (long long)m0 * nq; g.scm = 1; g.scn = nq;
    g.work = zgemm_work(c);
    zgemm(g, s);
  }
  GFCC_CUDA(cudaStreamSynchronize(s));
  ms.m = m1;
  // residual basis: coefficients of S_new and Z_new in Q
  std::vector<cplx> coef = basis_append(c, SZ.p, 2 * acc);
  grow_basis(c, ms.qn);
  grow_model(c, m1);
  put_cols(ms.RS, ms.q_cap, m0, coef, ms.qn, 0, acc, s);
  put_cols(ms.RZ, ms.q_cap, m0, coef, ms.qn, acc, acc, s);
  zgemm_work_check(c);
}

// Hessenberg form of the current reduced model, computed once per model version and reused by every
// evaluation and extrapolation: Householder reflections H_j = I - tau_j v_j v_j^H (j = 0..m-3),
// H = P^H Hhat P with P = H_0 H_1 ...; the left reflections go to bhat, the right ones to chat and
// (want_res) to the residual coefficient matrices.
static void hessenberg(gfcc_ctx* c, bool want_res) {
  MorState& ms = c->mor;
  if (ms.hess_version == ms.version && (!want_res || (ms.hess_res && ms.hess_qn == ms.qn))) return;
  cudaStream_t s = c->stream;
  ProfScope prof_h(PROF_EVAL_HESS, 0.0, s);
  const int m = ms.m, np = (int)ms.porb.size(), nq = (int)ms.qorb.size(), cap = ms.m_cap, qn = ms.qn;
  ms.hH.alloc((long long)m * m); ms.hb.alloc((long long)m * np); ms.hc.alloc((long long)nq * m);
  ms.hV.alloc((long long)m * m); ms.htau.alloc(m);
  cplx *Hw = ms.hH.p, *bw = ms.hb.p, *cw = ms.hc.p;
  GFCC_CUDA(cudaMemcpy2DAsync(Hw, sizeof(cplx) * m, ms.Hh.p, sizeof(cplx) * cap, sizeof(cplx) * m, m,
                              cudaMemcpyDeviceToDevice, s));
  GFCC_CUDA(cudaMemcpy2DAsync(bw, sizeof(cplx) * m, ms.bh.p, sizeof(cplx) * cap, sizeof(cplx) * m, np,
                              cudaMemcpyDeviceToDevice, s));
  GFCC_CUDA(cudaMemcpyAsync(cw, ms.ch.p, sizeof(cplx) * nq * m, cudaMemcpyDeviceToDevice, s));
  cplx *A1 = nullptr, *A2 = nullptr;
  if (want_res) {
    ms.hA1.alloc((long long)qn * m); ms.hA2.alloc((long long)qn * m); ms.hRB.alloc((long long)qn * np);
    A1 = ms.hA1.p; A2 = ms.hA2.p;
    GFCC_CUDA(cudaMemcpy2DAsync(A1, sizeof(cplx) * qn, ms.RS.p, sizeof(cplx) * ms.q_cap, sizeof(cplx) * qn, m,
                                cudaMemcpyDeviceToDevice, s));
    GFCC_CUDA(cudaMemcpy2DAsync(A2, sizeof(cplx) * qn, ms.RZ.p, sizeof(cplx) * ms.q_cap, sizeof(cplx) * qn, m,
                                cudaMemcpyDeviceToDevice, s));
    GFCC_CUDA(cudaMemcpy2DAsync(ms.hRB.p, sizeof(cplx) * qn, ms.RB.p, sizeof(cplx) * ms.q_cap, sizeof(cplx) * qn, np,
                                cudaMemcpyDeviceToDevice, s));
  }
  DBuf<cplx> wv;
  wv.alloc((long long)m + nq + 2LL * qn + 1);
  RightMats rm;
  rm.n = 0;
  auto add = [&](cplx* p, long long ld, int rows) {
    if (rows > 0) { rm.p[rm.n] = p; rm.ld[rm.n] = ld; rm.rows[rm.n] = rows; ++rm.n; }
  };
  add(Hw, m, m);
  add(cw, nq, nq);
  if (want_res) { add(A1, qn, qn); add(A2, qn, qn); }
  long long rows_all = 0, tiles_all = 0;
  for (int k = 0; k < rm.n; ++k) {
    rows_all += rm.rows[k];
    tiles_all += (rm.rows[k] + 31) / 32;
  }
  for (int j = 0; j + 2 < m; ++j) {
    const int len = m - j - 1;
    cplx* v = ms.hV.p + (long long)j * m;
    double* tau = ms.htau.p + j;
    house_kernel<<<1, 256, 0, s>>>(Hw + (long long)j * m + j + 1, len, v, tau);
    GFCC_LAUNCH_CHECK();
    // left: columns j.. of H and all np columns of bhat
    house_left2_kernel<<<(m - j) + np, 256, 0, s>>>(Hw, m, j, m - j, bw, m, np, j + 1, len, v, tau);
    GFCC_LAUNCH_CHECK();
    // right: H, chat and the residual coefficient matrices
    house_right_w4_kernel<<<(unsigned)tiles_all, 256, 0, s>>>(rm, j + 1, len, v, wv.p);
    GFCC_LAUNCH_CHECK();
    house_right_update4_kernel<<<grid_for(rows_all * len), 256, 0, s>>>(rm, j + 1, len, v, wv.p, tau,
                                                                        rows_all * len);
    GFCC_LAUNCH_CHECK();
  }
  {  // the evaluation reads H and bhat by rows
    ms.hHr.alloc((long long)m * m);
    ms.hbr.alloc((long long)m * np);
    int dh[3] = {m, m, 2}, db[3] = {np, m, 2}, pm[3] = {1, 0, 2};
    permute(reinterpret_cast<const double*>(Hw), dh, 3, pm, reinterpret_cast<double*>(ms.hHr.p), 1.0, 0.0, s);
    permute(reinterpret_cast<const double*>(bw), db, 3, pm, reinterpret_cast<double*>(ms.hbr.p), 1.0, 0.0, s);
  }
  GFCC_CUDA(cudaStreamSynchronize(s));   // wv is released on return
  ms.hess_version = ms.version;
  ms.hess_res = want_res;
  ms.hess_qn = qn;
}

void mor_eval(gfcc_ctx* c, const double* omegas_host, int nw, cplx* G_dev, double* A_dev, double* maxres_dev,
              cplx* dG_dev) {
  MorState& ms = c->mor;
  cudaStream_t s = c->stream;
  ProfScope prof(PROF_MOR_EVAL, 0.0, s);
  const int m = ms.m, np = (int)ms.porb.size(), nq = (int)ms.qorb.size(), qn = ms.qn;
  GFCC_CHECK(m > 0, GFCC_ERR_STATE, "mor_eval: empty reduced model");
  const bool want_res = maxres_dev != nullptr;
  hessenberg(c, want_res);
  const cplx* cw = ms.hc.p;
  const cplx *A1 = ms.hA1.p, *A2 = ms.hA2.p, *RBw = ms.hRB.p;
  DBuf<double> dbn;
  std::vector<int> qidx(np, -1);
  for (int p = 0; p < np; ++p)
    for (int q = 0; q < nq; ++q)
      if (ms.qorb[q] == ms.porb[p]) { qidx[p] = q; break; }
  DBuf<int> dq, dsing;
  DBuf<double> dom;
  dq.alloc(np); dsing.alloc(1); dom.alloc(nw); dbn.alloc(np);
  dsing.zero(s);
  GFCC_CUDA(cudaMemcpyAsync(dq.p, qidx.data(), sizeof(int) * np, cudaMemcpyHostToDevice, s));
  GFCC_CUDA(cudaMemcpyAsync(dom.p, omegas_host, sizeof(double) * nw, cudaMemcpyHostToDevice, s));
  GFCC_CUDA(cudaMemcpyAsync(dbn.p, ms.bnorm.data(), sizeof(double) * np, cudaMemcpyHostToDevice, s));
  // frequencies in batches: solutions Y [m][nb np] of a batch (about 2 GB at most), then Ghat = chat^T Y
  // and the residual coefficients (w - i eta) RS Y + RZ Y - RB as complex GEMMs over the whole batch
  const long long bw_max = std::max<long long>(1, (2LL << 30) / ((long long)m * np * (long long)sizeof(cplx)));
  const int nbw = (int)std::min<long long>(nw, bw_max);
  DBuf<cplx> Y, Ys, Cr, Gt, Yd;
  DBuf<double> rcol;
  EvalScratch es;
  eval_scratch_alloc(es, m, np, nbw);
  Y.alloc((long long)m * nbw * np);
  const bool want_G = G_dev != nullptr || A_dev != nullptr;
  if (want_G && !G_dev) Gt.alloc((long long)nbw * np * nq);
  if (dG_dev) Yd.alloc((long long)m * nbw * np);
  if (want_res) {
    Ys.alloc((long long)m * nbw * np);
    Cr.alloc((long long)qn * nbw * np);
    rcol.alloc((long long)nbw * np);
  }
  for (int w0 = 0; w0 < nw; w0 += nbw) {
    const int nb = std::min(nbw, nw - w0);
    const long long ldy = (long long)nb * np;
    EvalArgs ea;
    ea.m = m; ea.np = np; ea.nw = nb;
    ea.H = ms.hHr.p; ea.b = ms.hbr.p;
    ea.omegas = dom.p + w0; ea.eta = ms.eta;
    ea.Y = Y.p; ea.ldy = ldy; ea.singular = dsing.p;
    {
      ProfScope ps(PROF_EVAL_SOLVE, 0.0, s);
      launch_eval_solve(ea, es, s);
    }
    if (want_G) {   // G(q, n) = sum_k cw[q][k] Y[k][n], stored at Gb[n nq + q]
      cplx* Gb = G_dev ? G_dev + (long long)w0 * np * nq : Gt.p;
      ZGemmDesc g;
      g.M = nq; g.N = (int)ldy; g.K = m;
      g.A = cw; g.sam = 1; g.sak = nq;
      g.B = Y.p; g.sbk = ldy; g.sbn = 1;
      g.C = Gb; g.scm = 1; g.scn = nq;
      g.work = zgemm_work(c);
      zgemm(g, s);
      if (A_dev) {
        spectral_from_G_kernel<<<(nb + 127) / 128, 128, 0, s>>>(Gb, nb, np, nq, dq.p, A_dev + w0);
        GFCC_LAUNCH_CHECK();
      }
    }
    if (dG_dev) {   // dGhat/dw = -chat^T (w - i eta + H)^{-2} bhat: a second solve with y as right side
      GFCC_CUDA(cudaMemcpyAsync(Yd.p, Y.p, sizeof(cplx) * m * ldy, cudaMemcpyDeviceToDevice, s));
      EvalArgs eb = ea;
      eb.Y = Yd.p;
      eb.b = nullptr;
      launch_eval_solve(eb, es, s);
      ZGemmDesc g;
      g.M = nq; g.N = (int)ldy; g.K = m;
      g.A = cw; g.sam = 1; g.sak = nq;
      g.B = Yd.p; g.sbk = ldy; g.sbn = 1;
      g.C = dG_dev + (long long)w0 * np * nq; g.scm = 1; g.scn = nq;
      g.alpha = make_cuDoubleComplex(-1.0, 0.0);
      g.work = zgemm_work(c);
      zgemm(g, s);
    }
    if (want_res) {   // coefficients of r = (w - i eta) S y + Z y - b in the orthonormal residual basis
      shift_scale_kernel<<<grid_for((long long)m * ldy), 256, 0, s>>>(Y.p, ldy, m, np, nb, dom.p + w0, ms.eta, Ys.p);
      GFCC_LAUNCH_CHECK();
      ZGemmDesc g;
      g.M = qn; g.N = (int)ldy; g.K = m;
      g.A = A1; g.sam = 1; g.sak = qn;
      g.B = Ys.p; g.sbk = ldy; g.sbn = 1;
      g.C = Cr.p; g.scm = ldy; g.scn = 1;
      g.work = zgemm_work(c);
      zgemm(g, s);
      g.A = A2; g.B = Y.p; g.beta = make_cuDoubleComplex(1.0, 0.0);
      g.work = zgemm_work(c);
      zgemm(g, s);
      resnorm_kernel<<<(unsigned)((ldy + 255) / 256), 256, 0, s>>>(Cr.p, ldy, qn, RBw, np, nb, dbn.p, rcol.p);
      GFCC_LAUNCH_CHECK();
      rowmax_kernel<<<(nb + 127) / 128, 128, 0, s>>>(rcol.p, np, nb, maxres_dev + w0);
      GFCC_LAUNCH_CHECK();
    }
  }
  int hs = 0;
  GFCC_CUDA(cudaMemcpyAsync(&hs, dsing.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  GFCC_CHECK(hs == 0, GFCC_ERR_NONFINITE, "mor_eval: singular reduced system at a requested frequency");
  zgemm_work_check(c);
}

// Initial guesses for new frequencies: x0_p(w) = S yhat_p(w) with (w - i eta + Hhat) yhat_p = bhat_p.
// Hhat is reduced to Hessenberg form H = P^H Hhat P by Householder reflections (recorded), each
// frequency is a shifted Hessenberg solve (launch_eval_solve), yhat = P y_H applies the reflections
// in reverse order, and X0 = S yhat is one complex GEMM. X0: [D][nw np] batch-minor (column w np + p).
void mor_extrapolate(gfcc_ctx* c, const double* omegas_host, int nw, cplx* X0) {
  MorState& ms = c->mor;
  cudaStream_t s = c->stream;
  const int m = ms.m, np = (int)ms.porb.size(), cap = ms.m_cap;
  GFCC_CHECK(m > 0, GFCC_ERR_STATE, "mor_extrapolate: empty reduced model");
  const long long N = (long long)nw * np;
  hessenberg(c, false);
  DBuf<cplx> Y;
  DBuf<double> dom;
  DBuf<int> dsing;
  EvalScratch es;
  eval_scratch_alloc(es, m, np, nw);
  Y.alloc((long long)m * N);
  dom.alloc(nw); dsing.alloc(1);
  dsing.zero(s);
  GFCC_CUDA(cudaMemcpyAsync(dom.p, omegas_host, sizeof(double) * nw, cudaMemcpyHostToDevice, s));
  EvalArgs ea;
  ea.m = m; ea.np = np; ea.nw = nw;
  ea.H = ms.hHr.p; ea.b = ms.hbr.p;
  ea.omegas = dom.p; ea.eta = ms.eta;
  ea.Y = Y.p; ea.ldy = N; ea.singular = dsing.p;
  launch_eval_solve(ea, es, s);
  for (int j = m - 3; j >= 0; --j) {   // yhat = P y_H, P = H_0 H_1 ... (Hermitian reflectors)
    house_rows_kernel<<<(unsigned)((N + 127) / 128), 128, 0, s>>>(Y.p, N, N, j + 1, m - j - 1,
                                                                  ms.hV.p + (long long)j * m, ms.htau.p + j);
    GFCC_LAUNCH_CHECK();
  }
  ZGemmDesc g;   // X0[nu][n] = sum_k S[nu][k] yhat[k][n]
  g.M = (int)c->D; g.N = (int)N; g.K = m;
  g.A = ms.S.p; g.sam = cap; g.sak = 1;
  g.B = Y.p; g.sbk = N; g.sbn = 1;
  g.C = X0; g.scm = N; g.scn = 1;
  g.work = zgemm_work(c);
  zgemm(g, s);
  int hs = 0;
  GFCC_CUDA(cudaMemcpyAsync(&hs, dsing.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  GFCC_CHECK(hs == 0, GFCC_ERR_NONFINITE, "mor_extrapolate: singular reduced system at a new frequency");
  zgemm_work_check(c);
}

}  // namespace gfcc

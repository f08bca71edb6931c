// Batched restarted GMRES with iterative refinement for the shifted systems of Eq. xplin,
// (w_c - i eta + M) x_c = b_c, one column per (p, w) pair, all columns in lock step.
//
// Each restart cycle is one refinement step: the residual r = b - (shift x + M x) is formed with
// the FP64 sigma, then GMRES(k) on the correction runs with the sigma in the requested
// precision (classical Gram-Schmidt with one re-orthogonalisation, Givens least squares), and
// x += P V y with the Jacobi right preconditioner P = (shift + diag M)^{-1}.
// Columns whose FP64 residual meets the tolerance are written out and compacted away between
// cycles. The paper used a complex DIIS solver (convergence study after Table 1); any convergent
// solver reaches the same solution of Eq. xplin.
#include "gfcc_internal.cuh"
#include "precond.cuh"

#include <type_traits>

#include <algorithm>
#include <cmath>

namespace gfcc {
namespace {

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)std::min<long long>(std::max<long long>(g, 1), 152LL * 32);
}

// real component type of a complex vector element
template <typename VT> struct RealOf;
template <> struct RealOf<cplx> { using type = double; };
template <> struct RealOf<cuFloatComplex> { using type = float; };

constexpr int MD_TX = 32, MD_TY = 8, MD_MAXV = 32;   // blocks of the sweeps; basis vectors per sweep
// The kernels below are instantiated for NV = 4, 8, 16, 32 basis vectors (nv <= NV used).
template <typename F>
void with_nv(int nv, F&& f) {
  if (nv <= 4) f(std::integral_constant<int, 4>{});
  else if (nv <= 8) f(std::integral_constant<int, 8>{});
  else if (nv <= 16) f(std::integral_constant<int, 16>{});
  else f(std::integral_constant<int, 32>{});
}

// partial[chunk][i][c] = sum_{nu in chunk} conj(V_i[nu][c]) W[nu][c], i < nv (V_i = V + i*stride);
// per-thread sums in the vector's precision, partials written in FP64.
// Block (MD_TX columns) x (MD_TY): the MD_TY thread rows form IG = NV/8 groups (at least 1); group g
// owns the accumulators of basis vectors g, g + IG, ... (NPG = NV / IG at most), and its threads stride the
// chunk's rows by MD_TY / IG. Fewer accumulators per thread keep the registers, and so the number of
// resident warps, independent of the basis size; the groups' shares differ by one vector at most (with contiguous
// shares of 8 the groups of one warp scheduler held 14 of 22 vectors, those of another 8). Bound by the FP64 pipe:
// the products go into the sums by two multiply-adds per component (a sum of products added on would be a product, a
// multiply-add and an addition). 560 columns of D = 3,836, 17 to 28 vectors: 675 -> 523 us; update_kernel 382 -> 246 us
// (92 % of the FP64 rate); norms 77 us -> 12.
template <int NV> struct MdGroups {
  static constexpr int IG = NV >= 16 ? NV / 8 : 1;
  static constexpr int NPG = NV / IG;
  static constexpr int RPG = MD_TY / IG;   // thread rows per group
};
// sum the per-thread values acc[li] of group g over its RPG thread rows; partial for i = li IG + g
template <typename VT, int NV, typename R>
__device__ __forceinline__ void md_reduce(const R (&ax)[MdGroups<NV>::NPG], const R (&ay)[MdGroups<NV>::NPG], int nv,
                                          int c, int nb, cplx* __restrict__ partial, cplx (*red)[MD_TX]) {
  using G = MdGroups<NV>;
  const int g = threadIdx.y / G::RPG, yr = threadIdx.y % G::RPG;
#pragma unroll
  for (int li = 0; li < G::NPG; ++li) {
    red[threadIdx.y][threadIdx.x] = make_cuDoubleComplex((double)ax[li], (double)ay[li]);
    __syncthreads();
    const int i = li * G::IG + g;
    if (yr == 0 && c < nb && i < nv) {
      cplx s = red[threadIdx.y][threadIdx.x];
      for (int k = 1; k < G::RPG; ++k) { s.x += red[threadIdx.y + k][threadIdx.x].x; s.y += red[threadIdx.y + k][threadIdx.x].y; }
      partial[((long long)blockIdx.y * nv + i) * nb + c] = s;
    }
    __syncthreads();
  }
}

template <typename VT, int NV>
__global__ void __launch_bounds__(256, 2) multidot_kernel(const VT* __restrict__ V, long long vstride, int nv,
                                                          const VT* __restrict__ W, long long D, int nb,
                                                          long long rows_per_chunk, cplx* __restrict__ partial) {
  using R = typename RealOf<VT>::type;
  using G = MdGroups<NV>;
  __shared__ cplx red[MD_TY][MD_TX];
  const int c = blockIdx.x * MD_TX + threadIdx.x;
  const int g = threadIdx.y / G::RPG, yr = threadIdx.y % G::RPG;
  const long long r0 = blockIdx.y * rows_per_chunk;
  const long long r1 = min(D, r0 + rows_per_chunk);
  const VT* Vg = V + (long long)g * vstride;
  const int ng = (nv - g + G::IG - 1) / G::IG;   // vectors of this group present (may be <= 0)
  R ax[G::NPG], ay[G::NPG];
#pragma unroll
  for (int i = 0; i < G::NPG; ++i) { ax[i] = R(0); ay[i] = R(0); }
  if (c < nb && ng > 0) {
    for (long long nu = r0 + yr; nu < r1; nu += G::RPG) {
      const VT w = W[nu * nb + c];
      VT vv[G::NPG];   // all loads of a row before its arithmetic
#pragma unroll
      for (int i = 0; i < G::NPG; ++i) vv[i] = i < ng ? Vg[i * G::IG * vstride + nu * nb + c] : w;
#pragma unroll
      for (int i = 0; i < G::NPG; ++i) {
        if (i < ng) {
          ax[i] = fma(vv[i].x, w.x, fma(vv[i].y, w.y, ax[i]));
          ay[i] = fma(vv[i].x, w.y, fma(-vv[i].y, w.x, ay[i]));
        }
      }
    }
  }
  md_reduce<VT, NV, R>(ax, ay, nv, c, nb, partial, red);
}

// partial[chunk][c].x = sum_{nu in chunk} |W[nu][c]|^2 (block MD_TX columns x MD_TY rows, four rows of a thread in
// flight)
template <typename VT>
__global__ void __launch_bounds__(256) norm_partial_kernel(const VT* __restrict__ W, long long D, int nb,
                                                           long long rows_per_chunk, cplx* __restrict__ partial) {
  using R = typename RealOf<VT>::type;
  __shared__ double red[MD_TY][MD_TX];
  const int c = blockIdx.x * MD_TX + threadIdx.x;
  const long long r0 = blockIdx.y * rows_per_chunk, r1 = min(D, r0 + rows_per_chunk);
  R a[4] = {R(0), R(0), R(0), R(0)};
  if (c < nb)
    for (long long nu = r0 + threadIdx.y; nu < r1; nu += 4 * MD_TY) {
      VT w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = nu + u * MD_TY < r1;
        w[u] = W[(in ? nu + u * MD_TY : nu) * nb + c];
        if (!in) w[u].x = w[u].y = R(0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = fma(w[u].x, w[u].x, fma(w[u].y, w[u].y, a[u]));
    }
  red[threadIdx.y][threadIdx.x] = (double)((a[0] + a[1]) + (a[2] + a[3]));
  __syncthreads();
  if (threadIdx.y == 0 && c < nb) {
    double s = red[0][threadIdx.x];
    for (int k = 1; k < MD_TY; ++k) s += red[k][threadIdx.x];
    partial[(long long)blockIdx.y * nb + c] = make_cuDoubleComplex(s, 0.0);
  }
}

// ---- pipelined Gram-Schmidt sweeps of the FP32 basis ---------------------------------------------
// Classical Gram-Schmidt with re-orthogonalisation, the second pass of a vector delayed by one step, so that it shares
// its reads of the basis with the first pass of the next vector (the basis is read twice per step instead of three
// times, the sweeps being HBM-bound). At step j, with V_0 .. V_{j-1} final, a the normalised vector that has had its
// first pass and u the image of a:
//   sweep DOTS:    g_i = V_i^H a, r_i = V_i^H u (i < j), a^H a, a^H u
//   coefficients:  rho^2 = a^H a - |g|^2, s = (a^H u - g^H r) / rho; Hessenberg column (r_0 .. r_{j-1}, s)
//   sweep UPDATE:  V_j = (a - V g) / rho,  u -= V r + V_j s (u has had its first pass), partial sums of |u|^2
// What this leaves out, with w the image whose first pass gave hn a: a = V g + rho V_j, so that column j - 1 would gain hn g
// and its subdiagonal be hn rho. Both are at most |g| hn, and g is the rounding of the first pass, a few 2^-24 ||w|| / hn:
// the Arnoldi relation of that column holds to a few 2^-24 ||w||, however much the pass cancelled. Column j has the
// image u of a in the place of that of V_j, |g| ||A|| off: less than the rounding of the low-precision action itself (2^-11
// in TF32) while the pass cancels less than a factor of some thousand, more beyond that. It costs steps, not accuracy: the
// residual of every cycle is recomputed. A vector of which the second pass takes more than half (rho^2 <= a^H a / 2; the
// criterion of Daniel, Gragg, Kaufman and Stewart, Math. Comp. 30 (1976)) is rounding noise: its column ends its cycle with
// the vectors before it, so that 1 / rho is never above sqrt 2.
// (o = 30, v = 130, TF32 solves to 1e-10: kernels of the whole solve 276 -> 247 ms, all of it the sweeps; the numbers
// of Arnoldi steps did not change by more than 2 in 440.)
//
// The loads are decoupled from the arithmetic: every thread streams its own elements (its NPG basis vectors, a and u
// at one row per step) through a SW_STAGES-deep ring in shared memory by 8-byte asynchronous copies (cp.async,
// zero-filled outside the batch), so that about three steps of loads are in flight per block without holding
// registers. A block is CW columns wide (32, 16, 8 or 4: narrow batches keep every thread busy) and
// SW_THREADS / CW thread rows high; the thread rows form IG groups that each own NPG basis vectors, and the groups'
// shares of V g and V r are added through shared memory. Each thread reads only the ring slots it filled itself.
// Bases of more than MD_MAXV vectors take a pair of sweeps per MD_MAXV of them.
constexpr int SW_THREADS = 256, SW_STAGES = 4;
template <int NV> struct SwGroups {
  static constexpr int IG = NV >= 16 ? NV / 8 : 1;
  static constexpr int NPG = NV / IG;
};
template <int NV, int CW> constexpr size_t sweep_smem_bytes() {
  return sizeof(float2) * (size_t)SW_STAGES * (SwGroups<NV>::NPG + 2) * SW_THREADS   // load ring
         + sizeof(float4) * 2 * SW_THREADS;                                          // shares
}

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, bool pred) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(gmem), "r"(pred ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

struct SweepArgs {
  const float2* V;        // the nv basis vectors of this sweep (stride vstride)
  long long vstride;
  int nv;
  float2 *a, *u;          // read (DOTS), read and written (UPDATE)
  long long D;
  int nb;
  long long rows_per_chunk;
  // DOTS: partial[chunk][q][c], q < 2 nv (+ 2 when scalars): g_0 .. g_{nv-1}, r_0 .. r_{nv-1}, a^H a, a^H u
  cplx* partial;
  int scalars;
  // UPDATE: coefficients [i nb + c]; last: finish V_j and u with (1 / rho, s) per column and sum |u|^2
  const float2 *g, *r;
  const float4* fin;      // (1 / rho, s.x, s.y, -)
  int last;
};
template <int NV, bool UPDATE, int CW>
__global__ void __launch_bounds__(SW_THREADS, 2) sweep_kernel(SweepArgs p) {
  constexpr int TY = SW_THREADS / CW, IG = SwGroups<NV>::IG, NPG = SwGroups<NV>::NPG, RPG = TY / IG;
  constexpr int SLOTS = NPG + 2;
  static_assert(TY % IG == 0, "thread rows per group");
  extern __shared__ __align__(16) unsigned char sw_raw[];
  float2* ring = reinterpret_cast<float2*>(sw_raw);                                                    // [SW_STAGES][SLOTS][SW_THREADS]
  float4* share = reinterpret_cast<float4*>(ring + (size_t)SW_STAGES * SLOTS * SW_THREADS);             // [2][TY][CW]
  const int nv = p.nv, nb = p.nb;
  const int tid = threadIdx.x, x = tid % CW, y = tid / CW;
  const int gi = y / RPG, yr = y % RPG;
  const int c = blockIdx.x * CW + x;
  const int i0 = gi * NPG, ng = nv - i0;
  const long long r0 = blockIdx.y * p.rows_per_chunk;
  const long long r1 = min(p.D, r0 + p.rows_per_chunk);
  const long long nsteps = (r1 - r0 + RPG - 1) / RPG;   // the same for every thread (barriers inside)
  const float2* Vg = p.V + (long long)i0 * p.vstride;
  auto issue = [&](long long t) {
    float2* st = ring + (size_t)(t % SW_STAGES) * SLOTS * SW_THREADS + tid;
    const long long nu = r0 + t * RPG + yr;
    const bool ok = c < nb && nu < r1;
    const long long off = ok ? nu * nb + c : 0;
    // predicated-off copies zero-fill and read nothing; they are given a valid base address
#pragma unroll
    for (int li = 0; li < NPG; ++li) {
      const bool on = ok && li < ng;
      cp_async8(st + li * SW_THREADS, on ? Vg + li * p.vstride + off : p.a, on);
    }
    cp_async8(st + NPG * SW_THREADS, p.a + off, ok);
    cp_async8(st + (NPG + 1) * SW_THREADS, p.u + off, ok);
  };
  // UPDATE: coefficients of the thread's vectors; DOTS: accumulators
  float2 cg[NPG], cr[NPG];
#pragma unroll
  for (int li = 0; li < NPG; ++li) {
    const bool on = UPDATE && c < nb && li < ng;
    cg[li] = on ? p.g[(long long)(i0 + li) * nb + c] : make_float2(0.f, 0.f);
    cr[li] = on ? p.r[(long long)(i0 + li) * nb + c] : make_float2(0.f, 0.f);
  }
  float4 fin = make_float4(0.f, 0.f, 0.f, 0.f);
  if (UPDATE && p.last && c < nb) fin = p.fin[c];
  float aa = 0.f, aux = 0.f, auy = 0.f;   // DOTS: a^H a, a^H u; UPDATE: aa = |u|^2
#pragma unroll
  for (int t = 0; t < SW_STAGES - 1; ++t) {
    if (t < nsteps) issue(t);
    cp_async_commit();
  }
  for (long long t = 0; t < nsteps; ++t) {
    if (t + SW_STAGES - 1 < nsteps) issue(t + SW_STAGES - 1);
    cp_async_commit();
    cp_async_wait<SW_STAGES - 1>();   // this thread's copies of step t have landed
    const float2* st = ring + (size_t)(t % SW_STAGES) * SLOTS * SW_THREADS + tid;
    float2 a = st[NPG * SW_THREADS], u = st[(NPG + 1) * SW_THREADS];
    if constexpr (!UPDATE) {
#pragma unroll
      for (int li = 0; li < NPG; ++li) {
        const float2 v = st[li * SW_THREADS];
        cg[li].x = fma(v.x, a.x, fma(v.y, a.y, cg[li].x));
        cg[li].y = fma(v.x, a.y, fma(-v.y, a.x, cg[li].y));
        cr[li].x = fma(v.x, u.x, fma(v.y, u.y, cr[li].x));
        cr[li].y = fma(v.x, u.y, fma(-v.y, u.x, cr[li].y));
      }
      aa = fma(a.x, a.x, fma(a.y, a.y, aa));
      aux = fma(a.x, u.x, fma(a.y, u.y, aux));
      auy = fma(a.x, u.y, fma(-a.y, u.x, auy));
    } else {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);   // V g, V r
#pragma unroll
      for (int li = 0; li < NPG; ++li) {
        const float2 v = st[li * SW_THREADS];
        s.x = fma(v.x, cg[li].x, fma(-v.y, cg[li].y, s.x));
        s.y = fma(v.x, cg[li].y, fma(v.y, cg[li].x, s.y));
        s.z = fma(v.x, cr[li].x, fma(-v.y, cr[li].y, s.z));
        s.w = fma(v.x, cr[li].y, fma(v.y, cr[li].x, s.w));
      }
      if constexpr (IG > 1) {
        float4* sh = share + (size_t)(t & 1) * SW_THREADS;
        sh[tid] = s;
        __syncthreads();
        s = sh[yr * CW + x];
#pragma unroll
        for (int gg = 1; gg < IG; ++gg) {
          const float4 o = sh[(gg * RPG + yr) * CW + x];
          s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
        }
      }
      const long long nu = r0 + t * RPG + yr;
      if (gi == 0 && c < nb && nu < r1) {
        a.x -= s.x; a.y -= s.y;
        u.x -= s.z; u.y -= s.w;
        if (p.last) {
          a.x *= fin.x; a.y *= fin.x;
          u.x = fma(-a.x, fin.y, fma(a.y, fin.z, u.x));
          u.y = fma(-a.x, fin.z, fma(-a.y, fin.y, u.y));
          aa = fma(u.x, u.x, fma(u.y, u.y, aa));
        }
        p.a[nu * nb + c] = a;
        p.u[nu * nb + c] = u;
      }
    }
  }
  cp_async_wait<0>();
  // sums over the thread rows, in FP64. All of them go to shared memory at once (the load ring is free now) and the
  // whole block adds them, one output per thread and step: 2 RPG FP64 additions deep. (One basis vector at a time left
  // the additions to one warp: 5 us of a 20 us sweep at 264 columns of 4,785 rows.)
  __syncthreads();
  if constexpr (UPDATE) {
    if (!p.last) return;   // uniform
    double* part = reinterpret_cast<double*>(sw_raw);   // [TY][CW]
    if (gi == 0) part[tid] = (double)aa;                // the first RPG thread rows
    __syncthreads();
    double t2 = 0.0;                                    // four threads per column
    if (tid < 4 * CW)
      for (int k = tid / CW; k < RPG; k += 4) t2 += part[k * CW + tid % CW];
    __syncthreads();
    if (tid < 4 * CW) part[tid] = t2;
    __syncthreads();
    if (tid < CW && c < nb)
      p.partial[(long long)blockIdx.y * nb + c] =
          make_cuDoubleComplex((part[tid] + part[CW + tid]) + (part[2 * CW + tid] + part[3 * CW + tid]), 0.0);
  } else {
    float2* part = reinterpret_cast<float2*>(sw_raw);   // [2 NPG][TY][CW], then a^H a and a^H u [2][TY][CW]
    static_assert((2 * NPG + 2) <= SW_STAGES * SLOTS, "sums fit in the load ring");
#pragma unroll
    for (int li = 0; li < NPG; ++li) {
      part[li * SW_THREADS + tid] = cg[li];
      part[(NPG + li) * SW_THREADS + tid] = cr[li];
    }
    part[2 * NPG * SW_THREADS + tid] = make_float2(aa, 0.f);
    part[(2 * NPG + 1) * SW_THREADS + tid] = make_float2(aux, auy);
    __syncthreads();
    const int nq = 2 * nv + (p.scalars ? 2 : 0);
    for (int q = tid; q < (2 * NV + 2) * CW; q += SW_THREADS) {
      // output k = q / CW of column q % CW: g_i, r_i (i < NV) or a scalar (k = 2 NV, 2 NV + 1: summed by group 0)
      const int k = q / CW, xx = q % CW, cc = blockIdx.x * CW + xx;
      const bool sc = k >= 2 * NV;
      const int i = sc ? 0 : k % NV, kind = sc ? 0 : k / NV;
      if (cc >= nb || (sc ? !p.scalars : i >= nv)) continue;
      const int slot = sc ? k - 2 * NV + 2 * NPG : kind * NPG + i % NPG;
      const int row0 = sc ? 0 : (i / NPG) * RPG;
      cplx sum = make_cuDoubleComplex(0.0, 0.0);
      for (int m = 0; m < RPG; ++m) {
        const float2 v = part[slot * SW_THREADS + (row0 + m) * CW + xx];
        sum.x += (double)v.x;
        sum.y += (double)v.y;
      }
      const int out = sc ? 2 * nv + (k - 2 * NV) : kind * nv + i;
      p.partial[((long long)blockIdx.y * nq + out) * nb + cc] = sum;
    }
  }
}

// sums[q nb + c] = sum_chunk partial[chunk][q][c], also in FP32 (a block takes one q and 32 columns)
__global__ void __launch_bounds__(256) reduce_dots_kernel(const cplx* __restrict__ partial, int nchunk, int nq, int nb,
                                                          cplx* __restrict__ sums, float2* __restrict__ sums_f) {
  __shared__ cplx red[8][32];
  const int x = threadIdx.x, y = threadIdx.y, c = blockIdx.x * 32 + x, q = blockIdx.y;
  cplx s = make_cuDoubleComplex(0.0, 0.0);
  if (c < nb) {
#pragma unroll 4
    for (int k = y; k < nchunk; k += 8) {
      const cplx p = partial[((long long)k * nq + q) * nb + c];
      s.x += p.x; s.y += p.y;
    }
  }
  red[y][x] = s;
  __syncthreads();
  if (y == 0 && c < nb) {
    for (int k = 1; k < 8; ++k) { s.x += red[k][x].x; s.y += red[k][x].y; }
    sums[(long long)q * nb + c] = s;
    sums_f[(long long)q * nb + c] = make_float2((float)s.x, (float)s.y);
  }
}
// The coefficients of a column from its sums (g_i at g[i nb + c], r_i, a^H a and a^H u at sc): Hessenberg column Hc
// (entry (i, c) at i nb + c) and fin = (1 / rho, s), zero where a lies in the span of the basis. Eight lanes per column.
__global__ void __launch_bounds__(128) delayed_coef_kernel(const cplx* __restrict__ g, const cplx* __restrict__ r, int nv,
                                                           const cplx* __restrict__ sc, int nb, cplx* __restrict__ Hc,
                                                           float4* __restrict__ fin) {
  const int c = blockIdx.x * 16 + (threadIdx.x >> 3), q = threadIdx.x & 7;
  const bool on = c < nb;
  double gg = 0.0, gx = 0.0, gy = 0.0;
  if (on)
    for (int i = q; i < nv; i += 8) {
      const cplx a = g[(long long)i * nb + c], b = r[(long long)i * nb + c];
      gg = fma(a.x, a.x, fma(a.y, a.y, gg));
      gx = fma(a.x, b.x, fma(a.y, b.y, gx));   // conj(g) r
      gy = fma(a.x, b.y, fma(-a.y, b.x, gy));
      Hc[(long long)i * nb + c] = b;
    }
#pragma unroll
  for (int w = 4; w > 0; w >>= 1) {
    gg += __shfl_down_sync(0xffffffffu, gg, w, 8);
    gx += __shfl_down_sync(0xffffffffu, gx, w, 8);
    gy += __shfl_down_sync(0xffffffffu, gy, w, 8);
  }
  if (!on || q != 0) return;
  const double rho2 = sc[c].x - gg;
  // a zero column stays zero (rho^2 and a^H a are differences and sums of FP32 results: a difference far below them is noise)
  const double inv = rho2 > 0.5 * sc[c].x && isfinite(rho2) ? rsqrt(rho2) : 0.0;
  const cplx s = make_cuDoubleComplex((sc[nb + c].x - gx) * inv, (sc[nb + c].y - gy) * inv);
  Hc[(long long)nv * nb + c] = s;
  fin[c] = make_float4((float)inv, (float)s.x, (float)s.y, 0.f);
}

// column width of the sweep blocks for a batch of nb columns
int sweep_cw(int nb) { return nb >= 32 ? 32 : nb > 8 ? 16 : nb > 4 ? 8 : 4; }
// rows per chunk of the pipelined sweeps: at most one wave of two resident blocks per SM (a block count
// just above the resident slots would leave a short second wave that takes as long as the first)
long long sweep_rows(long long D, int nb) {
  const int cw = sweep_cw(nb);
  const long long gx = (nb + cw - 1) / cw;
  const long long nchunk = std::max<long long>(1, (152LL * 2) / gx);
  return std::max<long long>(64, (D + nchunk - 1) / nchunk);
}

template <int NV, bool UPDATE, int CW>
void launch_sweep_cw(SweepArgs p, cudaStream_t s) {
  static bool attr[64] = {};   // dynamic shared memory above 48 KB: set once per device
  int dev = 0;
  GFCC_CUDA(cudaGetDevice(&dev));
  GFCC_CHECK(dev >= 0 && dev < 64, GFCC_ERR_ARG, "device ordinal above 63");
  constexpr size_t bytes = sweep_smem_bytes<NV, CW>();
  if (!attr[dev]) {
    GFCC_CUDA(cudaFuncSetAttribute(sweep_kernel<NV, UPDATE, CW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    attr[dev] = true;
  }
  p.rows_per_chunk = sweep_rows(p.D, p.nb);
  const dim3 grid((unsigned)((p.nb + CW - 1) / CW), (unsigned)((p.D + p.rows_per_chunk - 1) / p.rows_per_chunk));
  sweep_kernel<NV, UPDATE, CW><<<grid, SW_THREADS, bytes, s>>>(p);
}
template <bool UPDATE>
void launch_sweep(const SweepArgs& p, cudaStream_t s) {
  with_nv(p.nv, [&](auto NVc) {
    constexpr int NV = decltype(NVc)::value;
    switch (sweep_cw(p.nb)) {
      case 32: launch_sweep_cw<NV, UPDATE, 32>(p, s); break;
      case 16: launch_sweep_cw<NV, UPDATE, 16>(p, s); break;
      case 8: launch_sweep_cw<NV, UPDATE, 8>(p, s); break;
      default: launch_sweep_cw<NV, UPDATE, 4>(p, s); break;
    }
  });
  GFCC_LAUNCH_CHECK();
}

// rows per chunk of the dot products of the FP64 basis and of norms: two whole waves of blocks (two resident per SM), short vectors in
// chunks of at least 16 rows (a third, partial wave cost 11 % at 560 columns of 3,836 rows; one chunk of 64 rows for
// 1024 columns of 52 left most SMs without a block)
long long cgs_rows(long long D, int nb) {
  const long long gx = (nb + MD_TX - 1) / MD_TX, slots = 152LL * 2;
  const long long nchunk = std::max<long long>(1, 2 * slots / gx);
  return std::max<long long>(16, (D + nchunk - 1) / nchunk);
}

// h[c*hld + hoff + i] = sum_chunk partial[chunk][i][c], also set in or added to the Hessenberg column Hc (entry
// (hoff + i, c) at (hoff + i) nb + c). A block takes one i and 32 columns, its eight warps sharing the chunks
// (one thread per sum walked them one after the other: 10 us for a few hundred chunks, now 2).
__global__ void __launch_bounds__(256) reduce_partial_kernel(const cplx* __restrict__ partial, int nchunk, int nv, int nb,
                                                             cplx* __restrict__ h, int hld, int hoff,
                                                             cplx* __restrict__ Hc, int accumulate) {
  __shared__ cplx red[8][32];
  const int x = threadIdx.x, y = threadIdx.y, c = blockIdx.x * 32 + x, i = blockIdx.y;
  cplx s = make_cuDoubleComplex(0.0, 0.0);
  if (c < nb) {
#pragma unroll 4
    for (int k = y; k < nchunk; k += 8) {
      const cplx p = partial[((long long)k * nv + i) * nb + c];
      s.x += p.x; s.y += p.y;
    }
  }
  red[y][x] = s;
  __syncthreads();
  if (y == 0 && c < nb) {
    for (int k = 1; k < 8; ++k) { s.x += red[k][x].x; s.y += red[k][x].y; }
    h[(long long)c * hld + hoff + i] = s;
    if (Hc) {
      cplx* d = Hc + (long long)(hoff + i) * nb + c;
      if (accumulate) { s.x += d->x; s.y += d->y; }
      *d = s;
    }
  }
}

// W[nu][c] -= sum_{i<nv} V_i[nu][c] h[c*hld + i] (blocks as in el_grid)
template <typename VT>
__global__ void __launch_bounds__(256) update_kernel(const VT* __restrict__ V, long long vstride, int nv,
                                                     VT* __restrict__ W, long long D, int nb,
                                                     const cplx* __restrict__ h, int hld) {
  using R = typename RealOf<VT>::type;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nb) return;
  const cplx* hc = h + (long long)c * hld;
  for (long long nu = blockIdx.y * (long long)blockDim.y + threadIdx.y; nu < D; nu += (long long)gridDim.y * blockDim.y) {
    const long long t = nu * nb + c;
    // four independent partial sums keep several loads in flight
    R sx[4] = {R(0), R(0), R(0), R(0)}, sy[4] = {R(0), R(0), R(0), R(0)};
    int i = 0;
    for (; i + 4 <= nv; i += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const VT vv = V[(long long)(i + u) * vstride + t];
        const R hx = (R)hc[i + u].x, hy = (R)hc[i + u].y;
        sx[u] = fma(vv.x, hx, fma(-vv.y, hy, sx[u]));
        sy[u] = fma(vv.x, hy, fma(vv.y, hx, sy[u]));
      }
    }
    for (; i < nv; ++i) {
      const VT vv = V[(long long)i * vstride + t];
      const R hx = (R)hc[i].x, hy = (R)hc[i].y;
      sx[0] = fma(vv.x, hx, fma(-vv.y, hy, sx[0]));
      sy[0] = fma(vv.x, hy, fma(vv.y, hx, sy[0]));
    }
    W[t].x -= (sx[0] + sx[1]) + (sx[2] + sx[3]);
    W[t].y -= (sy[0] + sy[1]) + (sy[2] + sy[3]);
  }
}

// out[c] = sqrt(sum_chunk partial[chunk][c].x) (32 columns a block, eight warps sharing the chunks)
__global__ void __launch_bounds__(256) reduce_norm_kernel(const cplx* __restrict__ partial, int nchunk, int nb,
                                                          double* __restrict__ out) {
  __shared__ double red[8][32];
  const int x = threadIdx.x, y = threadIdx.y, c = blockIdx.x * 32 + x;
  double s = 0.0;
  if (c < nb)
    for (int k = y; k < nchunk; k += 8) s += partial[(long long)k * nb + c].x;
  red[y][x] = s;
  __syncthreads();
  if (y == 0 && c < nb) {
    for (int k = 1; k < 8; ++k) s += red[k][x];
    out[c] = sqrt(fmax(s, 0.0));
  }
}

// Elementwise kernels over a batch-minor block: blocks of CW columns (CW = sweep_cw(nb)) and EL_T / CW thread
// rows, so that a thread keeps its column and what belongs to it (no division per element).
constexpr int EL_T = 256;
struct ElGrid {
  dim3 grid, block;
};
ElGrid el_grid(long long D, int nb) {
  const int cw = nb >= 32 ? 32 : nb > 8 ? 16 : nb > 4 ? 8 : 4;
  const long long gx = (nb + cw - 1) / cw, rows = EL_T / cw;
  // the same number of row steps for every block (up to the last)
  const long long most = std::max<long long>(1, 152LL * 24 / gx);
  const long long steps = std::max<long long>(1, (D + rows * most - 1) / (rows * most));
  const long long gy = std::max<long long>(1, (D + rows * steps - 1) / (rows * steps));
  return {dim3((unsigned)gx, (unsigned)std::min<long long>(gy, 65535)), dim3((unsigned)cw, (unsigned)(EL_T / cw))};
}

// V[nu][c] = W[nu][c] / nrm[c] (0 for broken-down columns), Z[nu][c] = V[nu][c] / (shift_c + mdiag[nu]) (FP64 basis)
__global__ void __launch_bounds__(EL_T) scale_precond_kernel(const cplx* __restrict__ W, const double* __restrict__ nrm,
                                                             cplx* __restrict__ V, cplx* __restrict__ Z,
                                                             const double* __restrict__ md,
                                                             const cplx* __restrict__ shift, long long D, int nb) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nb) return;
  const double n = nrm[c], s = (n > 0.0 && isfinite(n)) ? 1.0 / n : 0.0;
  const cplx sh = shift[c];
  for (long long nu = blockIdx.y * (long long)blockDim.y + threadIdx.y; nu < D; nu += (long long)gridDim.y * blockDim.y) {
    const long long t = nu * nb + c;
    cplx v = W[t];
    v.x *= s;
    v.y *= s;
    V[t] = v;
    const double dr = sh.x + md[nu], di = sh.y, inv = 1.0 / (dr * dr + di * di);
    Z[t] = make_cuDoubleComplex((v.x * dr + v.y * di) * inv, (v.y * dr - v.x * di) * inv);
  }
}
// inv[c] = 1 / nrm[c] in FP32 (0 for broken-down columns)
__global__ void inv_norm_kernel(const double* __restrict__ nrm, int nb, float* __restrict__ inv) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nb) return;
  const double n = nrm[c];
  inv[c] = (n > 0.0 && isfinite(n)) ? (float)(1.0 / n) : 0.f;
}

// R = B - Y and partial[chunk][c].x = sum_{nu in chunk} |R[nu][c]|^2 (chunk = blockIdx.y)
__global__ void __launch_bounds__(EL_T) residual_kernel(const cplx* __restrict__ B, const cplx* __restrict__ Y,
                                                        cplx* __restrict__ R, long long D, int nb,
                                                        cplx* __restrict__ partial) {
  __shared__ double red[EL_T];
  const int c = blockIdx.x * blockDim.x + threadIdx.x, tid = threadIdx.y * blockDim.x + threadIdx.x;
  double s = 0.0;
  if (c < nb)
    for (long long nu = blockIdx.y * (long long)blockDim.y + threadIdx.y; nu < D; nu += (long long)gridDim.y * blockDim.y) {
      const long long t = nu * nb + c;
      const cplx b = B[t], y = Y[t];
      const cplx r = make_cuDoubleComplex(b.x - y.x, b.y - y.y);
      R[t] = r;
      s = fma(r.x, r.x, fma(r.y, r.y, s));
    }
  red[tid] = s;
  __syncthreads();
  if (threadIdx.y == 0 && c < nb) {
    for (int k = 1; k < blockDim.y; ++k) s += red[k * blockDim.x + threadIdx.x];
    partial[(long long)blockIdx.y * nb + c] = make_cuDoubleComplex(s, 0.0);
  }
}

// End of Arnoldi step j: the norm of the new vector from its chunk sums (or, with nchunk = 0, already in nrm), its
// reciprocal for the next step, the j earlier Givens rotations on the new Hessenberg column, the new rotation, the
// residual estimate |g_{j+1}| / bnorm and the count of columns still above their threshold.
// H[(jj (k+1) + i) nb + c], cs, sn, g [i nb + c]. Rotations have a real cosine: t = c a + s b, u = c b - conj(s) a.
// Four lanes per column, one for each real component of (t, u): an FP64 instruction holds its scheduler for 75
// clocks whatever the lanes in use, and a thread per column issued 16 of them per rotation (21 us at 15
// rotations; four lanes issue 3).
constexpr int GV_T = 512;   // sixteen warps share the chunk sums of 32 columns; the first four rotate
__global__ void __launch_bounds__(GV_T) arnoldi_finish_kernel(const cplx* __restrict__ partial, int nchunk,
                                                              double* __restrict__ nrm, float* __restrict__ invf,
                                                              cplx* __restrict__ H, double* __restrict__ cs,
                                                              cplx* __restrict__ sn, cplx* __restrict__ g,
                                                              const double* __restrict__ bnorm, int* __restrict__ kc,
                                                              int* __restrict__ live, int nb, int k, int j,
                                                              const double* __restrict__ thr, int* __restrict__ n_live,
                                                              const float4* __restrict__ fin) {
  __shared__ double red[GV_T / 32][32];
  const int c0 = blockIdx.x * 32;
  if (nchunk > 0) {
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    double s = 0.0;
    if (c0 + x < nb) {
#pragma unroll 8
      for (int q = y; q < nchunk; q += GV_T / 32) s += partial[(long long)q * nb + c0 + x].x;
    }
    red[y][x] = s;
    __syncthreads();
    if (y == 0) {
      for (int q = 1; q < GV_T / 32; ++q) s += red[q][x];
      s = sqrt(fmax(s, 0.0));
      red[0][x] = s;
      if (c0 + x < nb) nrm[c0 + x] = s;
    }
    __syncthreads();
  }
  if (threadIdx.x >= 128) return;
  const int x = threadIdx.x >> 2, q = threadIdx.x & 3, c = c0 + x;
  // fin (FP32 basis): a column whose vector j was found in the span of the basis keeps its j vectors and ends its cycle
  const bool in = c < nb, was = in && live[c], broken = was && fin && fin[c].x == 0.f, on = was && !broken;
  __syncwarp();
  if (broken && q == 0) live[c] = 0;
  const double hn = in ? (nchunk > 0 ? red[0][x] : nrm[c]) : 0.0;
  if (in && q == 0) invf[c] = (hn > 0.0 && isfinite(hn)) ? (float)(1.0 / hn) : 0.f;
  if (!__any_sync(0xffffffffu, on)) return;
  cplx* col = H + (long long)j * (k + 1) * nb + c;
  // lanes: 0 t.re, 1 t.im, 2 u.re, 3 u.im of  ca a + cb b  with complex coefficients split into components
  const bool isu = q >= 2, im = q & 1;
  cplx a = on ? col[0] : make_cuDoubleComplex(0.0, 0.0);
  __syncwarp();           // every lane has read its column's first entry before lanes 0 and 1 replace it below; an entry
                          // further down is replaced only after a shuffle that follows every lane's read of it
  constexpr int PF = 4;   // rotations loaded ahead of the serial chain
  for (int i0 = 0; i0 < j; i0 += PF) {
    cplx b[PF], s[PF];
    double cc[PF];
#pragma unroll
    for (int r = 0; r < PF; ++r) {
      const bool ok = on && i0 + r < j;
      b[r] = ok ? col[(long long)(i0 + r + 1) * nb] : make_cuDoubleComplex(0.0, 0.0);
      s[r] = ok ? sn[(long long)(i0 + r) * nb + c] : make_cuDoubleComplex(0.0, 0.0);
      cc[r] = ok ? cs[(long long)(i0 + r) * nb + c] : 1.0;
    }
#pragma unroll
    for (int r = 0; r < PF; ++r) {
      if (i0 + r >= j) break;   // uniform
      // t = cc a + s b: (cc a.re + s.re b.re - s.im b.im, cc a.im + s.re b.im + s.im b.re)
      // u = cc b - conj(s) a: (cc b.re - s.re a.re - s.im a.im, cc b.im - s.re a.im + s.im a.re)
      const cplx p = isu ? b[r] : a, o = isu ? a : b[r];   // multiplied by cc, by s
      const double sr = isu ? -s[r].x : s[r].x;
      const double si = im ? s[r].y : -s[r].y;
      const double v = fma(cc[r], im ? p.y : p.x, fma(sr, im ? o.y : o.x, si * (im ? o.x : o.y)));
      if (on && !isu) reinterpret_cast<double*>(col + (long long)(i0 + r) * nb)[im] = v;
      a.x = __shfl_sync(0xffffffffu, v, 2, 4);
      a.y = __shfl_sync(0xffffffffu, v, 3, 4);
    }
  }
  if (!on || q != 0) return;
  // new rotation of (a, hn), hn real: with den^2 = |a|^2 + hn^2, cosine |a| / den, sine (a / |a|) hn / den, new
  // diagonal (a / |a|) den, all from one reciprocal root of |a|^2 den^2
  const double a2 = a.x * a.x + a.y * a.y, d2 = a2 + hn * hn, ad = a2 * d2;
  double cj, den;
  cplx sj, tj;
  if (ad > 1e-280 && ad < 1e280) {
    const double r = rsqrt(ad);   // 1 / (|a| den)
    cj = a2 * r;
    sj = make_cuDoubleComplex(a.x * hn * r, a.y * hn * r);
    tj = make_cuDoubleComplex(a.x * (d2 * r), a.y * (d2 * r));
    den = 1.0;   // not zero
  } else {
    const double aa = hypot(a.x, a.y);
    den = hypot(aa, hn);
    const cplx ph = aa > 0.0 ? make_cuDoubleComplex(a.x / aa, a.y / aa) : make_cuDoubleComplex(1.0, 0.0);
    cj = den > 0.0 ? aa / den : 1.0;
    const double hd = den > 0.0 ? hn / den : 0.0;
    sj = make_cuDoubleComplex(ph.x * hd, ph.y * hd);
    tj = make_cuDoubleComplex(ph.x * den, ph.y * den);
  }
  cs[(long long)j * nb + c] = cj;
  sn[(long long)j * nb + c] = sj;
  col[(long long)j * nb] = tj;
  col[(long long)(j + 1) * nb] = make_cuDoubleComplex(0.0, 0.0);
  const cplx gj = g[(long long)j * nb + c];
  const cplx gn = make_cuDoubleComplex(-(sj.x * gj.x + sj.y * gj.y), -(sj.x * gj.y - sj.y * gj.x));
  g[(long long)(j + 1) * nb + c] = gn;
  g[(long long)j * nb + c] = make_cuDoubleComplex(cj * gj.x, cj * gj.y);
  kc[c] = j + 1;
  // estimate |g_{j+1}| / bnorm against the threshold, squared
  const double est2 = gn.x * gn.x + gn.y * gn.y, lim = thr[c] * bnorm[c];
  if (!(est2 > lim * lim) || den == 0.0 || !isfinite(est2)) {
    live[c] = 0;   // converged (or broken down) within this cycle: stop extending its basis use
  } else {
    atomicAdd(n_live, 1);
  }
}

// y = H[:kc,:kc]^{-1} g (upper triangular), stored in g; also in the basis precision in y. One warp per column,
// column-oriented: row i of every remaining entry is updated by the lanes at once (at most 256 rows).
template <typename VT>
__global__ void __launch_bounds__(128) backsolve_kernel(const cplx* __restrict__ H, cplx* __restrict__ g,
                                                        const int* __restrict__ kc, int nb, int k, VT* __restrict__ y) {
  const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= nb) return;
  const int n = kc[c];
  for (int jj = n - 1; jj >= 0; --jj) {
    const cplx d = H[((long long)jj * (k + 1) + jj) * nb + c];
    const cplx v = g[(long long)jj * nb + c];
    const cplx yj = (d.x == 0.0 && d.y == 0.0) ? make_cuDoubleComplex(0.0, 0.0) : cuCdiv(v, d);
    __syncwarp();   // every lane has read g_jj before it is replaced
    if (lane == 0) g[(long long)jj * nb + c] = yj;
    for (int i = lane; i < jj; i += 32)
      g[(long long)i * nb + c] = cuCsub(g[(long long)i * nb + c], cuCmul(H[((long long)jj * (k + 1) + i) * nb + c], yj));
    __syncwarp();
  }
  for (int i = lane; i < k; i += 32) {
    const cplx v = i < n ? g[(long long)i * nb + c] : make_cuDoubleComplex(0.0, 0.0);
    VT r;
    r.x = v.x;
    r.y = v.y;
    y[(long long)i * nb + c] = r;
  }
}

// X[nu][c] += P_c[nu] * sum_{i < nv} V_i[nu][c] y_i[c]: the correction is formed in the basis precision, only its
// addition to x is FP64 (y [i nb + c], zero beyond a column's own steps). A vector whose coefficient is zero is not read:
// what a finished column's later vectors hold, made because its batch went on, stays out of the sum whatever it is.
template <typename VT>
__global__ void __launch_bounds__(EL_T) correct_kernel(const VT* __restrict__ V, long long vstride, int nv,
                                                       const VT* __restrict__ y, cplx* __restrict__ X,
                                                       const double* __restrict__ md, const RowF* __restrict__ mdf,
                                                       const cplx* __restrict__ shift,
                                                       const ShiftF* __restrict__ shiftf, long long D, int nb) {
  using R = typename RealOf<VT>::type;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nb) return;
  cplx sh = make_cuDoubleComplex(0.0, 0.0);
  ShiftF shf = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (sizeof(R) == 4) shf = shiftf[c];
  else sh = shift[c];
  auto vector = [&](int i, long long t, const VT& yy) {
    VT vv;
    vv.x = vv.y = R(0);
    if (yy.x != R(0) || yy.y != R(0)) vv = V[(long long)i * vstride + t];
    return vv;
  };
  for (long long nu = blockIdx.y * (long long)blockDim.y + threadIdx.y; nu < D; nu += (long long)gridDim.y * blockDim.y) {
    const long long t = nu * nb + c;
    R sr[4] = {R(0), R(0), R(0), R(0)}, si[4] = {R(0), R(0), R(0), R(0)};
    int i = 0;
    for (; i + 4 <= nv; i += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const VT yy = y[(long long)(i + u) * nb + c], vv = vector(i + u, t, yy);
        sr[u] = fma(vv.x, yy.x, fma(-vv.y, yy.y, sr[u]));
        si[u] = fma(vv.x, yy.y, fma(vv.y, yy.x, si[u]));
      }
    }
    for (; i < nv; ++i) {
      const VT yy = y[(long long)i * nb + c], vv = vector(i, t, yy);
      sr[0] = fma(vv.x, yy.x, fma(-vv.y, yy.y, sr[0]));
      si[0] = fma(vv.x, yy.y, fma(vv.y, yy.x, si[0]));
    }
    VT s;
    s.x = (sr[0] + sr[1]) + (sr[2] + sr[3]);
    s.y = (si[0] + si[1]) + (si[2] + si[3]);
    if constexpr (sizeof(R) == 4) {
      const float2 z = precond_f32(make_float2(s.x, s.y), mdf[nu], shf);
      s.x = z.x;
      s.y = z.y;
    } else {
      const double dr = sh.x + md[nu], di = sh.y, inv = 1.0 / (dr * dr + di * di);
      s = make_cuDoubleComplex((s.x * dr + s.y * di) * inv, (s.y * dr - s.x * di) * inv);
    }
    cplx x = X[t];
    x.x += (double)s.x;
    x.y += (double)s.y;
    X[t] = x;
  }
}

// dst[nu][k] = src[nu][cols[k]]  (column gather between batch-minor blocks)
__global__ void gather_cols_kernel(const cplx* __restrict__ src, int lds, const int* __restrict__ cols, int nk,
                                   cplx* __restrict__ dst, int ldd, long long D) {
  long long total = D * nk;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int k = (int)(t % nk);
    long long nu = t / nk;
    dst[nu * ldd + k] = src[nu * lds + cols[k]];
  }
}
// dst[nu][cols[k]] = src[nu][k]
__global__ void scatter_cols_kernel(const cplx* __restrict__ src, int lds, const int* __restrict__ cols, int nk,
                                    cplx* __restrict__ dst, int ldd, long long D) {
  long long total = D * nk;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int k = (int)(t % nk);
    long long nu = t / nk;
    dst[nu * ldd + cols[k]] = src[nu * lds + k];
  }
}

__global__ void nonfinite_cplx_kernel(const cplx* x, long long n, int* flag) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    if (!isfinite(x[t].x) || !isfinite(x[t].y)) *flag = 1;
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// column norms of a batch-minor block: out[c] = ||W_c||  (device array)
template <typename VT>
static void col_norms(const VT* W, long long D, int nb, double* out, DBuf<cplx>& partial, cudaStream_t s) {
  const long long rows = cgs_rows(D, nb);
  const int nchunk = (int)((D + rows - 1) / rows);
  partial.alloc((long long)nchunk * nb);
  dim3 grid((nb + MD_TX - 1) / MD_TX, nchunk);
  norm_partial_kernel<VT><<<grid, dim3(MD_TX, MD_TY), 0, s>>>(W, D, nb, rows, partial.p);
  GFCC_LAUNCH_CHECK();
  reduce_norm_kernel<<<(nb + 31) / 32, dim3(32, 8), 0, s>>>(partial.p, nchunk, nb, out);
  GFCC_LAUNCH_CHECK();
}

// h[c][i] = V_i^H W_c for i < nv, with chunked partial sums; set in or added to the Hessenberg column Hc
template <typename VT>
static void multidot(const VT* V, long long vstride, int nv, const VT* W, long long D, int nb, cplx* h, int hld,
                     cplx* Hc, bool accumulate, DBuf<cplx>& partial, cudaStream_t s) {
  for (int i0 = 0; i0 < nv; i0 += MD_MAXV) {
    int n = std::min(MD_MAXV, nv - i0);
    const long long rows = cgs_rows(D, nb);
    const int nchunk = (int)((D + rows - 1) / rows);
    partial.alloc((long long)nchunk * n * nb);
    dim3 grid((nb + MD_TX - 1) / MD_TX, nchunk);
    with_nv(n, [&](auto NVc) {
      multidot_kernel<VT, decltype(NVc)::value><<<grid, dim3(MD_TX, MD_TY), 0, s>>>(V + i0 * vstride, vstride, n, W, D,
                                                                                  nb, rows, partial.p);
    });
    GFCC_LAUNCH_CHECK();
    reduce_partial_kernel<<<dim3((nb + 31) / 32, n), dim3(32, 8), 0, s>>>(partial.p, nchunk, n, nb, h, hld, i0, Hc,
                                                                          accumulate ? 1 : 0);
    GFCC_LAUNCH_CHECK();
  }
}

// Restarted GMRES with iterative refinement; VT is the precision of the Krylov basis (FP64 for the
// plain FP64 path, FP32 when the inner sigma runs on the tensor cores: the residual of every cycle is
// recomputed with the FP64-accurate sigma and the solution is accumulated in FP64, so the basis
// precision only bounds the progress of one cycle, not the final accuracy).
template <typename VT>
static void gmres_impl(gfcc_ctx* c, const cplx* Bin, cplx* Xout, cplx* Rout, const cplx* shifts_dev, int nb0,
                       SolveStatus& st, bool transpose, const cplx* X0, bool polish) {
  cudaStream_t s = c->stream;
  const long long D = c->D;
  const int k = std::max(1, std::min(c->opts.restart, 256));
  const double tol = c->opts.tol;
  const int inner_prec = c->opts.precision;
  int resid_prec = c->opts.residual_precision;
  if (resid_prec < 0) resid_prec = inner_prec == GFCC_PREC_FP64 ? GFCC_PREC_FP64 : GFCC_PREC_FP64_TC;
  // a cycle with a low-precision inner operator cannot gain more than about its rounding level: stop
  // it once the inner estimate has dropped by this factor
  const double inner_rtol = (inner_prec == GFCC_PREC_FP64 || inner_prec == GFCC_PREC_FP64_TC) ? 0.0 : 1e-4;
  st.relres.assign(nb0, 0.0);
  st.iters.assign(nb0, 0);
  st.converged.assign(nb0, 0);
  if (nb0 == 0) return;

  std::vector<cplx> hshift(nb0);
  GFCC_CUDA(cudaMemcpyAsync(hshift.data(), shifts_dev, sizeof(cplx) * nb0, cudaMemcpyDeviceToHost, s));

  constexpr bool F32 = sizeof(VT) == sizeof(cuFloatComplex);
  DBuf<cplx> Bw, Xw, Rw, Yw, Ztmp, H, sn, g, partial, shw, hb;
  DBuf<VT> V, Zw, Ww, yv;
  DBuf<double> nrm, bnorm, thr, cs;
  DBuf<cplx> sums, gr;       // FP32 basis: the delayed pass's sums (and g, r of bases longer than one sweep)
  DBuf<float2> sums_f;
  DBuf<float4> fin;
  DBuf<float> invf;
  DBuf<int> kc, live, nlive, cols, flag;
  DBuf<float4> shf;
  if (F32) {
    ensure_row_split(c);
    shf.alloc(nb0);
    sums.alloc((long long)nb0 * (2 * k + 2));
    sums_f.alloc((long long)nb0 * (2 * k + 2));
    fin.alloc(nb0);
    if (k > MD_MAXV) gr.alloc((long long)nb0 * 2 * k);
  }
  if (!c->pin) GFCC_CUDA(cudaMallocHost(reinterpret_cast<void**>(&c->pin), sizeof(int)));
  if (!c->pin_event) GFCC_CUDA(cudaEventCreateWithFlags(&c->pin_event, cudaEventDisableTiming));
  Bw.alloc(D * nb0); Xw.alloc(D * nb0); Rw.alloc(D * nb0); Yw.alloc(D * nb0); Ztmp.alloc(D * nb0);
  if (!F32) Zw.alloc(D * nb0);   // the FP32 path forms z = P v where it is used
  Ww.alloc(D * nb0);
  V.alloc((long long)(k + 1) * D * nb0);
  V.zero(s);
  H.alloc((long long)nb0 * (k + 1) * k);
  cs.alloc((long long)nb0 * k); sn.alloc((long long)nb0 * k); g.alloc((long long)nb0 * (k + 1));
  hb.alloc((long long)nb0 * (k + 1));
  yv.alloc((long long)nb0 * k);
  invf.alloc(nb0);
  nrm.alloc(nb0); bnorm.alloc(nb0); thr.alloc(nb0); kc.alloc(nb0); live.alloc(nb0); nlive.alloc(k); cols.alloc(nb0);
  shw.alloc(nb0);
  flag.alloc(1);
  {  // chunk partial sums of the Gram-Schmidt sweeps and norms, at their largest (no regrowth per step)
    long long md = 0, el = 0;   // the chunk counts depend on the batch width
    for (int b = 1; b <= nb0; ++b) {
      md = std::max(md, (D + cgs_rows(D, b) - 1) / cgs_rows(D, b) * b);
      md = std::max(md, (D + sweep_rows(D, b) - 1) / sweep_rows(D, b) * b);
      el = std::max(el, (long long)el_grid(D, b).grid.y * b);   // one sum per chunk
    }
    const int nq = std::max(std::min(k + 1, MD_MAXV), 2 * std::min(k, MD_MAXV) + 2);   // sums per chunk
    partial.alloc(std::max(md * nq, el));
  }
  GFCC_CUDA(cudaMemcpyAsync(Bw.p, Bin, sizeof(cplx) * D * nb0, cudaMemcpyDeviceToDevice, s));
  GFCC_CUDA(cudaMemcpyAsync(shw.p, shifts_dev, sizeof(cplx) * nb0, cudaMemcpyDeviceToDevice, s));
  if (X0) GFCC_CUDA(cudaMemcpyAsync(Xw.p, X0, sizeof(cplx) * D * nb0, cudaMemcpyDeviceToDevice, s));
  else Xw.zero(s);
  {  // non-finite right-hand sides or shifts
    flag.zero(s);
    nonfinite_cplx_kernel<<<grid_for(D * nb0), 256, 0, s>>>(Bw.p, D * nb0, flag.p);
    GFCC_LAUNCH_CHECK();
    nonfinite_cplx_kernel<<<1, 256, 0, s>>>(shw.p, nb0, flag.p);
    GFCC_LAUNCH_CHECK();
    int hf = 0;
    GFCC_CUDA(cudaMemcpyAsync(&hf, flag.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    GFCC_CUDA(cudaStreamSynchronize(s));
    GFCC_CHECK(hf == 0, GFCC_ERR_NONFINITE, "solve: non-finite right-hand side or frequency");
  }
  col_norms<cplx>(Bw.p, D, nb0, bnorm.p, partial, s);
  std::vector<double> hbn(nb0);
  GFCC_CUDA(cudaMemcpyAsync(hbn.data(), bnorm.p, sizeof(double) * nb0, cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));

  std::vector<int> map(nb0);   // working column -> original column
  for (int i = 0; i < nb0; ++i) map[i] = i;
  int nb = nb0;
  std::vector<double> hres(nb0);
  std::vector<char> polished(nb0, 0);
  const double target = polish ? 0.1 : 0.5;   // of the tolerance, for the estimate that ends a cycle
  const int max_cycles = std::max(1, c->opts.max_restarts);

  for (int cycle = 0; cycle <= max_cycles && nb > 0; ++cycle) {
    // FP64-accurate residual R = B - (shift X + M X)
    sigma_batch(c, Xw.p, Yw.p, nb, nb, shw.p, resid_prec, transpose, s);
    {
      const ElGrid eg = el_grid(D, nb);
      residual_kernel<<<eg.grid, eg.block, 0, s>>>(Bw.p, Yw.p, Rw.p, D, nb, partial.p);
      GFCC_LAUNCH_CHECK();
      reduce_norm_kernel<<<(nb + 31) / 32, dim3(32, 8), 0, s>>>(partial.p, (int)eg.grid.y, nb, nrm.p);
      GFCC_LAUNCH_CHECK();
    }
    GFCC_CUDA(cudaMemcpyAsync(hres.data(), nrm.p, sizeof(double) * nb, cudaMemcpyDeviceToHost, s));
    GFCC_CUDA(cudaStreamSynchronize(s));
    c->stats.restarts++;
    if (c->opts.verbose) {
      double mx = 0.0;
      for (int w = 0; w < nb; ++w) mx = std::max(mx, hbn[map[w]] > 0.0 ? hres[w] / hbn[map[w]] : 0.0);
      fprintf(stderr, "gfcc gmres: cycle %d, %d columns, max relative residual %.3e\n", cycle, nb, mx);
    }
    if ((inner_prec != GFCC_PREC_FP64 || resid_prec != GFCC_PREC_FP64) && low_precision_error(c))
      throw Error{GFCC_ERR_CUDA, "solve: a tensor-core pipeline wait timed out"};

    // classify columns: done = written out, keep = iterated on. With polish, a column that first meets the tolerance
    // by less than a factor of four is written out and given one more cycle, whose result replaces it if its
    // residual is smaller.
    std::vector<int> done, keep;
    for (int w = 0; w < nb; ++w) {
      int orig = map[w];
      double bn = hbn[orig];
      double rel = bn > 0.0 ? hres[w] / bn : 0.0;
      if (polished[orig]) {   // (a residual that is not finite is not smaller: the solution in hand stays)
        if (rel < st.relres[orig]) {
          st.relres[orig] = rel;
          done.push_back(w);
        }
        continue;
      }
      GFCC_CHECK(std::isfinite(rel), GFCC_ERR_NONFINITE, "solve: non-finite residual (singular shift?)");
      st.relres[orig] = rel;
      if (rel <= tol || cycle == max_cycles) {
        done.push_back(w);
        st.converged[orig] = rel <= tol ? 1 : 0;
        if (polish && rel > 0.25 * tol && cycle < max_cycles) {
          polished[orig] = 1;
          keep.push_back(w);
        }
      } else {
        keep.push_back(w);
      }
    }
    if (!done.empty()) {  // write finished columns out
      std::vector<int> hd(done.size()), ho(done.size());
      for (size_t q = 0; q < done.size(); ++q) { hd[q] = done[q]; ho[q] = map[done[q]]; }
      DBuf<int> dsrc, ddst;
      dsrc.alloc(hd.size()); ddst.alloc(ho.size());
      GFCC_CUDA(cudaMemcpyAsync(dsrc.p, hd.data(), sizeof(int) * hd.size(), cudaMemcpyHostToDevice, s));
      GFCC_CUDA(cudaMemcpyAsync(ddst.p, ho.data(), sizeof(int) * ho.size(), cudaMemcpyHostToDevice, s));
      gather_cols_kernel<<<grid_for(D * hd.size()), 256, 0, s>>>(Xw.p, nb, dsrc.p, (int)hd.size(), Ztmp.p,
                                                                  (int)hd.size(), D);
      GFCC_LAUNCH_CHECK();
      scatter_cols_kernel<<<grid_for(D * hd.size()), 256, 0, s>>>(Ztmp.p, (int)hd.size(), ddst.p, (int)hd.size(),
                                                                   Xout, nb0, D);
      GFCC_LAUNCH_CHECK();
      if (Rout) {
        gather_cols_kernel<<<grid_for(D * hd.size()), 256, 0, s>>>(Rw.p, nb, dsrc.p, (int)hd.size(), Ztmp.p,
                                                                    (int)hd.size(), D);
        GFCC_LAUNCH_CHECK();
        scatter_cols_kernel<<<grid_for(D * hd.size()), 256, 0, s>>>(Ztmp.p, (int)hd.size(), ddst.p,
                                                                     (int)hd.size(), Rout, nb0, D);
        GFCC_LAUNCH_CHECK();
      }
      GFCC_CUDA(cudaStreamSynchronize(s));
    }
    if (keep.empty()) { nb = 0; break; }
    if ((int)keep.size() < nb) {  // compact B, X, R, shifts
      int nk = (int)keep.size();
      GFCC_CUDA(cudaMemcpyAsync(cols.p, keep.data(), sizeof(int) * nk, cudaMemcpyHostToDevice, s));
      for (DBuf<cplx>* b : {&Bw, &Xw, &Rw}) {
        gather_cols_kernel<<<grid_for(D * nk), 256, 0, s>>>(b->p, nb, cols.p, nk, Ztmp.p, nk, D);
        GFCC_LAUNCH_CHECK();
        GFCC_CUDA(cudaMemcpyAsync(b->p, Ztmp.p, sizeof(cplx) * D * nk, cudaMemcpyDeviceToDevice, s));
      }
      std::vector<cplx> nsh(nk);
      std::vector<int> nmap(nk);
      for (int q = 0; q < nk; ++q) { nsh[q] = hshift[map[keep[q]]]; nmap[q] = map[keep[q]]; }
      GFCC_CUDA(cudaMemcpyAsync(shw.p, nsh.data(), sizeof(cplx) * nk, cudaMemcpyHostToDevice, s));
      std::vector<double> nres(nk);
      for (int q = 0; q < nk; ++q) nres[q] = hres[keep[q]];
      GFCC_CUDA(cudaMemcpyAsync(nrm.p, nres.data(), sizeof(double) * nk, cudaMemcpyHostToDevice, s));
      hres = nres;
      map = nmap;
      nb = nk;
      GFCC_CUDA(cudaStreamSynchronize(s));
    }
    {  // ||b|| of the working set and the per-column stopping level of this cycle
      std::vector<double> wb(nb), th(nb);
      for (int q = 0; q < nb; ++q) {
        wb[q] = hbn[map[q]];
        th[q] = std::max(target * tol, inner_rtol * hres[q] / wb[q]);
      }
      GFCC_CUDA(cudaMemcpyAsync(bnorm.p, wb.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, s));
      GFCC_CUDA(cudaMemcpyAsync(thr.p, th.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, s));
    }
    // GMRES(k) on the correction: V0 = R / ||R||, g = (||R||, 0, ...)
    {
      std::vector<cplx> g0((size_t)nb * (k + 1), make_cuDoubleComplex(0.0, 0.0));
      for (int q = 0; q < nb; ++q) g0[q] = make_cuDoubleComplex(hres[q], 0.0);
      GFCC_CUDA(cudaMemcpyAsync(g.p, g0.data(), sizeof(cplx) * g0.size(), cudaMemcpyHostToDevice, s));
      std::vector<int> ones(nb, 1);
      GFCC_CUDA(cudaMemcpyAsync(live.p, ones.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, s));
      GFCC_CUDA(cudaMemsetAsync(kc.p, 0, sizeof(int) * nb, s));
      GFCC_CUDA(cudaMemsetAsync(nlive.p, 0, sizeof(int) * k, s));
      GFCC_CUDA(cudaMemsetAsync(H.p, 0, sizeof(cplx) * (size_t)nb * (k + 1) * k, s));
    }
    const long long vstride = D * nb;
    const ElGrid eg = el_grid(D, nb);
    // v_j = w / ||w|| and what the inner action needs of z = P v_j: its operands (FP32 basis) or z itself
    auto start_step = [&](const auto* w, int j) {
      ProfScope pk(PROF_KRYLOV, 0.0, s);
      if constexpr (F32) {
        sigma_lp_prepare(c, w, invf.p, V.p + j * vstride, nb, shf.p, s, transpose);
      } else {
        scale_precond_kernel<<<eg.grid, eg.block, 0, s>>>(w, nrm.p, V.p + j * vstride, Zw.p, c->op.mdiag.p, shw.p, D, nb);
        GFCC_LAUNCH_CHECK();
      }
    };
    if (F32) {
      split_shifts(shw.p, nb, shf.p, s);
      inv_norm_kernel<<<(nb + 127) / 128, 128, 0, s>>>(nrm.p, nb, invf.p);
      GFCC_LAUNCH_CHECK();
    }
    start_step(Rw.p, 0);
    int steps = 0;
    for (int j = 0; j < k; ++j) {
      VT* Vj = V.p + j * vstride;
      if constexpr (F32) sigma_lp_apply(c, Vj, Ww.p, nb, shf.p, s, transpose);
      else sigma_batch(c, Zw.p, Ww.p, nb, nb, shw.p, inner_prec, transpose, s);
      ProfScope pk2(PROF_KRYLOV, 0.0, s);
      const int nv = j + 1;
      cplx* Hc = H.p + (long long)j * (k + 1) * nb;
      int norm_chunks = 0;   // chunk sums of ||w||^2 left in partial
      if constexpr (F32) {
        // CGS with delayed re-orthogonalisation (see the sweeps): final V_j, w through its first pass, ||w||^2
        // algorithmic HBM bytes: V read twice; a and u read twice and written once
        const double vbytes = (double)D * nb * sizeof(VT);   // one vector of the batch
        ProfScope pcgs(PROF_KRYLOV_CGS, (2.0 * j + 6.0) * vbytes, s);
        const long long rows = sweep_rows(D, nb);
        const int nchunk = (int)((D + rows - 1) / rows), small = nb < MD_TX ? 1 : 0;
        SweepArgs sa{};
        sa.vstride = vstride;
        sa.a = reinterpret_cast<float2*>(Vj);
        sa.u = reinterpret_cast<float2*>(Ww.p);
        sa.D = D; sa.nb = nb;
        sa.partial = partial.p;
        // sums [g (j) | r (j) | scalars (2)]: a part of i0 .. i0 + n of the basis writes its g and r next to each other,
        // from 2 i0 on
        for (int i0 = 0; i0 == 0 || i0 < j; i0 += MD_MAXV) {
          const int n = std::min(MD_MAXV, j - i0);
          const int nq = 2 * n + (i0 == 0 ? 2 : 0);
          sa.V = reinterpret_cast<const float2*>(V.p) + i0 * vstride;
          sa.nv = n;
          sa.scalars = i0 == 0;
          {
            ProfScope pk(small ? PROF_CGS_SMALL_NB : PROF_CGS_DOTS, (n + 2.0) * vbytes, s);
            launch_sweep<false>(sa, s);
          }
          // the first part's scalars follow its g and r; later parts start behind them
          const long long o0 = (i0 == 0 ? 0 : 2LL * i0 + 2) * nb;
          reduce_dots_kernel<<<dim3((nb + 31) / 32, nq), dim3(32, 8), 0, s>>>(partial.p, nchunk, nq, nb, sums.p + o0,
                                                                             sums_f.p + o0);
          GFCC_LAUNCH_CHECK();
        }
        const int n0 = std::min(MD_MAXV, j);
        if (j > n0) {   // g and r of all parts in two rows of blocks
          for (int i0 = 0; i0 < j; i0 += MD_MAXV) {
            const int n = std::min(MD_MAXV, j - i0);
            const cplx* src = sums.p + (i0 == 0 ? 0 : 2LL * i0 + 2) * nb;
            GFCC_CUDA(cudaMemcpyAsync(gr.p + (long long)i0 * nb, src, sizeof(cplx) * n * nb, cudaMemcpyDeviceToDevice, s));
            GFCC_CUDA(cudaMemcpyAsync(gr.p + (long long)(j + i0) * nb, src + (long long)n * nb, sizeof(cplx) * n * nb,
                                      cudaMemcpyDeviceToDevice, s));
          }
        }
        const cplx* gp = j > n0 ? gr.p : sums.p;
        delayed_coef_kernel<<<(nb + 15) / 16, 128, 0, s>>>(gp, gp + (long long)j * nb, j, sums.p + 2LL * n0 * nb, nb, Hc,
                                                           fin.p);
        GFCC_LAUNCH_CHECK();
        for (int i0 = 0; i0 == 0 || i0 < j; i0 += MD_MAXV) {
          const int n = std::min(MD_MAXV, j - i0);
          const long long o0 = (i0 == 0 ? 0 : 2LL * i0 + 2) * nb;
          sa.V = reinterpret_cast<const float2*>(V.p) + i0 * vstride;
          sa.nv = n;
          sa.g = sums_f.p + o0;
          sa.r = sums_f.p + o0 + (long long)n * nb;
          sa.fin = fin.p;
          sa.last = i0 + MD_MAXV >= j;
          ProfScope pk(small ? PROF_CGS_SMALL_NB : PROF_CGS_UPDATE, (n + 4.0) * vbytes, s);
          launch_sweep<true>(sa, s);
        }
        norm_chunks = nchunk;
      } else {
        // CGS with one re-orthogonalisation: h1 = V^H w, w -= V h1, h2 = V^H w, w -= V h2; H[:, j] = h1 + h2
        for (int pass = 0; pass < 2; ++pass) {
          multidot<VT>(V.p, vstride, nv, Ww.p, D, nb, hb.p, k + 1, Hc, pass == 1, partial, s);
          update_kernel<VT><<<eg.grid, eg.block, 0, s>>>(V.p, vstride, nv, Ww.p, D, nb, hb.p, k + 1);
          GFCC_LAUNCH_CHECK();
        }
        col_norms<VT>(Ww.p, D, nb, nrm.p, partial, s);
      }
      arnoldi_finish_kernel<<<(nb + 31) / 32, GV_T, 0, s>>>(partial.p, norm_chunks, nrm.p, invf.p, H.p, cs.p, sn.p, g.p,
                                                            bnorm.p, kc.p, live.p, nb, k, j, thr.p, nlive.p + j,
                                                            F32 ? fin.p : nullptr);
      GFCC_LAUNCH_CHECK();
      GFCC_CUDA(cudaMemcpyAsync(c->pin, nlive.p + j, sizeof(int), cudaMemcpyDeviceToHost, s));
      GFCC_CUDA(cudaEventRecord(c->pin_event, s));
      // the next step's first kernels run while the host waits for the count (if no column is left, they wrote
      // one more basis vector that nothing uses)
      if (j + 1 < k) start_step(Ww.p, j + 1);
      GFCC_CUDA(cudaEventSynchronize(c->pin_event));
      const int hl = *c->pin;
      steps = j + 1;
      c->stats.gmres_iters++;
      for (int q = 0; q < nb; ++q) st.iters[map[q]]++;
      if (hl == 0) break;
    }
    backsolve_kernel<VT><<<(nb + 3) / 4, 128, 0, s>>>(H.p, g.p, kc.p, nb, k, yv.p);
    GFCC_LAUNCH_CHECK();
    // X += P V y (only the first kc basis vectors carry weight; later y entries are zero)
    correct_kernel<VT><<<eg.grid, eg.block, 0, s>>>(V.p, vstride, steps, yv.p, Xw.p, c->op.mdiag.p, c->op.rowf.p,
                                                    shw.p, shf.p, D, nb);
    GFCC_LAUNCH_CHECK();
  }
  GFCC_CUDA(cudaStreamSynchronize(s));
}

void gmres_batched(gfcc_ctx* c, const cplx* Bin, cplx* Xout, cplx* Rout, const cplx* shifts_dev, int nb0,
                   SolveStatus& st, bool transpose, const cplx* X0, bool polish) {
  const bool f32 = c->opts.precision == GFCC_PREC_TF32 || c->opts.precision == GFCC_PREC_BF16;
  if (f32) gmres_impl<cuFloatComplex>(c, Bin, Xout, Rout, shifts_dev, nb0, st, transpose, X0, polish);
  else gmres_impl<cplx>(c, Bin, Xout, Rout, shifts_dev, nb0, st, transpose, X0, polish);
}

// ------------------------------------------------------------------------------------------------
namespace {
__global__ void gather_rows_kernel(const double* __restrict__ src, int ld_src, const int* __restrict__ rows,
                                   int nrows, long long D, cplx* __restrict__ dst, int ldb) {
  long long total = D * nrows;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int kq = (int)(t % nrows);
    long long nu = t / nrows;
    dst[nu * ldb + kq] = make_cuDoubleComplex(src[(long long)rows[kq] * ld_src + nu], 0.0);
  }
}
__global__ void cols_to_batch_kernel(const cplx* __restrict__ src, int lds, int ncols, long long D,
                                     cplx* __restrict__ dst, int ldb) {
  long long total = D * ncols;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int cc = (int)(t % ncols);
    long long nu = t / ncols;
    dst[nu * ldb + cc] = src[(long long)cc * lds + nu];
  }
}
__global__ void batch_to_cols_kernel(const cplx* __restrict__ src, int ldb, int ncols, long long D,
                                     cplx* __restrict__ dst, int ldd) {
  long long total = D * ncols;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    long long nu = t % D;
    int cc = (int)(t / D);
    dst[(long long)cc * ldd + nu] = src[nu * ldb + cc];
  }
}
}  // namespace

void gather_rows_real_to_cplx(const double* src, int ld_src, const int* rows, int nrows, int D, cplx* dst,
                              int ldb, cudaStream_t s) {
  if (nrows == 0) return;
  gather_rows_kernel<<<grid_for((long long)D * nrows), 256, 0, s>>>(src, ld_src, rows, nrows, D, dst, ldb);
  GFCC_LAUNCH_CHECK();
}
void pack_cols_to_batch(const cplx* src, int ld_src, int ncols, int D, cplx* dst, int ldb, cudaStream_t s) {
  if (ncols == 0) return;
  cols_to_batch_kernel<<<grid_for((long long)D * ncols), 256, 0, s>>>(src, ld_src, ncols, D, dst, ldb);
  GFCC_LAUNCH_CHECK();
}
void batch_to_cols(const cplx* src, int ldb, int ncols, int D, cplx* dst, int ld_dst, cudaStream_t s) {
  if (ncols == 0) return;
  batch_to_cols_kernel<<<grid_for((long long)D * ncols), 256, 0, s>>>(src, ldb, ncols, D, dst, ld_dst);
  GFCC_LAUNCH_CHECK();
}

// G[c][q] = sum_nu c_q[nu] X[nu][c]  as a complex GEMM with a real-valued left operand: do it as a
// real GEMM on the interleaved columns: G'[q][2c+r] = sum_nu cvec[q][nu] X'[nu][2c+r]
// G[c][q] = sum_nu c_q[nu] X[nu][c]: each block reduces a chunk of rows for every (q, c) pair
// (threads over pairs, X rows read coalesced, c_q[nu] broadcast), then the chunks are summed.
namespace {
__global__ void green_partial_kernel(const double* __restrict__ cq, long long D, int nq, const cplx* __restrict__ X,
                                     int ldb, int ncols, long long rows, cplx* __restrict__ part) {
  const long long r0 = blockIdx.x * rows, r1 = min(D, r0 + rows);
  const int npair = nq * ncols;
  for (int t = blockIdx.y * blockDim.x + threadIdx.x; t < npair; t += gridDim.y * blockDim.x) {
    const int q = t / ncols, c = t % ncols;
    const double* cr = cq + (long long)q * D;
    double sr = 0.0, si = 0.0;
    for (long long nu = r0; nu < r1; ++nu) {
      const double w = cr[nu];
      const cplx x = X[nu * ldb + c];
      sr = fma(w, x.x, sr);
      si = fma(w, x.y, si);
    }
    part[(long long)blockIdx.x * npair + t] = make_cuDoubleComplex(sr, si);
  }
}
__global__ void green_reduce_kernel(const cplx* __restrict__ part, int nchunk, int nq, int ncols, cplx* __restrict__ G) {
  const int npair = nq * ncols;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= npair) return;
  double sr = 0.0, si = 0.0;
  for (int k = 0; k < nchunk; ++k) {
    sr += part[(long long)k * npair + t].x;
    si += part[(long long)k * npair + t].y;
  }
  const int q = t / ncols, c = t % ncols;
  G[(long long)c * nq + q] = make_cuDoubleComplex(sr, si);
}
}  // namespace

void green_from_batch(const double* cvec, int D, const int* qrows_host, int nq, const cplx* X, int ldb,
                      int ncols, cplx* G, cudaStream_t s) {
  if (nq == 0 || ncols == 0) return;
  DBuf<double> Cq;
  DBuf<cplx> part;
  Cq.alloc((long long)nq * D);
  for (int q = 0; q < nq; ++q)
    GFCC_CUDA(cudaMemcpyAsync(Cq.p + (long long)q * D, cvec + (long long)qrows_host[q] * D, sizeof(double) * D,
                              cudaMemcpyDeviceToDevice, s));
  const long long rows = std::max<long long>(64, (D + 2 * 152 * 4 - 1) / (2 * 152 * 4));
  const int nchunk = (int)((D + rows - 1) / rows);
  part.alloc((long long)nchunk * nq * ncols);
  // few chunks (small D): the pairs are spread over blocks too
  const int gy = (int)std::max<long long>(1, std::min<long long>(((long long)nq * ncols + 255) / 256, 1216 / nchunk));
  green_partial_kernel<<<dim3(nchunk, gy), 256, 0, s>>>(Cq.p, D, nq, X, ldb, ncols, rows, part.p);
  GFCC_LAUNCH_CHECK();
  green_reduce_kernel<<<(nq * ncols + 255) / 256, 256, 0, s>>>(part.p, nchunk, nq, ncols, G);
  GFCC_LAUNCH_CHECK();
  GFCC_CUDA(cudaStreamSynchronize(s));
}

}  // namespace gfcc

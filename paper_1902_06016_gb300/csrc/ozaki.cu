// Exact-slice FP64 GEMM on the tensor cores (see ozaki.cuh).
#include "ozaki.cuh"
#include "tc_gemm.cuh"

#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>
#include <cstdlib>

namespace gfcc {
namespace {

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)std::min<long long>(std::max<long long>(g, 1), 152LL * 32);
}

// ---- integer slicing -----------------------------------------------------------------------------
// Every step below is integer arithmetic on the FP64 bit patterns (FP64 instructions run on a narrow
// pipe on this GPU). For non-negative doubles the bit patterns order like the values, so the row
// maximum of |x| is an integer maximum, and the row exponent e (max |x| < 2^e, as frexp) is read
// from its exponent field; a row whose maximum is zero or subnormal is treated as zero.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFULL;
}
constexpr int ZERO_ROW = -100000;   // row exponent marker of a zero (or subnormal-only) row
__device__ __forceinline__ int row_exponent(unsigned long long maxbits) {
  const int ex = (int)(maxbits >> 52);
  return ex == 0 ? ZERO_ROW : ex - 1022;
}
// Balanced digits of B bits of x relative to 2^(e - B + 1), for B = 9:  x ~ 2^(e-8) sum_{i<ns} a_i 2^(-9i), |a_i| <= 256.
// V = round(|x| 2^(8 - e + 9(ns-1))) is formed exactly from the mantissa (|V| <= 2^(8 + 9(ns-1)) <= 2^62);
// digit i is V / 2^(9(ns-1-i)) rounded half up, V keeps the remainder (|remainder| <= 2^(shift-1)), and
// the signs of all digits follow x (so -x gives exactly the negated digits). a[i] holds digit i. The slice
// count NS is a template argument (no predicated iterations, constant shifts).
template <int NS, int B = OZ_BITS>
__device__ __forceinline__ void digits_t(double x, int e, int (&a)[NS]) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  long long V = 0;
  if (ex != 0 && e != ZERO_ROW) {
    const long long m = (bits & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
    const int t = ex - 1075 + (B - 1) - e + B * (NS - 1);
    if (t >= 0) V = m << t;
    else if (t > -62) V = (m + (1LL << (-t - 1))) >> (-t);
  }
  const bool neg = bits < 0;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int shift = B * (NS - 1 - i);
    const long long d = (i < NS - 1) ? ((V + (1LL << (shift - 1))) >> shift) : V;
    V -= d << shift;
    a[i] = neg ? -(int)d : (int)d;
  }
}
// digits of two adjacent elements of a row, written as one f16 pair per slot (k even)
template <int NS>
__device__ __forceinline__ void slice_pair(double x0, double x1, int e, __half* __restrict__ o, long long kp,
                                           int reversed, long long k) {
  int a0[NS], a1[NS];
  digits_t<NS>(x0, e, a0);
  digits_t<NS>(x1, e, a1);
#pragma unroll
  for (int i = 0; i < NS; ++i)
    *reinterpret_cast<__half2*>(o + (long long)(reversed ? NS - 1 - i : i) * kp + k) =
        __halves2half2(__int2half_rn(a0[i]), __int2half_rn(a1[i]));
}

// Real rows (row-major, row stride ldx, K used columns): one block per row (grid-stride) for long
// rows; slices [r][slot][kp] with slot = i (or ns-1-i when reversed), zeros for K <= k < kp.
template <int NS>
__global__ void __launch_bounds__(256) slice_kernel(const double* __restrict__ X, long long ldx, long long rows,
                                                    long long K, long long kp, int reversed,
                                                    __half* __restrict__ out, int* __restrict__ expo) {
  __shared__ unsigned long long red[8];
  for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
    const double* x = X + r * ldx;
    unsigned long long mx = 0;
    for (long long k = threadIdx.x; k < K; k += blockDim.x) mx = max(mx, abs_bits(x[k]));
    for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, red[w]);
    const int e = row_exponent(mx);
    __syncthreads();
    if (threadIdx.x == 0) expo[r] = e == ZERO_ROW ? 0 : e;
    __half* o = out + r * (long long)NS * kp;
    for (long long k = 2LL * threadIdx.x; k < kp; k += 2LL * blockDim.x)
      slice_pair<NS>(k < K ? x[k] : 0.0, k + 1 < K ? x[k + 1] : 0.0, e, o, kp, reversed, k);
  }
}
// The same for short rows: one warp per row.
template <int NS>
__global__ void __launch_bounds__(256) slice_rows_warp_kernel(const double* __restrict__ X, long long ldx,
                                                              long long rows, long long K, long long kp, int reversed,
                                                              __half* __restrict__ out, int* __restrict__ expo) {
  const long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  const double* x = X + r * ldx;
  unsigned long long mx = 0;
  for (long long k = lane; k < K; k += 32) mx = max(mx, abs_bits(x[k]));
  for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  const int e = row_exponent(mx);
  if (lane == 0) expo[r] = e == ZERO_ROW ? 0 : e;
  __half* o = out + r * (long long)NS * kp;
  for (long long k = 2LL * lane; k < kp; k += 64)
    slice_pair<NS>(k < K ? x[k] : 0.0, k + 1 < K ? x[k + 1] : 0.0, e, o, kp, reversed, k);
}

// The same for a few long rows (fewer rows than it takes to occupy the GPU with a block each): the
// row maxima over chunks of SL_CH elements (atomic integer maxima of the bit patterns; rowmax zeroed by
// the caller), then the digits chunk by chunk.
constexpr long long SL_CH = 8192;
__global__ void __launch_bounds__(256) rowmax_chunk_kernel(const double* __restrict__ X, long long ldx, long long K,
                                                           unsigned long long* __restrict__ rowmax) {
  __shared__ unsigned long long red[8];
  const long long r = blockIdx.y, k0 = blockIdx.x * SL_CH, k1 = min(K, k0 + SL_CH);
  const double* x = X + r * ldx;
  unsigned long long mx = 0;
  for (long long k = k0 + threadIdx.x; k < k1; k += blockDim.x) mx = max(mx, abs_bits(x[k]));
  for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, red[w]);
    if (mx > 0) atomicMax(rowmax + r, mx);
  }
}
template <int NS>
__global__ void __launch_bounds__(256) slice_chunk_kernel(const double* __restrict__ X, long long ldx, long long K,
                                                          long long kp, int reversed,
                                                          const unsigned long long* __restrict__ rowmax,
                                                          __half* __restrict__ out, int* __restrict__ expo) {
  const long long r = blockIdx.y, k0 = blockIdx.x * SL_CH, k1 = min(kp, k0 + SL_CH);   // SL_CH is even
  const double* x = X + r * ldx;
  const int e = row_exponent(rowmax[r]);
  if (blockIdx.x == 0 && threadIdx.x == 0) expo[r] = e == ZERO_ROW ? 0 : e;
  __half* o = out + r * (long long)NS * kp;
  for (long long k = k0 + 2LL * threadIdx.x; k < k1; k += 2LL * blockDim.x)
    slice_pair<NS>(k < K ? x[k] : 0.0, k + 1 < K ? x[k + 1] : 0.0, e, o, kp, reversed, k);
}

// the slice count of a launch as a template argument (2..7 slices)
template <typename F>
void with_ns(int ns, F&& f) {
  switch (ns) {
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    default: f(std::integral_constant<int, 7>{}); break;
  }
}

// and the digits' width: 9 bits, or 7 with 7 slices (see OZ_BITS_MOR)
template <typename F>
void with_digits(int ns, int bits, F&& f) {
  if (bits == OZ_BITS) with_ns(ns, [&](auto NSc) { f(NSc, std::integral_constant<int, OZ_BITS>{}); });
  else f(std::integral_constant<int, OZ_SLICES_MOR>{}, std::integral_constant<int, OZ_BITS_MOR>{});
}

// ---- complex operands of zgemm_oz, sliced straight from their strided storage ----------------------
// Operand element (r, k) = Z[r * s_r + k * s_k] (complex), conjugated when conj. Real rows written:
//   mode 0 (left operand):  row r      = (Re, Im) interleaved along k
//   mode 1 (right operand): row r      = (Re, -Im)    and row R + r = (Im, Re)
// so that sum over the 2K real columns of left row m times right row n (or R + n) gives the real
// (imaginary) part of the complex product. Tiles of 32 rows x 64 complex k go through shared memory
// so that both the strided reads and the row-contiguous slice writes are coalesced; the blocks walk the row
// tiles (any number of rows).
constexpr int ZT_R = 32, ZT_K = 64;

__device__ __forceinline__ void load_ztile(const cplx* __restrict__ Z, long long s_r, long long s_k, int conj,
                                           long long R, long long K, long long r0, long long k0,
                                           cplx (*tile)[ZT_K + 1]) {
  if (s_r == 1) {   // consecutive rows are adjacent: threads along r
    const int tr = threadIdx.x & 31;
    for (int tk = threadIdx.x >> 5; tk < ZT_K; tk += blockDim.x >> 5) {
      const long long r = r0 + tr, k = k0 + tk;
      cplx v = make_cuDoubleComplex(0.0, 0.0);
      if (r < R && k < K) v = Z[r + k * s_k];
      if (conj) v.y = -v.y;
      tile[tr][tk] = v;
    }
  } else {          // threads along k
    for (int i = threadIdx.x; i < ZT_R * ZT_K; i += blockDim.x) {
      const int tr = i / ZT_K, tk = i % ZT_K;
      const long long r = r0 + tr, k = k0 + tk;
      cplx v = make_cuDoubleComplex(0.0, 0.0);
      if (r < R && k < K) v = Z[r * s_r + k * s_k];
      if (conj) v.y = -v.y;
      tile[tr][tk] = v;
    }
  }
}

// rowmax[r] = max over k of the bit patterns of |Re|, |Im| (atomic; rowmax zeroed by the caller)
__global__ void __launch_bounds__(256) zrowmax_kernel(const cplx* __restrict__ Z, long long s_r, long long s_k,
                                                      long long R, long long K,
                                                      unsigned long long* __restrict__ rowmax) {
  __shared__ cplx tile[ZT_R][ZT_K + 1];
  const long long k0 = (long long)blockIdx.x * ZT_K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long r0 = (long long)blockIdx.y * ZT_R; r0 < R; r0 += (long long)gridDim.y * ZT_R) {
    load_ztile(Z, s_r, s_k, 0, R, K, r0, k0, tile);
    __syncthreads();
    for (int tr = warp; tr < ZT_R; tr += blockDim.x >> 5) {
      unsigned long long mx = 0;
      for (int tk = lane; tk < ZT_K; tk += 32) mx = max(mx, max(abs_bits(tile[tr][tk].x), abs_bits(tile[tr][tk].y)));
      for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      if (lane == 0 && r0 + tr < R && mx > 0) atomicMax(rowmax + r0 + tr, mx);
    }
    __syncthreads();
  }
}

// Slices of row r at (r ns + slot) kp (row-major), or with slot_major at (slot rows_total + r) kp, where
// rows_total = R (mode 0) or 2R (mode 1): then slots 0..j of all rows form one contiguous block of rows.
template <int NS, int B>
__global__ void __launch_bounds__(256) zslice_kernel(const cplx* __restrict__ Z, long long s_r, long long s_k,
                                                     int conj, long long R, long long K, int mode,
                                                     const unsigned long long* __restrict__ rowmax, long long kp,
                                                     int reversed, __half* __restrict__ out,
                                                     int* __restrict__ expo, int slot_major = 0) {
  constexpr int ns = NS;
  __shared__ cplx tile[ZT_R][ZT_K + 1];
  const long long k0 = (long long)blockIdx.x * ZT_K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long r0 = (long long)blockIdx.y * ZT_R; r0 < R; r0 += (long long)gridDim.y * ZT_R) {
    load_ztile(Z, s_r, s_k, conj, R, K, r0, k0, tile);
    __syncthreads();
    for (int tr = warp; tr < ZT_R; tr += blockDim.x >> 5) {
      const long long r = r0 + tr;
      if (r >= R) break;
      const int e = row_exponent(rowmax[r]);
      if (k0 == 0 && lane == 0) {
        expo[r] = e == ZERO_ROW ? 0 : e;
        if (mode == 1) expo[R + r] = e == ZERO_ROW ? 0 : e;
      }
      const long long rows_total = mode == 1 ? 2 * R : R;
      // element offset of slot 0 of a row and the distance between its slots
      const long long b0 = slot_major ? r * kp : r * (long long)ns * kp;
      const long long b1 = slot_major ? (R + r) * kp : (R + r) * (long long)ns * kp;
      const long long sstep = slot_major ? rows_total * kp : kp;
      __half* o0 = out + b0;
      __half* o1 = out + b1;
      for (int tk = lane; tk < ZT_K; tk += 32) {
        const long long k = k0 + tk;
        if (2 * k >= kp) break;
        const cplx v = tile[tr][tk];
        int are[NS], aim[NS];
        digits_t<NS, B>(v.x, e, are);
        digits_t<NS, B>(v.y, e, aim);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
          {
            const long long off = (long long)(reversed ? ns - 1 - i : i) * sstep + 2 * k;
            if (mode == 0) {
              *reinterpret_cast<__half2*>(o0 + off) = __halves2half2(__int2half_rn(are[i]),
                                                                                 __int2half_rn(aim[i]));
            } else {
              *reinterpret_cast<__half2*>(o0 + off) = __halves2half2(__int2half_rn(are[i]),
                                                                                 __int2half_rn(-aim[i]));
              *reinterpret_cast<__half2*>(o1 + off) = __halves2half2(__int2half_rn(aim[i]),
                                                                                 __int2half_rn(are[i]));
            }
          }
        }
      }
    }
    __syncthreads();
  }
}

// Output of an exact-slice product: real, out[m ldo + n] = alpha P[m][n] + beta out (alpha real); or complex (the real
// columns n and N + n of P hold the real and imaginary parts), C(m, n) = alpha P(m, n) + beta C(m, n).
struct OzOut {
  bool complex_out = false;
  double* out = nullptr;
  long long ldo = 0;
  double beta = 0.0;
  cplx* C = nullptr;
  long long scm = 0, scn = 0;
  int bits = OZ_BITS;   // of the operands' digits
  cplx alpha = {1.0, 0.0}, cbeta = {0.0, 0.0};
  // the common cases, so that the output pass spends no FP64 multiplications on them (set by set_kinds):
  // alpha_kind 1: alpha = 1, 2: alpha = -1, 0: general; beta_kind 0: beta = 0, 1: beta = 1, 2: general
  int alpha_kind = 1, beta_kind = 0;
  void set_kinds() {
    alpha_kind = (alpha.y == 0.0 && alpha.x == 1.0) ? 1 : (alpha.y == 0.0 && alpha.x == -1.0) ? 2 : 0;
    if (complex_out) beta_kind = (cbeta.x == 0.0 && cbeta.y == 0.0) ? 0 : (cbeta.x == 1.0 && cbeta.y == 0.0) ? 1 : 2;
    else beta_kind = beta == 0.0 ? 0 : beta == 1.0 ? 1 : 2;
  }
};

// x 2^k by one multiplication with an exact power of two when 2^k is a normal number (ldexp otherwise)
__device__ __forceinline__ double scale_pow2(double x, int k) {
  if (k >= -1022 && k <= 1023) return x * __longlong_as_double((long long)(k + 1023) << 52);
  return ldexp(x, k);
}
// 2^e sum_d S_d 2^(B (NS - 1 - d)) for NS <= 7, B <= 9 per-diagonal integer sums |S_d| < 2^43, rounded once to nearest: the sum
// is formed exactly (three diagonals at a time in 64 bits, joined in 128) and the double assembled from its bits.
// Integer instructions throughout: the FP64 form (two conversions, a fused multiply-add, a scaling) held each
// scheduler for 300 clocks per warp and bound the output passes.
template <int NS, int B>
__device__ __forceinline__ double diag_value(const long long (&S)[NS], int e) {
  constexpr int H = NS < 3 ? NS : 3, L = NS < 6 ? NS : 6;   // diagonals [0, H), [H, L), [L, NS)
  long long hi = 0, mid = 0, lo = 0;
#pragma unroll
  for (int d = 0; d < NS; ++d) {
    if (d < H) hi += S[d] * (1LL << (B * (H - 1 - d)));
    else if (d < L) mid += S[d] * (1LL << (B * (L - 1 - d)));
    else lo += S[d];
  }
  const __int128 T = (__int128)hi * ((__int128)1 << (B * (NS - H))) + (__int128)mid * ((__int128)1 << (B * (NS - L))) + lo;
  if (T == 0) return 0.0;
  const bool neg = T < 0;
  const unsigned __int128 A = neg ? -(unsigned __int128)T : (unsigned __int128)T;
  const unsigned long long ah = (unsigned long long)(A >> 64), al = (unsigned long long)A;
  const int n = ah ? 128 - __clzll((long long)ah) : 64 - __clzll((long long)al);   // bits
  // the top 64 bits, left-aligned, and whether anything is left below them
  const int sh = 128 - n;
  const unsigned __int128 Al = A << sh;
  const unsigned long long top = (unsigned long long)(Al >> 64);
  const bool rest = (unsigned long long)Al != 0;
  unsigned long long m = top >> 11;                       // 53 bits
  const unsigned long long low = top & 0x7FFULL;          // and 11 more
  if (low > 0x400ULL || (low == 0x400ULL && (rest || (m & 1)))) ++m;   // to nearest, ties to even
  const int E = n - 1 + e + 1023 + (int)(m >> 53);        // a carry out of the mantissa leaves m = 2^53
  if (E < 1 || E > 2046) {                                // subnormal or overflowing: by the library
    const double v = ldexp((double)m, n - 53 + e);
    return neg ? -v : v;
  }
  const unsigned long long bits = ((unsigned long long)E << 52) | (m & 0xFFFFFFFFFFFFFULL);
  return __longlong_as_double((long long)(neg ? bits | 0x8000000000000000ULL : bits));
}
// complex output value: alpha (re + i im) + beta C
__device__ __forceinline__ cplx out_value(const OzOut& o, double re, double im, const cplx* p) {
  cplx r;
  if (o.alpha_kind == 1) r = make_cuDoubleComplex(re, im);
  else if (o.alpha_kind == 2) r = make_cuDoubleComplex(-re, -im);
  else r = cuCmul(o.alpha, make_cuDoubleComplex(re, im));
  if (o.beta_kind == 1) {
    const cplx q = *p;
    r.x += q.x;
    r.y += q.y;
  } else if (o.beta_kind == 2) {
    r = cuCadd(r, cuCmul(o.cbeta, *p));
  }
  return r;
}
// real output value: alpha v + beta out
__device__ __forceinline__ double out_value_real(const OzOut& o, double v, const double* p) {
  if (o.alpha_kind != 1) v = o.alpha_kind == 2 ? -v : o.alpha.x * v;
  return o.beta_kind == 0 ? v : o.beta_kind == 1 ? v + *p : o.beta * (*p) + v;
}

// sum over the zs int32 split sums p[z stride], exactly in 64-bit integers; WARP: the lanes share the
// splits and every lane returns the total (integer sums do not depend on the grouping)
template <bool WARP>
__device__ __forceinline__ long long split_sum(const int* __restrict__ p, int zs, long long stride, int lane) {
  long long sum = 0;
  if constexpr (WARP) {
    for (int z = lane; z < zs; z += 32) sum += p[(long long)z * stride];
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  } else {
    (void)lane;
    long long s1 = 0, s2 = 0, s3 = 0;   // four independent loads in flight
    int z = 0;
    for (; z + 4 <= zs; z += 4) {
      sum += p[(long long)z * stride];
      s1 += p[(long long)(z + 1) * stride];
      s2 += p[(long long)(z + 2) * stride];
      s3 += p[(long long)(z + 3) * stride];
    }
    for (; z < zs; ++z) sum += p[(long long)z * stride];
    sum += s1 + s2 + s3;
  }
  return sum;
}

// One diagonal of a column chunk (Np real columns): its split sums, weighted by scale = 2^(-bits d), are
// added to the FP64 accumulator acc[m][n'] (MODE 0; first: acc is set), or, on the last diagonal, added
// to acc, scaled by 2^(ea[m] + eb[n'] - 2 (bits - 1)) and written to a real (MODE 1) or complex (MODE 2) output.
// One thread per element, or (WARP) one warp for outputs too small to occupy the GPU that have many K
// splits. Only the last diagonal needs the (m, n) of an element; 32-bit division when it fits.
template <typename I>
__device__ __forceinline__ void divmod(long long t, long long N, long long& m, long long& n) {
  m = (long long)((I)t / (I)N);
  n = t - m * N;
}
template <bool WARP, int MODE, typename I>
__global__ void __launch_bounds__(256) oz_accumulate_kernel(const int* __restrict__ part, int zs, long long M,
                                                            long long Np, double scale, int first,
                                                            double* __restrict__ acc, const int* __restrict__ ea,
                                                            const int* __restrict__ eb, OzOut o) {
  const long long stride = M * Np;
  const long long total = MODE == 2 ? M * (Np / 2) : stride;
  const int lane = threadIdx.x & 31;
  const bool writer = !WARP || lane == 0;
  const long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long nthreads = (long long)gridDim.x * blockDim.x;
  const long long start = WARP ? gid >> 5 : gid, step = WARP ? nthreads >> 5 : nthreads;
  for (long long t = start; t < total; t += step) {
    if constexpr (MODE == 0) {
      double a = scale * (double)split_sum<WARP>(part + t, zs, stride, lane);
      if (!first) a = acc[t] + a;
      if (writer) acc[t] = a;
    } else if constexpr (MODE == 1) {
      double a = scale * (double)split_sum<WARP>(part + t, zs, stride, lane);
      if (!first) a = acc[t] + a;
      long long m, n;
      divmod<I>(t, Np, m, n);
      const double v = scale_pow2(a, ea[m] + eb[n] - 2 * (o.bits - 1));
      if (writer) {
        double* p = o.out + m * o.ldo + n;
        *p = out_value_real(o, v, p);
      }
    } else {
      const long long N = Np / 2;
      long long m, n;
      divmod<I>(t, N, m, n);
      const long long tr = m * Np + n, ti = tr + N;
      double ar = scale * (double)split_sum<WARP>(part + tr, zs, stride, lane);
      double ai = scale * (double)split_sum<WARP>(part + ti, zs, stride, lane);
      if (!first) {
        ar = acc[tr] + ar;
        ai = acc[ti] + ai;
      }
      const double re = scale_pow2(ar, ea[m] + eb[n] - 2 * (o.bits - 1)),
                   im = scale_pow2(ai, ea[m] + eb[N + n] - 2 * (o.bits - 1));
      if (writer) {
        cplx* p = o.C + m * o.scm + n * o.scn;
        *p = out_value(o, re, im, p);
      }
    }
  }
}
// All diagonals at once: their split sums held side by side, summed and written to the output in one pass.
// The partial sums of a real column col of row m, diagonal d, are those of the pieces i (one per diagonal in the plain
// form: i = d; in the stacked form, below, the products i = 0..d): piece i starts at off[i], has rows of ncol[i], zs[i]
// splits, and holds the value at column (STACK ? (d - i) Np : 0) + col.
struct OzParts {
  long long off[OZ_SLICES_MAX];
  long long ncol[OZ_SLICES_MAX];
  int zs[OZ_SLICES_MAX];
};
template <int NS, bool STACK>
__device__ __forceinline__ void diag_sums(const int* __restrict__ slabs, const OzParts& q, long long M, long long Np,
                                          long long m, long long col, int z0, int zstep, long long (&S)[NS]) {
#pragma unroll
  for (int d = 0; d < NS; ++d) S[d] = 0;
  if (z0 == 0) {   // the first split of every piece, all loads in flight together
#pragma unroll
    for (int d = 0; d < NS; ++d) {
#pragma unroll
      for (int i = STACK ? 0 : d; i <= d; ++i) S[d] += slabs[q.off[i] + m * q.ncol[i] + (STACK ? (d - i) * Np : 0) + col];
    }
  }
#pragma unroll
  for (int d = 0; d < NS; ++d) {
#pragma unroll
    for (int i = STACK ? 0 : d; i <= d; ++i) {
      const long long stride = M * q.ncol[i];
      const int* p = slabs + q.off[i] + m * q.ncol[i] + (STACK ? (d - i) * Np : 0) + col;
#pragma unroll 4
      for (int z = z0 == 0 ? zstep : z0; z < q.zs[i]; z += zstep) S[d] += p[z * stride];
    }
  }
}
// One thread per output element (complex: both parts).
template <int NS, int B, bool STACK, bool CPLX, typename I>
__global__ void __launch_bounds__(256) oz_output_kernel(const int* __restrict__ slabs, OzParts q, long long M,
                                                        long long Np, const int* __restrict__ ea,
                                                        const int* __restrict__ eb, OzOut o) {
  const long long N = CPLX ? Np / 2 : Np, total = M * N;
  constexpr int sh = -2 * (B - 1) - B * (NS - 1);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    long long m, n;
    divmod<I>(t, N, m, n);
    long long S[NS];
    diag_sums<NS, STACK>(slabs, q, M, Np, m, n, 0, 1, S);
    const double re = diag_value<NS, B>(S, ea[m] + eb[n] + sh);
    if constexpr (CPLX) {
      diag_sums<NS, STACK>(slabs, q, M, Np, m, N + n, 0, 1, S);
      const double im = diag_value<NS, B>(S, ea[m] + eb[N + n] + sh);
      cplx* p = o.C + m * o.scm + n * o.scn;
      *p = out_value(o, re, im, p);
    } else {
      double* p = o.out + m * o.ldo + n;
      *p = out_value_real(o, re, p);
    }
  }
}
// Outputs too small to occupy the GPU that have many K splits: 32 elements per block (coalesced along the row), whose
// splits the eight warps share (a warp per element read one 4-byte sum per 32-byte sector: 87 us for a 270 x 32 product
// with 100 splits).
template <int NS, int B, bool STACK, bool CPLX>
__global__ void __launch_bounds__(256) oz_output_split_kernel(const int* __restrict__ slabs, OzParts q, long long M,
                                                              long long Np, const int* __restrict__ ea,
                                                              const int* __restrict__ eb, OzOut o) {
  __shared__ long long red[8][NS][32];
  __shared__ double val[2][32];
  const long long N = CPLX ? Np / 2 : Np, total = M * N;
  constexpr int sh = -2 * (B - 1) - B * (NS - 1);
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (long long t0 = blockIdx.x * 32LL; t0 < total; t0 += gridDim.x * 32LL) {
    const long long t = t0 + x, m = t / N, n = t - m * N;
    const bool on = t < total;
#pragma unroll
    for (int part = 0; part < (CPLX ? 2 : 1); ++part) {
      const long long col = part ? N + n : n;
      long long S[NS];
      if (on) diag_sums<NS, STACK>(slabs, q, M, Np, m, col, y, 8, S);
#pragma unroll
      for (int d = 0; d < NS; ++d) red[y][d][x] = on ? S[d] : 0;
      __syncthreads();
      if (y < NS) {
        long long s = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) s += red[k][y][x];
        red[0][y][x] = s;   // read and written by this thread alone
      }
      __syncthreads();
      if (y == 0 && on) {
#pragma unroll
        for (int d = 0; d < NS; ++d) S[d] = red[0][d][x];
        val[part][x] = diag_value<NS, B>(S, ea[m] + eb[col] + sh);
      }
      __syncthreads();
    }
    if (y == 0 && on) {
      if constexpr (CPLX) {
        cplx* p = o.C + m * o.scm + n * o.scn;
        *p = out_value(o, val[0][x], val[1][x], p);
      } else {
        double* p = o.out + m * o.ldo + n;
        *p = out_value_real(o, val[0][x], p);
      }
    }
  }
}
template <bool STACK, bool CPLX>
void launch_output(int ns, int splits, cudaStream_t s, const int* slabs, const OzParts& q, long long M, long long Np,
                   const int* ea, const int* eb, const OzOut& o) {
  const long long elements = M * (CPLX ? Np / 2 : Np);
  const bool split = elements < 152LL * 256 && splits > 4 * ns;
  const bool small = M * Np < (1LL << 32);
  auto launch = [&](auto NSc, auto Bc) {
    constexpr int NS = decltype(NSc)::value, B = decltype(Bc)::value;
    if (split)
      oz_output_split_kernel<NS, B, STACK, CPLX><<<(unsigned)((elements + 31) / 32), 256, 0, s>>>(slabs, q, M, Np, ea, eb,
                                                                                                o);
    else if (small)
      oz_output_kernel<NS, B, STACK, CPLX, unsigned><<<grid_for(elements), 256, 0, s>>>(slabs, q, M, Np, ea, eb, o);
    else
      oz_output_kernel<NS, B, STACK, CPLX, unsigned long long><<<grid_for(elements), 256, 0, s>>>(slabs, q, M, Np, ea, eb,
                                                                                                o);
  };
  if constexpr (CPLX) with_digits(ns, o.bits, launch);
  else with_ns(ns, [&](auto NSc) { launch(NSc, std::integral_constant<int, OZ_BITS>{}); });
  GFCC_LAUNCH_CHECK();
}

// ---- stacked form for a narrow right operand --------------------------------------------------------
// When B has few rows and A is large, one product per A slice i multiplies it by B slices 0..ns-1-i
// stacked as rows (B sliced slot-major), so that A is read ns times instead of ns(ns+1)/2 times and the
// narrow B fills more of each tile. Partials of slice i: slabs + off[i], [zs[i]][M][ncol[i]] with
// ncol[i] = (ns - i) Np rounded up to a multiple of four, B slice j in columns [j Np, (j + 1) Np). Diagonal d = i + j is summed exactly
// in 64-bit integers, so the result equals the diagonal-by-diagonal one.

template <bool WARP, int MODE>
void launch_accumulate(bool small, int grid, cudaStream_t s, const int* part, int zs, long long M, long long Np,
                       double scale, int first, double* acc, const int* ea, const int* eb, const OzOut& o) {
  if (small)
    oz_accumulate_kernel<WARP, MODE, unsigned><<<grid, 256, 0, s>>>(part, zs, M, Np, scale, first, acc, ea, eb, o);
  else
    oz_accumulate_kernel<WARP, MODE, unsigned long long><<<grid, 256, 0, s>>>(part, zs, M, Np, scale, first, acc, ea,
                                                                             eb, o);
}

}  // namespace

namespace {
// algorithmic bytes of writing an M x Np output (a complex output holds Np / 2 complex columns), with a
// read of the old values when it is accumulated into
double out_bytes(const OzOut& o, long long M, long long Np) {
  if (o.complex_out) {
    const bool rd = o.cbeta.x != 0.0 || o.cbeta.y != 0.0;
    return (rd ? 2.0 : 1.0) * 16.0 * (double)M * (double)(Np / 2);
  }
  return (o.beta != 0.0 ? 2.0 : 1.0) * 8.0 * (double)M * (double)Np;
}

// Exact product of sliced rows into o. When the int32 split sums of all diagonals fit in 4 GB they are
// kept side by side and summed into the output in one pass. Otherwise the diagonal GEMMs run one at a
// time, each followed by its accumulation into an FP64 buffer, over column chunks that bound the
// split-sum memory (a complex output is one chunk, its real and imaginary columns being finalised
// together).
void oz_run(const SlicedRows& A, const SlicedRows& B, long long M, long long Np, const OzOut& o, OzWork& w,
            cudaStream_t s) {
  const int ns = A.ns;
  const double slab_bytes = oz_slab_bytes();
  const long long kp = A.kp, ld = (long long)ns * kp;
  const __half* As = reinterpret_cast<const __half*>(A.slices.p);
  const __half* Bs = reinterpret_cast<const __half*>(B.slices.p);
  // the diagonals' products, longest first: diagonal d is A slices 0..d against B slices d..0, concatenated along K
  TcExactGroup eg[OZ_SLICES_MAX];
  long long Ns[OZ_SLICES_MAX], ks[OZ_SLICES_MAX], off = 0;
  for (int q = 0; q < ns; ++q) {
    Ns[q] = Np;
    ks[q] = (long long)(ns - q) * kp;
  }
  const int nk_split = tc_exact_nk_split(M, Ns, ks, ns);
  OzParts dg;
  int splits = 0;
  const long long Np4 = (Np + 3) / 4 * 4;   // rows of split sums start on 16 bytes (vector epilogue stores)
  for (int q = 0; q < ns; ++q) {
    const int d = ns - 1 - q;
    eg[q].kA = 0;
    eg[q].kB = (long long)q * kp;
    eg[q].k_pad = ks[q];
    eg[q].N = Np; eg[q].ldp = Np4; eg[q].split_stride = M * Np4;
    eg[q].nk_split = nk_split;
    dg.zs[d] = eg[q].zs();
    dg.off[d] = off;
    dg.ncol[d] = Np4;
    splits += dg.zs[d];
    off += (long long)dg.zs[d] * M * Np4;
  }
  if (4.0 * (double)off <= slab_bytes) {
    // every diagonal's split sums side by side, then one pass that sums them into the output: the
    // output is touched once instead of once per diagonal
    w.islabs.alloc((size_t)off);
    if (w.err.n == 0) { w.err.alloc(1); w.err.zero(s); }
    for (int q = 0; q < ns; ++q) eg[q].P = w.islabs.p + dg.off[ns - 1 - q];
    tc_gemm_exact(TcOperand(As, M, ld, ld), TcOperand(Bs, Np, ld, ld), M, eg, ns, w.err.p, s, PROF_TC_SLICE);
    // bytes: every int32 split sum read once, the output written once
    ProfScope pa(PROF_OZ_ACCUM, 4.0 * splits * (double)M * (double)Np + out_bytes(o, M, Np), s);
    if (o.complex_out) launch_output<false, true>(ns, splits, s, w.islabs.p, dg, M, Np, A.expo.p, B.expo.p, o);
    else launch_output<false, false>(ns, splits, s, w.islabs.p, dg, M, Np, A.expo.p, B.expo.p, o);
    return;
  }
  // bytes of int32 split sums at a time (half the bound above)
  const long long slab_budget = (long long)std::max(1.0, std::min(2.0 * (1LL << 30), 0.5 * slab_bytes));
  const int max_splits = dg.zs[ns - 1];   // of the longest diagonal
  long long nc = std::max<long long>(1, slab_budget / (4LL * M * max_splits));
  nc = std::min<long long>(Np, std::max<long long>(256, nc / 256 * 256));
  if (o.complex_out) nc = Np;
  w.islabs.alloc((size_t)max_splits * M * nc);
  w.acc.alloc((size_t)M * nc);
  if (w.err.n == 0) { w.err.alloc(1); w.err.zero(s); }
  for (long long n0 = 0; n0 < Np; n0 += nc) {
    const long long nn = std::min(nc, Np - n0);
    OzOut oc = o;
    if (!o.complex_out) oc.out = o.out + n0;
    for (int d = 0; d < ns; ++d) {
      TcExactGroup g = eg[ns - 1 - d];
      g.N = nn; g.ldp = nn; g.split_stride = M * nn;   // oz_accumulate_kernel's layout
      g.P = w.islabs.p;
      tc_gemm_exact(TcOperand(As, M, ld, ld), TcOperand(Bs + n0 * ld, nn, ld, ld), M, &g, 1, w.err.p, s, PROF_TC_SLICE);
      const int zeff = g.zs();
      const double scale = ldexp(1.0, -o.bits * d);
      const int first = d == 0 ? 1 : 0;
      const int mode = d < ns - 1 ? 0 : (o.complex_out ? 2 : 1);
      const long long elements = mode == 2 ? M * (nn / 2) : M * nn;
      const bool warp = elements < 152LL * 256 && zeff > 8;
      const int grid = warp ? (int)std::min<long long>(std::max<long long>((elements * 32 + 255) / 256, 1), 152LL * 32)
                            : grid_for(elements);
      const bool small = M * nn < (1LL << 32);
      const int* eb = B.expo.p + n0;
      // bytes: the split sums read, the FP64 accumulator read (after the first diagonal) and written (or,
      // on the last diagonal, the output written)
      ProfScope pa(PROF_OZ_ACCUM, 4.0 * zeff * (double)M * (double)nn + (first ? 0.0 : 8.0 * (double)M * (double)nn) +
                                      (mode == 0 ? 8.0 * (double)M * (double)nn : out_bytes(oc, M, nn)), s);
      if (mode == 0) {
        if (warp) launch_accumulate<true, 0>(small, grid, s, w.islabs.p, zeff, M, nn, scale, first, w.acc.p, A.expo.p, eb, oc);
        else launch_accumulate<false, 0>(small, grid, s, w.islabs.p, zeff, M, nn, scale, first, w.acc.p, A.expo.p, eb, oc);
      } else if (mode == 1) {
        if (warp) launch_accumulate<true, 1>(small, grid, s, w.islabs.p, zeff, M, nn, scale, first, w.acc.p, A.expo.p, eb, oc);
        else launch_accumulate<false, 1>(small, grid, s, w.islabs.p, zeff, M, nn, scale, first, w.acc.p, A.expo.p, eb, oc);
      } else {
        if (warp) launch_accumulate<true, 2>(small, grid, s, w.islabs.p, zeff, M, nn, scale, first, w.acc.p, A.expo.p, eb, oc);
        else launch_accumulate<false, 2>(small, grid, s, w.islabs.p, zeff, M, nn, scale, first, w.acc.p, A.expo.p, eb, oc);
      }
      GFCC_LAUNCH_CHECK();
    }
  }
}

// The products of the stacked form (A slice i against B slices 0..ns-1-i, longest first) and the bytes of their
// int32 partials.
void stack_groups(long long M, long long Np, long long kp, int ns, TcExactGroup (&eg)[OZ_SLICES_MAX], OzParts& st,
                  double& bytes) {
  long long Ns[OZ_SLICES_MAX], ks[OZ_SLICES_MAX], off = 0;
  for (int i = 0; i < ns; ++i) {
    Ns[i] = (ns - i) * Np;
    ks[i] = kp;
  }
  const int nk_split = tc_exact_nk_split(M, Ns, ks, ns);
  for (int i = 0; i < ns; ++i) {
    eg[i].kA = (long long)i * kp;
    eg[i].kB = 0;
    eg[i].k_pad = kp;
    const long long ld4 = (Ns[i] + 3) / 4 * 4;   // rows of partials start on 16 bytes (vector epilogue stores)
    eg[i].N = Ns[i]; eg[i].ldp = ld4; eg[i].split_stride = M * ld4;
    eg[i].nk_split = nk_split;
    st.off[i] = off;
    st.ncol[i] = ld4;
    st.zs[i] = eg[i].zs();
    off += (long long)st.zs[i] * M * ld4;
  }
  bytes = 4.0 * (double)off;
}
// The stacked form pays when the A rows saved from re-reading, ns(ns-1)/2 kp f16 per row, outweigh the
// extra partial sums it writes and reads back, about the same count times Np int32 per split, and its
// partials fit in 4 GB.
bool use_stacked(long long M, long long Np, long long kp, int ns) {
  TcExactGroup eg[OZ_SLICES_MAX];
  OzParts st;
  double bytes;
  stack_groups(M, Np, kp, ns, eg, st, bytes);
  return kp >= 4LL * Np * st.zs[0] && bytes <= oz_slab_bytes();
}
// Exact complex product in the stacked form: A sliced row-major (normal order), Bsm sliced slot-major
// (normal order) with Np = 2N rows per slot.
void oz_run_stacked(const SlicedRows& A, const SlicedRows& Bsm, long long M, long long Np, const OzOut& o,
                    OzWork& w, cudaStream_t s) {
  const int ns = A.ns;
  const long long kp = A.kp, ld = (long long)ns * kp;
  TcExactGroup eg[OZ_SLICES_MAX];
  OzParts st;
  double bytes;
  stack_groups(M, Np, kp, ns, eg, st, bytes);
  w.islabs.alloc((size_t)(bytes / 4.0));
  if (w.err.n == 0) { w.err.alloc(1); w.err.zero(s); }
  int splits = 0;
  double part_bytes = 0.0;
  for (int i = 0; i < ns; ++i) {
    eg[i].P = w.islabs.p + st.off[i];
    splits += st.zs[i];
    part_bytes += 4.0 * st.zs[i] * (double)M * (double)st.ncol[i];
  }
  tc_gemm_exact(TcOperand(reinterpret_cast<const __half*>(A.slices.p), M, ld, ld),
                TcOperand(reinterpret_cast<const __half*>(Bsm.slices.p), ns * Np, kp, kp), M, eg, ns, w.err.p, s,
                PROF_TC_SLICE);
  ProfScope pa(PROF_OZ_ACCUM, part_bytes + out_bytes(o, M, Np), s);
  launch_output<true, true>(ns, splits, s, w.islabs.p, st, M, Np, A.expo.p, Bsm.expo.p, o);
}
}  // namespace

double oz_slab_bytes() {
  double v = 4.0 * (1LL << 30);
  if (const char* env = getenv("GFCC_OZ_SLAB_BYTES")) v = atof(env);
  return v;
}

double oz_min_macs() {
  // a complex multiply-add is four FP64 ones: 1.6e7 of them keep the FP64 pipe busy for 0.13 ms at best
  double v = 1.6e7;
  if (const char* env = getenv("GFCC_OZ_MIN_MACS")) v = atof(env);
  return v;
}

namespace {
struct ZSliceCache {   // slices of a left operand kept for several products with it
  SlicedRows sa;
  bool valid = false;
  const cplx* A = nullptr;   // the operand they were made from (checked on reuse)
  long long M = 0, K = 0, sam = 0, sak = 0;
  int ns = 0, bits = 0;
  bool conjA = false;
};
struct ZWork {          // buffers of zgemm_oz, kept between calls (grow-only)
  SlicedRows sa, sb;
  DBuf<unsigned long long> mxa, mxb;
  OzWork w;
  ZSliceCache cache[2];
};
}  // namespace

void* zgemm_work(gfcc_ctx* c) {
  if (!c->zwork) c->zwork = new ZWork();
  return c->zwork;
}
void* zgemm_slice_cache(gfcc_ctx* c, int i) {
  GFCC_CHECK(i == 0 || i == 1, GFCC_ERR_ARG, "zgemm_slice_cache: index");
  return &static_cast<ZWork*>(zgemm_work(c))->cache[i];
}
void zgemm_slice_cache_reset(void* cache) { static_cast<ZSliceCache*>(cache)->valid = false; }
void zgemm_work_free(gfcc_ctx* c) {
  delete static_cast<ZWork*>(c->zwork);
  c->zwork = nullptr;
}

bool zgemm_oz_fits(const ZGemmDesc& g, int ns) {
  const double kp = (double)tc_pad_k(TcKind::F16, 2LL * g.K), out = 2.0 * (double)g.M * (double)g.N;
  const double sums = 4.0 * ns * out;   // one split of every diagonal; beyond the limit, of one diagonal and its FP64 sum
  const double need = 2.0 * ns * kp * ((double)g.M + 2.0 * g.N) + (sums <= oz_slab_bytes() ? sums : 12.0 * out);
  if (need <= (double)(1LL << 30)) return true;
  double have = (double)device_free_bytes();
  if (g.work) {
    const ZWork& z = *static_cast<const ZWork*>(g.work);
    have += (double)(z.sa.slices.n + z.sb.slices.n) + 4.0 * (double)z.w.islabs.n + 8.0 * (double)z.w.acc.n;
  }
  return need <= 0.25 * have;
}

void zgemm_oz(const ZGemmDesc& g, int ns, cudaStream_t s, int bits) {
  const long long M = g.M, N = g.N, K = g.K;
  GFCC_CHECK(g.batch == 1, GFCC_ERR_ARG, "zgemm_oz: no batches");
  GFCC_CHECK(ns >= 2 && ns <= OZ_SLICES_MAX, GFCC_ERR_ARG, "zgemm_oz: 2..7 slices");
  GFCC_CHECK(bits == OZ_BITS || (bits == OZ_BITS_MOR && ns == OZ_SLICES_MOR), GFCC_ERR_ARG, "zgemm_oz: digits");
  if (M <= 0 || N <= 0) return;
  ProfScope prof(PROF_OZ_ZGEMM, 8.0 * (double)M * (double)N * (double)K, s);
  ZWork local;
  ZWork& z = g.work ? *static_cast<ZWork*>(g.work) : local;
  ZSliceCache* cache = static_cast<ZSliceCache*>(g.a_cache);
  const bool reuse = cache && cache->valid && cache->A == g.A && cache->M == M && cache->K == K &&
                     cache->sam == g.sam && cache->sak == g.sak && cache->ns == ns && cache->bits == bits &&
                     cache->conjA == g.conjA;
  SlicedRows& sa = cache ? cache->sa : z.sa;
  SlicedRows& sb = z.sb;
  sa.rows = M; sa.kp = tc_pad_k(TcKind::BF16, 2 * K); sa.ns = ns; sa.reversed = false;
  const bool stacked = use_stacked(M, 2 * N, sa.kp, ns);
  sb.rows = 2 * N; sb.kp = sa.kp; sb.ns = ns; sb.reversed = !stacked;
  if (!reuse) {
    sa.slices.alloc(sizeof(__half) * M * ns * sa.kp);
    sa.expo.alloc(M);
  }
  sb.slices.alloc(sizeof(__half) * 2 * N * ns * sb.kp);
  sb.expo.alloc(2 * N);
  {
    // bytes: each complex operand read once and its slices written once (A only when not cached)
    const double sb_bytes = 16.0 * (double)N * (double)K + 2.0 * (double)(2 * N) * ns * (double)sb.kp;
    const double sa_bytes = reuse ? 0.0 : 16.0 * (double)M * (double)K + 2.0 * (double)M * ns * (double)sa.kp;
    ProfScope ps(PROF_OZ_SLICE, sa_bytes + sb_bytes, s);
    DBuf<unsigned long long>& mxa = z.mxa;
    DBuf<unsigned long long>& mxb = z.mxb;
    mxa.alloc(M);
    mxb.alloc(N);
    GFCC_CUDA(cudaMemsetAsync(mxa.p, 0, sizeof(unsigned long long) * M, s));
    GFCC_CUDA(cudaMemsetAsync(mxb.p, 0, sizeof(unsigned long long) * N, s));
    const long long kt = (sa.kp / 2 + ZT_K - 1) / ZT_K;   // k tiles covering the padded width
    const long long kt_in = (K + ZT_K - 1) / ZT_K;
    // row tiles on grid.y, which ends at 65535 (2,097,120 rows): the blocks walk what is beyond
    const unsigned rtA = (unsigned)std::min<long long>((M + ZT_R - 1) / ZT_R, 65535);
    const unsigned rtB = (unsigned)std::min<long long>((N + ZT_R - 1) / ZT_R, 65535);
    // A(m, k) = A[m sam + k sak]; B rows n: B(k, n) = B[k sbk + n sbn] -> r = n, s_r = sbn, s_k = sbk
    if (!reuse) {
      zrowmax_kernel<<<dim3((unsigned)kt_in, rtA), 256, 0, s>>>(g.A, g.sam, g.sak, M, K, mxa.p);
      GFCC_LAUNCH_CHECK();
    }
    zrowmax_kernel<<<dim3((unsigned)kt_in, rtB), 256, 0, s>>>(g.B, g.sbn, g.sbk, N, K, mxb.p);
    GFCC_LAUNCH_CHECK();
    if (!reuse) {
      with_digits(ns, bits, [&](auto NSc, auto Bc) {
        const dim3 grid((unsigned)kt, rtA);
        zslice_kernel<decltype(NSc)::value, decltype(Bc)::value><<<grid, 256, 0, s>>>(
            g.A, g.sam, g.sak, g.conjA ? 1 : 0, M, K, 0, mxa.p, sa.kp, 0,
            reinterpret_cast<__half*>(sa.slices.p), sa.expo.p);
      });
      GFCC_LAUNCH_CHECK();
      if (cache) {
        cache->valid = true;
        cache->A = g.A; cache->M = M; cache->K = K; cache->sam = g.sam; cache->sak = g.sak;
        cache->ns = ns; cache->bits = bits; cache->conjA = g.conjA;
      }
    }
    with_digits(ns, bits, [&](auto NSc, auto Bc) {
      const dim3 grid((unsigned)kt, rtB);
      zslice_kernel<decltype(NSc)::value, decltype(Bc)::value><<<grid, 256, 0, s>>>(
          g.B, g.sbn, g.sbk, g.conjB ? 1 : 0, N, K, 1, mxb.p, sb.kp, stacked ? 0 : 1,
          reinterpret_cast<__half*>(sb.slices.p), sb.expo.p, stacked ? 1 : 0);
    });
    GFCC_LAUNCH_CHECK();
  }
  OzOut o;
  o.complex_out = true;
  o.C = g.C;
  o.scm = g.scm;
  o.scn = g.scn;
  o.alpha = g.alpha;
  o.cbeta = g.beta;
  o.bits = bits;
  o.set_kinds();
  OzWork& w = z.w;
  if (stacked) oz_run_stacked(sa, sb, M, 2 * N, o, w, s);
  else oz_run(sa, sb, M, 2 * N, o, w, s);
  if (g.work) return;   // the caller checks the workspace's error flag (zgemm_work_check) later
  int herr = 0;
  GFCC_CUDA(cudaMemcpyAsync(&herr, w.err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  GFCC_CUDA(cudaStreamSynchronize(s));
  GFCC_CHECK(herr == 0, GFCC_ERR_CUDA, "zgemm_oz: tensor-core pipeline wait timed out");
}

void zgemm_work_check(gfcc_ctx* c) {
  if (!c->zwork) return;
  ZWork* z = static_cast<ZWork*>(c->zwork);
  if (z->w.err.n == 0) return;
  int herr = 0;
  GFCC_CUDA(cudaMemcpyAsync(&herr, z->w.err.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  GFCC_CUDA(cudaStreamSynchronize(c->stream));
  GFCC_CHECK(herr == 0, GFCC_ERR_CUDA, "exact-slice GEMM: tensor-core pipeline wait timed out");
}

void oz_slice_into(const double* X, long long ldx, long long nrows, long long K, SlicedRows& out, long long row0,
                   cudaStream_t s) {
  GFCC_CHECK(row0 >= 0 && row0 + nrows <= out.rows && K <= out.kp, GFCC_ERR_ARG, "oz_slice_into: out of range");
  if (nrows == 0) return;
  // bytes: the FP64 rows read once, their slices written once
  ProfScope prof(PROF_OZ_SLICE, 8.0 * (double)nrows * (double)K + 2.0 * (double)nrows * out.ns * (double)out.kp, s);
  __half* o = reinterpret_cast<__half*>(out.slices.p) + row0 * out.ns * out.kp;
  if (out.kp <= 2048) {   // short rows: a warp per row
    with_ns(out.ns, [&](auto NSc) {
      slice_rows_warp_kernel<decltype(NSc)::value><<<(unsigned)((nrows * 32 + 255) / 256), 256, 0, s>>>(
          X, ldx, nrows, K, out.kp, out.reversed ? 1 : 0, o, out.expo.p + row0);
    });
  } else if (nrows < 152LL * 4 && nrows <= 65535) {   // few long rows: split each row over blocks
    DBuf<unsigned long long> mx;
    mx.alloc(nrows);
    mx.zero(s);
    const long long chunks_in = (K + SL_CH - 1) / SL_CH, chunks = (out.kp + SL_CH - 1) / SL_CH;
    rowmax_chunk_kernel<<<dim3((unsigned)std::max<long long>(chunks_in, 1), (unsigned)nrows), 256, 0, s>>>(X, ldx, K,
                                                                                                         mx.p);
    GFCC_LAUNCH_CHECK();
    with_ns(out.ns, [&](auto NSc) {
      slice_chunk_kernel<decltype(NSc)::value><<<dim3((unsigned)chunks, (unsigned)nrows), 256, 0, s>>>(
          X, ldx, K, out.kp, out.reversed ? 1 : 0, mx.p, o, out.expo.p + row0);
    });
    GFCC_LAUNCH_CHECK();
    GFCC_CUDA(cudaStreamSynchronize(s));   // mx is released on return
    return;
  } else {
    const int grid = (int)std::min<long long>(nrows, 152LL * 16);
    with_ns(out.ns, [&](auto NSc) {
      slice_kernel<decltype(NSc)::value><<<grid, 256, 0, s>>>(X, ldx, nrows, K, out.kp, out.reversed ? 1 : 0, o,
                                                             out.expo.p + row0);
    });
  }
  GFCC_LAUNCH_CHECK();
}

void oz_slice(const double* X, long long ldx, long long rows, long long K, bool reversed, SlicedRows& out,
              cudaStream_t s, int ns) {
  GFCC_CHECK(ns >= 2 && ns <= OZ_SLICES_MAX, GFCC_ERR_ARG, "oz_slice: 2..7 slices");
  out.rows = rows;
  out.kp = tc_pad_k(TcKind::BF16, K);
  out.ns = ns;
  out.reversed = reversed;
  out.slices.alloc(sizeof(__half) * std::max<long long>(rows, 1) * ns * out.kp);
  out.expo.alloc(std::max<long long>(rows, 1));
  oz_slice_into(X, ldx, rows, K, out, 0, s);
}

void oz_gemm(const SlicedRows& A, const SlicedRows& B, long long M, long long N, double* out, long long ldo,
             double beta, OzWork& w, cudaStream_t s, double alpha) {
  if (M <= 0 || N <= 0) return;
  GFCC_CHECK(!A.reversed && B.reversed && A.kp == B.kp && A.ns == B.ns, GFCC_ERR_ARG,
             "oz_gemm: operand slicing mismatch");
  GFCC_CHECK(A.rows >= M && B.rows >= N, GFCC_ERR_ARG, "oz_gemm: operand rows");
  OzOut o;
  o.out = out;
  o.ldo = ldo;
  o.beta = beta;
  o.alpha = make_cuDoubleComplex(alpha, 0.0);
  o.set_kinds();
  oz_run(A, B, M, N, o, w, s);
}

}  // namespace gfcc

// Dense-tensor helpers for the one-time H-bar build: strided permutation and a two-operand
// contraction (permute -> FP64 GEMM -> permute-accumulate) driven by index labels.
#include "gfcc_internal.cuh"
#include "tensor.h"
#include "ozaki.cuh"

#include <algorithm>
#include <cstdlib>
#include <map>

namespace gfcc {
namespace {

struct PermArgs {
  int nd;
  long long dst_dims[6];
  long long src_stride[6];   // stride in src of the source axis placed at dst position k
  long long total;
  double alpha, beta;
};

__device__ __forceinline__ void perm_store(double* d, double v, double alpha, double beta) {
  v *= alpha;
  *d = (beta == 0.0) ? v : v + beta * *d;
}
// source offset of the leading n axes at linear index t (row-major over them), 32-bit arithmetic when it fits
template <typename I>
__device__ __forceinline__ long long perm_offset(const PermArgs& a, int n, long long t) {
  I rem = (I)t;
  long long off = 0;
#pragma unroll
  for (int k = 5; k >= 0; --k) {
    if (k >= n) continue;
    const I d = (I)a.dst_dims[k], q = rem / d;
    off += (long long)(rem - q * d) * a.src_stride[k];
    rem = q;
  }
  return off;
}
template <typename I>
__global__ void permute_kernel(const double* __restrict__ src, double* __restrict__ dst, PermArgs a) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < a.total;
       t += (long long)gridDim.x * blockDim.x)
    perm_store(dst + t, src[perm_offset<I>(a, a.nd, t)], a.alpha, a.beta);
}
// The last axis is contiguous in both: a warp per row, the index arithmetic once per row instead of per element.
__global__ void __launch_bounds__(256) permute_rows_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                                           PermArgs a) {
  const int n = (int)a.dst_dims[a.nd - 1], lane = threadIdx.x & 31;
  const long long rows = a.total / n;
  for (long long r = (blockIdx.x * 256LL + threadIdx.x) >> 5; r < rows; r += gridDim.x * 8LL) {
    const double* s = src + perm_offset<long long>(a, a.nd - 1, r);
    double* d = dst + r * n;
#pragma unroll 4
    for (int k = lane; k < n; k += 32) perm_store(d + k, s[k], a.alpha, a.beta);
  }
}
// The source's contiguous axis is dst axis q, not the last: 32 x 32 tiles of (q, last) through shared memory, so
// that both sides move along their contiguous axis; the other axes are the batch (blocks walk the tiles).
__global__ void __launch_bounds__(256) permute_tiles_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                                            PermArgs a, int q, long long tiles, int tq, int tn) {
  __shared__ double tile[32][33];
  const int nq = (int)a.dst_dims[q], n = (int)a.dst_dims[a.nd - 1];
  const long long sn = a.src_stride[a.nd - 1];
  long long dq = 1;   // dst stride of axis q
  for (int k = q + 1; k < a.nd; ++k) dq *= a.dst_dims[k];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    long long rem = t / ((long long)tq * tn);
    const int w = (int)(t - rem * tq * tn), q0 = w / tn * 32, n0 = w % tn * 32;
    long long so = 0, doff = 0, dstr = n;
    for (int k = a.nd - 2; k >= 0; --k) {   // the batch axes
      if (k != q) {
        const long long d = a.dst_dims[k], i = rem % d;
        rem /= d;
        so += i * a.src_stride[k];
        doff += i * dstr;
      }
      dstr *= a.dst_dims[k];
    }
#pragma unroll
    for (int h = 0; h < 4; ++h)
      if (const int r = y + 8 * h; q0 + x < nq && n0 + r < n) tile[r][x] = src[so + (q0 + x) + (long long)(n0 + r) * sn];
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 4; ++h)
      if (const int r = y + 8 * h; q0 + r < nq && n0 + x < n) perm_store(dst + doff + (q0 + r) * dq + n0 + x, tile[x][r], a.alpha, a.beta);
    __syncthreads();
  }
}

__global__ void axpby_kernel(long long n, double alpha, const double* __restrict__ x, double beta,
                             double* __restrict__ y) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    y[t] = alpha * x[t] + (beta == 0.0 ? 0.0 : beta * y[t]);
}

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)std::min<long long>(std::max<long long>(g, 1), 152LL * 32);
}

}  // namespace

void permute(const double* src, const int* dims, int nd, const int* perm, double* dst, double alpha,
             double beta, cudaStream_t s) {
  GFCC_CHECK(nd >= 1 && nd <= 6, GFCC_ERR_ARG, "permute: 1..6 dims");
  long long stride[6];
  stride[nd - 1] = 1;
  for (int k = nd - 2; k >= 0; --k) stride[k] = stride[k + 1] * dims[k + 1];
  PermArgs a{};
  a.nd = nd;
  a.total = 1;
  for (int k = 0; k < nd; ++k) {
    a.dst_dims[k] = dims[perm[k]];
    a.src_stride[k] = stride[perm[k]];
    a.total *= dims[perm[k]];
  }
  a.alpha = alpha;
  a.beta = beta;
  if (a.total == 0) return;
  // axes that stay neighbours are one axis
  for (int k = 0; k + 1 < a.nd;) {
    if (a.dst_dims[k + 1] == 1 || a.dst_dims[k] == 1 || a.src_stride[k] == a.dst_dims[k + 1] * a.src_stride[k + 1]) {
      const bool keep = a.dst_dims[k + 1] == 1;   // a unit axis disappears, whichever side it is on
      const long long st = keep ? a.src_stride[k] : a.src_stride[k + 1];
      a.dst_dims[k] *= a.dst_dims[k + 1];
      a.src_stride[k] = st;
      for (int j = k + 1; j + 1 < a.nd; ++j) {
        a.dst_dims[j] = a.dst_dims[j + 1];
        a.src_stride[j] = a.src_stride[j + 1];
      }
      --a.nd;
    } else {
      ++k;
    }
  }
  // Rows and tiles read and write whole lines with an index computation per row or tile; the element-wise kernel
  // computes one per element (61 M elements of a 4-index tensor: 283 us; they are 150 us of HBM time).
  const int last = a.nd - 1;
  int q = -1;
  for (int k = 0; k < a.nd; ++k)
    if (a.src_stride[k] == 1 && a.dst_dims[k] > 1) q = k;
  constexpr long long kInt = 0x7fffffffLL;
  if (a.nd == 1 && a.src_stride[0] == 1) {   // a copy
    axpby(a.total, alpha, src, beta, dst, s);
    return;
  }
  if (q == last && a.dst_dims[last] >= 32 && a.dst_dims[last] <= kInt && a.total / a.dst_dims[last] >= 2048) {
    const long long rows = a.total / a.dst_dims[last];
    permute_rows_kernel<<<(unsigned)std::min<long long>((rows + 7) / 8, 152LL * 32), 256, 0, s>>>(src, dst, a);
  } else if (q >= 0 && q < last && a.dst_dims[q] >= 8 && a.dst_dims[last] >= 8 && a.dst_dims[q] <= kInt &&
             a.dst_dims[last] <= kInt) {
    const long long tq = (a.dst_dims[q] + 31) / 32, tn = (a.dst_dims[last] + 31) / 32;
    const long long tiles = a.total / (a.dst_dims[q] * a.dst_dims[last]) * tq * tn;
    permute_tiles_kernel<<<(unsigned)std::min<long long>(tiles, 152LL * 16), 256, 0, s>>>(src, dst, a, q, tiles, (int)tq,
                                                                                         (int)tn);
  } else if (a.total < (1LL << 32)) {
    permute_kernel<unsigned><<<grid_for(a.total), 256, 0, s>>>(src, dst, a);
  } else {
    permute_kernel<unsigned long long><<<grid_for(a.total), 256, 0, s>>>(src, dst, a);
  }
  GFCC_LAUNCH_CHECK();
}

void axpby(long long n, double alpha, const double* x, double beta, double* y, cudaStream_t s) {
  if (n <= 0) return;
  axpby_kernel<<<grid_for(n), 256, 0, s>>>(n, alpha, x, beta, y);
  GFCC_LAUNCH_CHECK();
}

// ---------------------------------------------------------------------------------------------
Tensor::Tensor(std::string l, std::vector<int> d) : labels(std::move(l)), dims(std::move(d)) {
  GFCC_CHECK(labels.size() == dims.size(), GFCC_ERR_ARG, "tensor labels/dims mismatch");
  buf.alloc(size());
}
long long Tensor::size() const {
  long long n = 1;
  for (int d : dims) n *= d;
  return n;
}
TV Tensor::as(const std::string& l) const {
  GFCC_CHECK(l.size() == dims.size(), GFCC_ERR_ARG, "tensor relabel: rank mismatch");
  return TV{buf.p, l, dims};
}

void contract(double alpha, const TV& A, const TV& B, double beta, const TV& C, cudaStream_t s, double packed) {
  const std::string &la = A.l, &lb = B.l, &lc = C.l;
  std::map<char, int> size;
  auto reg = [&](const std::string& l, const std::vector<int>& d) {
    GFCC_CHECK(l.size() == d.size(), GFCC_ERR_ARG, "contract: labels/dims mismatch");
    for (size_t k = 0; k < l.size(); ++k) {
      auto it = size.find(l[k]);
      GFCC_CHECK(it == size.end() || it->second == d[k], GFCC_ERR_ARG,
                 std::string("contract: size clash on label ") + l[k]);
      size[l[k]] = d[k];
    }
  };
  reg(la, A.d); reg(lb, B.d); reg(lc, C.d);
  std::string Ml, Nl, Kl;
  for (char ch : la) {
    bool inB = lb.find(ch) != std::string::npos, inC = lc.find(ch) != std::string::npos;
    GFCC_CHECK(!(inB && inC), GFCC_ERR_ARG, "contract: batch labels unsupported");
    GFCC_CHECK(inB || inC, GFCC_ERR_ARG, "contract: dangling label in A");
    if (inC) Ml += ch; else Kl += ch;
  }
  for (char ch : lb) {
    bool inA = la.find(ch) != std::string::npos, inC = lc.find(ch) != std::string::npos;
    GFCC_CHECK(inA || inC, GFCC_ERR_ARG, "contract: dangling label in B");
    if (!inA) Nl += ch;
  }
  GFCC_CHECK(Ml.size() + Nl.size() == lc.size(), GFCC_ERR_ARG, "contract: output labels");
  long long M = 1, N = 1, K = 1;
  for (char ch : Ml) M *= size[ch];
  for (char ch : Nl) N *= size[ch];
  for (char ch : Kl) K *= size[ch];

  auto perm_of = [&](const std::string& from, const std::string& to) {
    std::vector<int> p;
    for (char ch : to) p.push_back((int)from.find(ch));
    return p;
  };
  auto identity = [](const std::vector<int>& p) {
    for (size_t k = 0; k < p.size(); ++k)
      if (p[k] != (int)k) return false;
    return true;
  };
  DBuf<double> Ap, Bp, Cp;
  std::string lt0 = Ml + Nl;
  std::vector<int> pc0 = perm_of(lt0, lc);
  // contractions above this many multiply-adds use the tensor cores (GFCC_OZ_MIN_MACS overrides it,
  // which the tests use to exercise this path at small sizes). The digits keep 62 bits below a row's largest element:
  // closer to 64 bits than FP64 sums where a row is of one magnitude, but an element more than 2^9 below its row's
  // largest keeps fewer than its 53 bits, and small operators, whose contractions are all below this, stay free of that.
  // A sum over packed pairs counts with the multiply-adds of the sum it stands for: it had the digits before it was
  // packed, with 55 bits. (A line at 3e7 gains about 3 % of the whole method at o = 30, v = 130, and 12 % of the gradient
  // at o = 19, v = 67.)
  double min_macs = 5e8;
  if (const char* env = getenv("GFCC_OZ_MIN_MACS")) min_macs = atof(env);
  if (packed * (double)M * (double)N * (double)K >= min_macs && M >= 16 && N >= 16) {
    // FP64-accurate GEMM from exact f16 slices on the tensor cores (7 slices: FP64-level accuracy)
    const double* Aop2 = A.p;
    std::vector<int> pa2 = perm_of(la, Ml + Kl);
    if (!identity(pa2)) {
      Ap.alloc(M * K);
      permute(A.p, A.d.data(), (int)A.d.size(), pa2.data(), Ap.p, 1.0, 0.0, s);
      Aop2 = Ap.p;
    }
    const double* Bop2 = B.p;
    std::vector<int> pb2 = perm_of(lb, Nl + Kl);   // K-major rows for the tensor cores
    if (!identity(pb2)) {
      Bp.alloc(K * N);
      permute(B.p, B.d.data(), (int)B.d.size(), pb2.data(), Bp.p, 1.0, 0.0, s);
      Bop2 = Bp.p;
    }
    SlicedRows sa, sb;
    oz_slice(Aop2, K, M, K, false, sa, s, OZ_SLICES_MAX);
    oz_slice(Bop2, K, N, K, true, sb, s, OZ_SLICES_MAX);
    Ap.release();
    Bp.release();
    OzWork w;
    if (identity(pc0)) {   // straight into C
      oz_gemm(sa, sb, M, N, C.p, N, beta, w, s, alpha);
    } else {
      Cp.alloc(M * N);
      oz_gemm(sa, sb, M, N, Cp.p, N, 0.0, w, s);
      std::vector<int> dt;
      for (char ch : lt0) dt.push_back(size[ch]);
      permute(Cp.p, dt.data(), (int)dt.size(), pc0.data(), C.p, alpha, beta, s);
    }
    int herr = 0;
    GFCC_CUDA(cudaMemcpyAsync(&herr, w.err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    GFCC_CUDA(cudaStreamSynchronize(s));
    GFCC_CHECK(herr == 0, GFCC_ERR_CUDA, "contract: tensor-core pipeline wait timed out");
    return;
  }
  const double* Aop = A.p;
  std::vector<int> pa = perm_of(la, Ml + Kl);
  if (!identity(pa)) {
    Ap.alloc(M * K);
    permute(A.p, A.d.data(), (int)A.d.size(), pa.data(), Ap.p, 1.0, 0.0, s);
    Aop = Ap.p;
  }
  const double* Bop = B.p;
  std::vector<int> pb = perm_of(lb, Kl + Nl);
  if (!identity(pb)) {
    Bp.alloc(K * N);
    permute(B.p, B.d.data(), (int)B.d.size(), pb.data(), Bp.p, 1.0, 0.0, s);
    Bop = Bp.p;
  }
  std::string lt = Ml + Nl;
  std::vector<int> pc = perm_of(lt, lc);
  GFCC_CHECK(M < (1LL << 31) && N < (1LL << 31) && K < (1LL << 31), GFCC_ERR_ARG, "contract: too big");
  // Few tiles and K of some hundreds: short splits keep the SMs at work. A packed sum is half as long as the one it stands
  // for and has fewer tiles (400 x 45 x 780 of o = 10, v = 40: 7 tiles, 805 us whole, 85 split; the unpacked
  // 400 x 100 x 1600 was in splits of 256 and took 281).
  constexpr int split_k = 64;
  if (identity(pc)) {
    dgemm_rm((int)M, (int)N, (int)K, alpha, Aop, (int)K, false, Bop, (int)N, false, beta, C.p, (int)N, s, split_k);
  } else {
    Cp.alloc(M * N);
    dgemm_rm((int)M, (int)N, (int)K, 1.0, Aop, (int)K, false, Bop, (int)N, false, 0.0, Cp.p, (int)N, s, split_k);
    std::vector<int> dt;
    for (char ch : lt) dt.push_back(size[ch]);
    permute(Cp.p, dt.data(), (int)dt.size(), pc.data(), C.p, alpha, beta, s);
  }
  // temporaries are released when they leave scope: the stream must be done with them first
  GFCC_CUDA(cudaStreamSynchronize(s));
}

void perm(const TV& src, double alpha, double beta, const TV& dst, cudaStream_t s) {
  GFCC_CHECK(src.l.size() == dst.l.size(), GFCC_ERR_ARG, "perm: rank mismatch");
  std::vector<int> p;
  for (size_t k = 0; k < dst.l.size(); ++k) {
    size_t j = src.l.find(dst.l[k]);
    GFCC_CHECK(j != std::string::npos, GFCC_ERR_ARG, "perm: label missing");
    GFCC_CHECK(src.d[j] == dst.d[k], GFCC_ERR_ARG, "perm: size clash");
    p.push_back((int)j);
  }
  permute(src.p, src.d.data(), (int)src.d.size(), p.data(), dst.p, alpha, beta, s);
}

}  // namespace gfcc

// Orthonormalisation of the subspace iteration (App. D.2 step 2): Cholesky QR, G = Y^T Y = L L^T, Q = Y L^-T.
//
// gram_kernel       the lower tiles of G in fp64, the long sum over Y's rows cut into slices (added in a fixed order)
// cholesky_kernel   L^-T in fp64 by one cluster of CTAs, rounded to fp32
// gemm_f32          Q = Y L^-T, with the products exact to fp32 (conversion_gemm.cu)
// For a basis of 512 columns of length 8064: 0.24 + 1.86 + 0.74 ms in the form this one replaced (whole G, one block for the
// factor, a triangular solve per row), now 0.13 + 0.22 + 0.03.
#include "conversion.cuh"
#include "common.cuh"

namespace transmla {
namespace conv {

namespace {

// ------------------------------------------------------------------------------------------------ Gram matrix
// 128 x 128 tile, 256 threads x (8 x 8) fp64 sums, 16 rows of Y a step through two shared-memory buffers, converted to fp64
// on the way in.  Bound by the fp64 units: 64 multiply-adds a thread and step against eight 16-byte reads.
constexpr int GT = 128, GK = 16;
constexpr int kGramSmem = 2 * 2 * GK * GT * 8;

struct GramRegs { float4 v[2]; };
__device__ __forceinline__ void gram_fetch(GramRegs& t, const float* Y, bool vec, int r, int c0, int k0, int k_end, int tid) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int f = tid + 256 * u, k = k0 + f / 32, c = c0 + (f % 32) * 4;
    float x[4] = {0.f, 0.f, 0.f, 0.f};
    if (k < k_end) {
      const float* src = Y + static_cast<size_t>(k) * r + c;
      if (vec && c + 3 < r) { const float4 q = *reinterpret_cast<const float4*>(src); x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w; }
      else {
#pragma unroll
        for (int i = 0; i < 4; ++i) if (c + i < r) x[i] = src[i];
      }
    }
    t.v[u] = make_float4(x[0], x[1], x[2], x[3]);
  }
}
__device__ __forceinline__ void gram_stash(const GramRegs& t, double* S, int tid) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int f = tid + 256 * u;
    double2* d = reinterpret_cast<double2*>(S + (f / 32) * GT + (f % 32) * 4);
    d[0] = make_double2(t.v[u].x, t.v[u].y);
    d[1] = make_double2(t.v[u].z, t.v[u].w);
  }
}

__global__ void __launch_bounds__(256) gram_kernel(const float* Y, int m, int r, int ks, double* partial) {
  extern __shared__ __align__(16) unsigned char gram_smem[];
  double* As = reinterpret_cast<double*>(gram_smem);   // [2][GK][GT]
  double* Bs = As + 2 * GK * GT;
  int ti = 0, tj = blockIdx.x;
  while (tj > ti) tj -= ++ti;
  const int i0 = ti * GT, j0 = tj * GT, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const bool diag = ti == tj, vec = (r & 3) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
  const int k_lo = blockIdx.y * ks, k_hi = min(m, k_lo + ks);
  double acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
  GramRegs ra, rb;
  auto fetch = [&](int k) {
    gram_fetch(ra, Y, vec, r, i0, k, k_hi, tid);
    if (!diag) gram_fetch(rb, Y, vec, r, j0, k, k_hi, tid);
  };
  auto stash = [&](int buf) {
    gram_stash(ra, As + buf * GK * GT, tid);
    if (!diag) gram_stash(rb, Bs + buf * GK * GT, tid);
  };
  fetch(k_lo);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (int k = k_lo; k < k_hi; k += GK, buf ^= 1) {
    const bool more = k + GK < k_hi;
    if (more) fetch(k + GK);
    const double* a_s = As + buf * GK * GT;
    const double* b_s = diag ? a_s : Bs + buf * GK * GT;
#pragma unroll 4
    for (int kk = 0; kk < GK; ++kk) {
      double a[8], b[8];
#pragma unroll
      for (int h = 0; h < 4; ++h) {  // pairs of columns, 32 apart: consecutive lanes read consecutive pairs
        const double2 a2 = *reinterpret_cast<const double2*>(a_s + kk * GT + h * 32 + ty * 2);
        const double2 b2 = *reinterpret_cast<const double2*>(b_s + kk * GT + h * 32 + tx * 2);
        a[2 * h] = a2.x; a[2 * h + 1] = a2.y;
        b[2 * h] = b2.x; b[2 * h + 1] = b2.y;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
  }
  double* out = partial + static_cast<size_t>(blockIdx.y) * r * r;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = i0 + ty * 2 + (i & 1) + (i >> 1) * 32;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int col = j0 + tx * 2 + (j & 1) + (j >> 1) * 32;
      if (row < r && col <= row) out[static_cast<size_t>(row) * r + col] = acc[i][j];
    }
  }
}

__global__ void sum_slices_kernel(const double* part, int r, int slices, double* out) {
  const int row = blockIdx.y, col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col > row) return;
  const size_t e = static_cast<size_t>(row) * r + col, count = static_cast<size_t>(r) * r;
  double s = 0.0;
  for (int i = 0; i < slices; ++i) s += part[i * count + e];
  out[e] = s;
}

// ------------------------------------------------------------------------------------------------ Cholesky factor
// Right-looking blocked factorisation in blocks of 32, with the rows of an identity carried along below G: what the
// factorisation does to them makes them X = L^-T (X L^T = I).  One cluster; per panel p, with P(.,p) the finished columns
//   all CTAs   D = G(p,p) - P(p,p-1) P(p,p-1)^T, factored and inverted by warp 0 of each (the same bits everywhere, which
//              saves a meeting), while warps 1-7 apply panel p-1 to the rest: first to this CTA's blocks of column p, then to
//              its share of the blocks behind column p
//   each CTA   P(R,p) = B(R,p) L(p,p)^-T for its blocks R of column p: G rows below p, and X rows up to p
// and one cluster barrier.  What bounds it is the chain of r square roots and the updates between them, about 300 cycles
// each, with the fp64 units beside it: a block's product takes one SM's units 1000 cycles, and a panel has about 100 of them.
// (A device that cannot hold 16 such CTAs in a cluster gets 8, 4, .. of them: what it holds at once is asked.)
// At r = 512: 359 us by 8 CTAs with the own blocks one a warp, 221 us by 16 (the cluster's size limit with the opt-in), four
// rows of a block a warp and whole lines moved.  Rows and columns beyond r behave as an identity.
constexpr int NB = 32, kCluster = kOrthCluster, kCholThreads = 256, kPitch = NB + 1, kBlock = NB * kPitch;
constexpr int kMaxBlocks = 1024 / NB, kMaxOwn = kMaxBlocks / kCluster;
// doubles: D, W, P(p,p-1), col[2][32], the CTA's blocks of column p, two operands for each of warps 1-7
constexpr int kCholSmem = (3 * kBlock + 2 * NB + kMaxOwn * kBlock + 14 * kBlock) * 8;
static_assert(kCholSmem <= 232448, "shared memory budget");

struct CholView {
  double* G;   // [r, r], lower
  double* X;   // [r, r], upper
  int r, n;    // n block rows of each
  bool even;   // pairs of elements are aligned
  __device__ __forceinline__ bool next(int c, int j) const { return c * NB + j + 1 < r; }
  // element (i, j) of block (R, c): R < n rows of G, otherwise rows of X
  __device__ __forceinline__ double* at(int R, int c, int i, int j, bool& in) const {
    const int row = (R < n ? R : R - n) * NB + i, col = c * NB + j;
    in = row < r && col < r;
    return (R < n ? G : X) + static_cast<size_t>(row) * r + col;
  }
};
// A warp copies block (R, c) to shared memory (pitch 33).
__device__ __forceinline__ void load_block(const CholView& v, int R, int c, double* dst, int lane) {
  double x[NB];  // all on their way before the first is stored
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    bool in;
    const double* p = v.at(R, c, i, lane, in);
    x[i] = in ? __ldcg(p) : 0.0;
  }
#pragma unroll
  for (int i = 0; i < NB; ++i) dst[i * kPitch + lane] = x[i];
}
// A lane's elements of a product: rows l/8 + 4i for i from `from`, columns 2 (l%8) + {0, 1} + 16h: eight lanes move one line.
template <int kRows>
__device__ __forceinline__ void load_elements(const CholView& v, int R, int c, int from, double (&x)[kRows][4], int lane) {
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bool in;
      const double* p = v.at(R, c, (lane >> 3) + 4 * (from + i), 2 * (lane & 7) + 16 * h, in);
      double2 e = make_double2(0.0, 0.0);
      if (in && v.even) e = __ldcg(reinterpret_cast<const double2*>(p));  // an even order has both or neither
      else if (in) { e.x = __ldcg(p); if (v.next(c, 2 * (lane & 7) + 16 * h)) e.y = __ldcg(p + 1); }
      x[i][2 * h] = e.x;
      x[i][2 * h + 1] = e.y;
    }
  }
}
template <int kRows>
__device__ __forceinline__ void store_elements(const CholView& v, int R, int c, const double (&x)[kRows][4], int lane) {
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bool in;
      double* p = v.at(R, c, (lane >> 3) + 4 * i, 2 * (lane & 7) + 16 * h, in);
      if (in && v.even) __stcg(reinterpret_cast<double2*>(p), make_double2(x[i][2 * h], x[i][2 * h + 1]));
      else if (in) { __stcg(p, x[i][2 * h]); if (v.next(c, 2 * (lane & 7) + 16 * h)) __stcg(p + 1, x[i][2 * h + 1]); }
    }
  }
}
// acc -= A B^T at the lane's elements; A's first row is that of acc's
template <int kRows>
__device__ __forceinline__ void warp_product(double (&acc)[kRows][4], const double* A, const double* B, int lane) {
  const double* ar = A + (lane >> 3) * kPitch;
  const double* br = B + 2 * (lane & 7) * kPitch;
#pragma unroll 4
  for (int k = 0; k < NB; ++k) {
    double a[kRows], b[4];
#pragma unroll
    for (int i = 0; i < kRows; ++i) a[i] = ar[4 * i * kPitch + k];
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = br[((j & 1) + 16 * (j >> 1)) * kPitch + k];
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fma(-a[i], b[j], acc[i][j]);
  }
}
__global__ void __launch_bounds__(kCholThreads, 1)
cholesky_kernel(double* G, double* X, int r, float* X32, int diagonal, int32_t* dev_status) {
  extern __shared__ __align__(16) double cs[];
  double* D = cs;                     // the panel's diagonal block
  double* W = D + kBlock;             // L(p,p)^-T
  double* Pp = W + kBlock;            // P(p,p-1)
  double* col = Pp + kBlock;          // [2][32]
  double* Bs = col + 2 * NB;          // [kMaxOwn] blocks of column p
  double* ops = Bs + kMaxOwn * kBlock;  // [7][2]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x, ctas = gridDim.x;
  const CholView v = {G, X, r, (r + NB - 1) / NB, (r & 1) == 0};
  const int n = v.n;
  double* opA = ops + (warp - 1) * 2 * kBlock;  // warps 1-7
  double* opB = opA + kBlock;
  bool bad = false;

  // The blocks of column p of this CTA: list entry e is G row p + 1 + e, then X rows 0 .. p.  At most kMaxOwn at a time,
  // entries `first`, first + ctas ..: formed in Bs by warps 1-7, four rows a warp, then multiplied by W by all.
  auto form_blocks = [&](int p, int first) {
    for (int own = 0, e = first; own < kMaxOwn && e < n; e += ctas, ++own) {
      const int R = e < n - 1 - p ? p + 1 + e : n + e - (n - 1 - p), q = R - n;  // (q < 0 for G rows)
      double* B = Bs + own * kBlock;
      for (int slab = warp - 1; slab < NB / 4; slab += 7) {
        double acc[1][4] = {{0.0, 0.0, 0.0, 0.0}};
        const int row = 4 * slab + (lane >> 3);
        if (q == p) {  // nothing stored yet in X rows p - 1 (zeros) and p (the identity's block)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[0][j] = row == 2 * (lane & 7) + (j & 1) + 16 * (j >> 1) ? 1.0 : 0.0;
        } else {
          if (R < n || q < p - 1) load_elements(v, R, p, slab, acc, lane);
          if (p > 0) {
            double x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              bool in;
              const double* g = v.at(R, p - 1, 4 * slab + i, lane, in);
              x[i] = in ? __ldcg(g) : 0.0;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) opA[i * kPitch + lane] = x[i];
            __syncwarp();
            warp_product(acc, opA, Pp, lane);
            __syncwarp();
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) B[row * kPitch + 2 * (lane & 7) + (j & 1) + 16 * (j >> 1)] = acc[0][j];
      }
    }
  };
  // P(R,p) = B W.  W is an upper triangle: a warp's four columns need only the rows of W up to the last of them
  auto finish_blocks = [&](int p, int first) {
    const int lo = tid & 15, up = tid >> 4;
    for (int own = 0, e = first; own < kMaxOwn && e < n; e += ctas, ++own) {
      const int R = e < n - 1 - p ? p + 1 + e : n + e - (n - 1 - p);
      const double* B = Bs + own * kBlock;
      const double* b = B + lo * kPitch;
      const double* w = W + 2 * up;
      double o[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 4
      for (int k = 0; k < 4 * warp + 4; ++k) {
        const double b0 = b[k], b1 = b[16 * kPitch + k], w0 = w[k * kPitch], w1 = w[k * kPitch + 1];
        o[0][0] = fma(b0, w0, o[0][0]); o[0][1] = fma(b0, w1, o[0][1]);
        o[1][0] = fma(b1, w0, o[1][0]); o[1][1] = fma(b1, w1, o[1][1]);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          bool in;
          double* g = v.at(R, p, lo + 16 * i, 2 * up + j, in);
          if (in) __stcg(g, o[i][j]);
        }
    }
  };

  for (int p = 0; p < n; ++p) {
    // ---- D, by all warps: 4 elements a thread
    const int lo = tid & 15, up = tid >> 4;  // rows and columns lo, lo + 16, up, up + 16 of a block
    {
      double d[2][2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int a = up + 16 * i, b = lo + 16 * j;
          bool in;
          const double* g = v.at(p, p, max(a, b), min(a, b), in);
          d[i][j] = in ? __ldcg(g) : (a == b ? 1.0 : 0.0);
        }
      if (p > 0) {
        double x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          bool in;
          const double* g = v.at(p, p - 1, warp * 4 + i, lane, in);
          x[i] = in ? __ldcg(g) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) Pp[(warp * 4 + i) * kPitch + lane] = x[i];
        __syncthreads();
        const double* a = Pp + up * kPitch;
        const double* b = Pp + lo * kPitch;
#pragma unroll 8
        for (int k = 0; k < NB; ++k) {
          const double a0 = a[k], a1 = a[16 * kPitch + k], b0 = b[k], b1 = b[16 * kPitch + k];
          d[0][0] = fma(-a0, b0, d[0][0]); d[0][1] = fma(-a0, b1, d[0][1]);
          d[1][0] = fma(-a1, b0, d[1][0]); d[1][1] = fma(-a1, b1, d[1][1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) D[(up + 16 * i) * kPitch + lo + 16 * j] = d[i][j];
    }
    __syncthreads();
    if (warp == 0) {
      // ---- lane i holds row i of D and of the identity
      double a[NB], x[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) { a[j] = D[lane * kPitch + j]; x[j] = j == lane ? 1.0 : 0.0; }
      double pivot = a[0];
      const int left = r - p * NB;  // what is behind is an identity's already
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        if (k % 8 == 0 && k >= left) break;
        double d = __shfl_sync(0xffffffffu, pivot, k);
        if (!(d > 0.0)) { bad = true; d = 1.0; }
        const double inv = rsqrt(d);
        const double l = a[k] * inv;
        if (k + 1 < NB) pivot = fma(-l, l, a[k + 1]);  // in lane k + 1: the next step need not wait for the exchange
        x[k] *= inv;
        col[(k & 1) * NB + lane] = l;
        __syncwarp();
#pragma unroll
        for (int j = k + 1; j < NB; ++j) {
          const double lj = col[(k & 1) * NB + j];
          a[j] = fma(-l, lj, a[j]);
          x[j] = fma(-x[k], lj, x[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < NB; ++j) W[lane * kPitch + j] = x[j];
    } else {
      form_blocks(p, cta);
      // ---- panel p - 1 on the blocks behind column p: column j takes G rows j .. n-1 and X rows 0 .. p-1
      if (p > 0) {
        int t = cta * 7 + warp - 1;
        for (int j = p + 1; j < n; ++j) {
          const int count = n - j + p;
          for (; t < count; t += ctas * 7) {
            const int R = t < n - j ? j + t : n + t - (n - j);
            double acc[8][4] = {};
            if (R != n + p - 1) load_elements(v, R, j, 0, acc, lane);
            load_block(v, R, p - 1, opA, lane);
            load_block(v, j, p - 1, opB, lane);
            __syncwarp();
            warp_product(acc, opA, opB, lane);
            store_elements(v, R, j, acc, lane);
            __syncwarp();
          }
          t -= count;
        }
      }
    }
    __syncthreads();
    finish_blocks(p, cta);
    for (int first = cta + kMaxOwn * ctas; first < n; first += kMaxOwn * ctas) {  // (a cluster below its full size)
      __syncthreads();
      if (warp > 0) form_blocks(p, first);
      __syncthreads();
      finish_blocks(p, first);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  for (int e = cta * kCholThreads + tid; e < r * r; e += ctas * kCholThreads) {
    const int row = e / r, c = e % r;
    X32[e] = c < row || (c == row && !diagonal) ? 0.f : static_cast<float>(__ldcg(X + e));
  }
  if (bad && tid == 0 && cta == 0 && dev_status != nullptr) atomicOr(dev_status, TRANSMLA_DEV_NUMERIC);
}

// Q <- P + Q diag(X), in fp64 per element: the rest of the last pass (see cholesky_qr_last).
__global__ void __launch_bounds__(256) add_diagonal_kernel(const float* P, float* Q, int m, int r, const double* X) {
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= r) return;
  const double d = X[static_cast<size_t>(c) * r + c];
#pragma unroll 8
  for (int i = blockIdx.y; i < m; i += gridDim.y) {
    const size_t e = static_cast<size_t>(i) * r + c;
    Q[e] = static_cast<float>(fma(static_cast<double>(Q[e]), d, static_cast<double>(P[e])));
  }
}

}  // namespace

int gram_slices(int r) {  // slices of the sum over rows: what fills the device once
  const int t = (r + GT - 1) / GT, tiles = t * (t + 1) / 2;
  const int s = 148 / tiles;
  return s < 1 ? 1 : s > 16 ? 16 : s;
}

// X = L^-T of Y^T Y = L L^T, in fp64, and X32 in fp32, with its diagonal or without.
static cudaError_t inverse_factor(const float* Y, int m, int r, double* partial, double* G, double* X, float* X32, int diagonal,
                                  int most_ctas, int32_t* dev_status, cudaStream_t stream) {
  if (r > kMaxBlocks * NB) return cudaErrorInvalidValue;
  static PerDeviceFlag gram_set, chol_set;
  if (cudaError_t e = ensure_dynamic_smem(gram_kernel, kGramSmem, gram_set); e != cudaSuccess) return e;
  if (cudaError_t e = ensure_dynamic_smem(cholesky_kernel, kCholSmem, chol_set); e != cudaSuccess) return e;
  const int t = (r + GT - 1) / GT, slices = gram_slices(r);
  const int ks = ((m + slices - 1) / slices + GK - 1) / GK * GK;
  gram_kernel<<<dim3(t * (t + 1) / 2, slices), 256, kGramSmem, stream>>>(Y, m, r, ks, partial);
  sum_slices_kernel<<<dim3((r + 127) / 128, r), 128, 0, stream>>>(partial, r, slices, G);
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kCholThreads);
  cfg.dynamicSmemBytes = kCholSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // One cluster, of no more CTAs than a panel has blocks for, and no more than the device holds at once in a cluster.
  static PerDeviceFlag fits[kMaxBlocks];  // by size: 1 it does, -1 it does not, 0 not asked yet
  const int slot = current_device_slot();
  int ctas = 1;
  while (ctas < most_ctas && ctas < (r + NB - 1) / NB) ctas *= 2;
  for (; ctas > 1; ctas /= 2) {
    int known = slot >= 0 ? fits[ctas].value[slot].load(std::memory_order_acquire) : 0;
    if (known == 0) {
      int clusters = 0;
      cfg.gridDim = dim3(ctas);
      attr[0].val.clusterDim.x = ctas;
      if ((ctas > 8 && cudaFuncSetAttribute(cholesky_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
          cudaOccupancyMaxActiveClusters(&clusters, cholesky_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        clusters = 0;
      }
      known = clusters > 0 ? 1 : -1;
      if (slot >= 0) fits[ctas].value[slot].store(known, std::memory_order_release);
    }
    if (known > 0) break;
  }
  cfg.gridDim = dim3(ctas);
  attr[0].val.clusterDim.x = ctas;
  return cudaLaunchKernelEx(&cfg, cholesky_kernel, G, X, r, X32, diagonal, dev_status);
}

cudaError_t cholesky_qr(const float* Y, int m, int r, double* partial, double* G, double* X, float* X32, float* Q,
                        int32_t* dev_status, cudaStream_t stream, int most_ctas) {
  if (cudaError_t e = inverse_factor(Y, m, r, partial, G, X, X32, 1, most_ctas, dev_status, stream); e != cudaSuccess) return e;
  return gemm_f32(0, 0, m, r, r, 1.f, Y, r, 0, X32, r, 0, Q, r, 0, 1, dev_status, stream);
}

// A column of Q = Y X is its own diagonal product and little else, and a product through the split is up to 2^-23 short (the
// accumulator truncates): the columns came out 4.5e-8 short, all alike, which made Q^T Q differ from I by 9.5e-8 of sqrt(r)
// (a triangular solve: 6.1e-8).  So the diagonal is left out of the matrix product and added in fp64: 3.4e-8.
cudaError_t cholesky_qr_last(float* Q, int m, int r, double* partial, double* G, double* X, float* X32, float* P,
                             int32_t* dev_status, cudaStream_t stream, int most_ctas) {
  if (cudaError_t e = inverse_factor(Q, m, r, partial, G, X, X32, 0, most_ctas, dev_status, stream); e != cudaSuccess) return e;
  if (cudaError_t e = gemm_f32(0, 0, m, r, r, 1.f, Q, r, 0, X32, r, 0, P, r, 0, 1, dev_status, stream); e != cudaSuccess) return e;
  const int columns = (r + 255) / 256, rows = 1184 / columns;
  add_diagonal_kernel<<<dim3(columns, m < rows ? m : rows), 256, 0, stream>>>(P, Q, m, r, X);
  return cudaGetLastError();
}

}  // namespace conv
}  // namespace transmla

// Orthonormalisation of the subspace iteration (App. D.2 step 2): Cholesky QR, G = Y^T Y = L L^T, Q = Y L^-T.
//
// gram_kernel       the lower tiles of G in fp64, the long sum over Y's rows cut into slices (added in a fixed order)
// cholesky_kernel   L^-T in fp64 by one cluster of CTAs, rounded to fp32
// gemm_f32          Q = Y L^-T, with the products exact to fp32 (conversion_gemm.cu)
// For a basis of 512 columns of length 8064: 0.24 + 1.86 + 0.74 ms in the form this one replaced (whole G, one block for the
// factor, a triangular solve per row), now 0.13 + 0.36 + 0.03.
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
// each.  Rows and columns beyond r behave as an identity.
constexpr int NB = 32, kCluster = 8, kCholThreads = 256, kPitch = NB + 1, kBlock = NB * kPitch;
constexpr int kMaxBlocks = 1024 / NB, kMaxOwn = kMaxBlocks / kCluster;
// doubles: D, W, P(p,p-1), col[2][32], the CTA's blocks of column p, two operands for each of warps 1-7
constexpr int kCholSmem = (3 * kBlock + 2 * NB + kMaxOwn * kBlock + 14 * kBlock) * 8;
static_assert(kCholSmem <= 232448, "shared memory budget");

struct CholView {
  double* G;   // [r, r], lower
  double* X;   // [r, r], upper
  int r, n;    // n block rows of each
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
// The lane's elements of block (R, c), at the places of its elements of a product: rows l/4 + 8a, columns l%4 + 4b.
__device__ __forceinline__ void load_elements(const CholView& v, int R, int c, bool fresh, double (&x)[4][8], int lane) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      bool in;
      const double* p = v.at(R, c, (lane >> 2) + 8 * i, (lane & 3) + 4 * j, in);
      x[i][j] = in && !fresh ? __ldcg(p) : 0.0;
    }
  }
}
// acc[a][b] -= sum_k A[row][k] B[col][k] for the lane's rows l/4 + 8a and columns l%4 + 4b
__device__ __forceinline__ void warp_product(double (&acc)[4][8], const double* A, const double* B, int lane) {
  const double* ar = A + (lane >> 2) * kPitch;
  const double* br = B + (lane & 3) * kPitch;
#pragma unroll 4
  for (int k = 0; k < NB; ++k) {
    double a[4], b[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = ar[8 * i * kPitch + k];
#pragma unroll
    for (int j = 0; j < 8; ++j) b[j] = br[4 * j * kPitch + k];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = fma(-a[i], b[j], acc[i][j]);
  }
}
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kCholThreads, 1)
cholesky_kernel(double* G, double* X, int r, float* X32, int32_t* dev_status) {
  extern __shared__ __align__(16) double cs[];
  double* D = cs;                     // the panel's diagonal block
  double* W = D + kBlock;             // L(p,p)^-T
  double* Pp = W + kBlock;            // P(p,p-1)
  double* col = Pp + kBlock;          // [2][32]
  double* Bs = col + 2 * NB;          // [kMaxOwn] blocks of column p
  double* ops = Bs + kMaxOwn * kBlock;  // [7][2]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x;
  const CholView v = {G, X, r, (r + NB - 1) / NB};
  const int n = v.n;
  double* opA = ops + (warp - 1) * 2 * kBlock;  // warps 1-7
  double* opB = opA + kBlock;
  bool bad = false;

  for (int p = 0; p < n; ++p) {
    // ---- D, by all warps: 4 elements a thread
    if (p > 0) {
      if (warp == 0) load_block(v, p, p - 1, Pp, lane);
      __syncthreads();
    }
    for (int e = tid; e < NB * NB; e += kCholThreads) {
      const int i = e >> 5, j = e & 31, hi = max(i, j), lo = min(i, j);
      bool in;
      const double* g = v.at(p, p, hi, lo, in);
      double d = in ? __ldcg(g) : (i == j ? 1.0 : 0.0);
      if (p > 0) {
        double s = 0.0;
#pragma unroll 8
        for (int k = 0; k < NB; ++k) s = fma(Pp[i * kPitch + k], Pp[j * kPitch + k], s);
        d -= s;
      }
      D[i * kPitch + j] = d;
    }
    __syncthreads();
    if (warp == 0) {
      // ---- lane i holds row i of D and of the identity
      double a[NB], x[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) { a[j] = D[lane * kPitch + j]; x[j] = j == lane ? 1.0 : 0.0; }
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        double d = __shfl_sync(0xffffffffu, a[k], k);
        if (!(d > 0.0)) { bad = true; d = 1.0; }
        const double inv = rsqrt(d);
        const double l = a[k] * inv;
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
      // ---- this CTA's blocks of column p: list entry e is G row p + 1 + e, then X rows 0 .. p
      int own = 0;
      for (int e = cta; e < n; e += kCluster, ++own) {
        if (own % 7 != warp - 1) continue;
        const int R = e < n - 1 - p ? p + 1 + e : n + e - (n - 1 - p), q = R - n;  // (q < 0 for G rows)
        double* B = Bs + own * kBlock;
        double acc[4][8];
        // nothing stored yet in X rows p - 1 (zeros) and p (the identity's block)
        load_elements(v, R, p, R >= n && q >= p - 1, acc, lane);
        if (q == p) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = (lane >> 2) + 8 * i == (lane & 3) + 4 * j ? 1.0 : 0.0;
        } else if (p > 0) {
          load_block(v, R, p - 1, opA, lane);
          __syncwarp();
          warp_product(acc, opA, Pp, lane);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) B[((lane >> 2) + 8 * i) * kPitch + (lane & 3) + 4 * j] = acc[i][j];
        __syncwarp();
      }
      // ---- panel p - 1 on the blocks behind column p: column j takes G rows j .. n-1 and X rows 0 .. p-1
      if (p > 0) {
        int t = cta * 7 + warp - 1;
        for (int j = p + 1; j < n; ++j) {
          const int count = n - j + p;
          for (; t < count; t += kCluster * 7) {
            const int R = t < n - j ? j + t : n + t - (n - j);
            double acc[4][8];
            load_elements(v, R, j, R >= n && R - n == p - 1, acc, lane);
            load_block(v, R, p - 1, opA, lane);
            load_block(v, j, p - 1, opB, lane);
            __syncwarp();
            warp_product(acc, opA, opB, lane);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
              for (int jj = 0; jj < 8; ++jj) {
                bool in;
                double* g = v.at(R, j, (lane >> 2) + 8 * i, (lane & 3) + 4 * jj, in);
                if (in) __stcg(g, acc[i][jj]);
              }
            }
            __syncwarp();
          }
          t -= count;
        }
      }
    }
    __syncthreads();
    // ---- P(R,p) = B W: one warp a block, the product with W's columns as rows of its transpose
    {
      int own = 0;
      for (int e = cta; e < n; e += kCluster, ++own) {
        const int R = e < n - 1 - p ? p + 1 + e : n + e - (n - 1 - p);
        const double* B = Bs + own * kBlock;
        for (int o = tid; o < NB * NB; o += kCholThreads) {
          const int row = o >> 5, c = o & 31;
          double s = 0.0;
#pragma unroll 8
          for (int k = 0; k < NB; ++k) s = fma(B[row * kPitch + k], W[k * kPitch + c], s);
          bool in;
          double* g = v.at(R, p, row, c, in);
          if (in) __stcg(g, s);
        }
      }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  for (int e = cta * kCholThreads + tid; e < r * r; e += kCluster * kCholThreads) {
    const int row = e / r, c = e % r;
    X32[e] = c < row ? 0.f : static_cast<float>(__ldcg(X + e));
  }
  if (bad && tid == 0 && cta == 0 && dev_status != nullptr) atomicOr(dev_status, TRANSMLA_DEV_NUMERIC);
}

}  // namespace

int gram_slices(int r) {  // slices of the sum over rows: what fills the device once
  const int t = (r + GT - 1) / GT, tiles = t * (t + 1) / 2;
  const int s = 148 / tiles;
  return s < 1 ? 1 : s > 16 ? 16 : s;
}

cudaError_t cholesky_qr(const float* Y, int m, int r, double* partial, double* G, double* X, float* X32, float* Q,
                        int32_t* dev_status, cudaStream_t stream) {
  if (r > kMaxBlocks * NB) return cudaErrorInvalidValue;
  static PerDeviceFlag gram_set, chol_set;
  if (cudaError_t e = ensure_dynamic_smem(gram_kernel, kGramSmem, gram_set); e != cudaSuccess) return e;
  if (cudaError_t e = ensure_dynamic_smem(cholesky_kernel, kCholSmem, chol_set); e != cudaSuccess) return e;
  const int t = (r + GT - 1) / GT, slices = gram_slices(r);
  const int ks = ((m + slices - 1) / slices + GK - 1) / GK * GK;
  gram_kernel<<<dim3(t * (t + 1) / 2, slices), 256, kGramSmem, stream>>>(Y, m, r, ks, partial);
  sum_slices_kernel<<<dim3((r + 127) / 128, r), 128, 0, stream>>>(partial, r, slices, G);
  cholesky_kernel<<<kCluster, kCholThreads, kCholSmem, stream>>>(G, X, r, X32, dev_status);
  if (cudaError_t e = cudaGetLastError(); e != cudaSuccess) return e;
  return gemm_f32(0, 0, m, r, r, 1.f, Y, r, 0, X32, r, 0, Q, r, 0, 1, stream);
}

}  // namespace conv
}  // namespace transmla

// Orthonormalisation of the subspace iteration (App. D.2 step 2): Cholesky QR, G = Y^T Y = L L^T, Q = Y L^-T.
//
// gram_kernel       the lower tiles of G in fp64, the long sum over Y's rows cut into slices (added in a fixed order)
// cholesky_kernel   L^-T in fp64 by one cluster of CTAs, rounded to fp32
// gemm_f32          Q = Y L^-T, with the products exact to fp32 (conversion_gemm.cu)
// For a basis of 512 columns of length 8064: 0.24 + 1.86 + 0.74 ms in the form this one replaced (whole G, one block for the
// factor, a triangular solve per row), now 0.10 + 0.14 + 0.03.
#include <type_traits>

#include "common.cuh"
#include "conversion.cuh"

namespace transmla {
namespace conv {

namespace {

// c += a b for 8 x 8 x 4: lane l has a(l/4, l%4), b(l%4, l/4) and c(l/4, 2 (l%4) + {0, 1}).
__device__ __forceinline__ void mma_f64(double2& c, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c.x), "+d"(c.y) : "d"(a), "d"(b));
}

// ------------------------------------------------------------------------------------------------ Gram matrix
// 128 x 128 tile, eight warps with 64 x 32 fp64 sums each, 16 rows of Y a step through two shared-memory buffers, converted to
// fp64 on the way in.  Bound by the fp64 units: tensor instructions run at their rate (64 multiply-adds a cycle and SM) and leave
// the issue slots to the loads and conversions, which multiply-adds of single threads compete with.  8064 x 512: 124 -> 100 us.
constexpr int GT = 128, GK = 16, GP = GT + 4;  // pitch: conflict-free fragments
constexpr int kGramSmem = 2 * 2 * GK * GP * 8;

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
    double2* d = reinterpret_cast<double2*>(S + (f / 32) * GP + (f % 32) * 4);
    d[0] = make_double2(t.v[u].x, t.v[u].y);
    d[1] = make_double2(t.v[u].z, t.v[u].w);
  }
}

__global__ void __launch_bounds__(256) gram_kernel(const float* Y, int m, int r, int ks, double* partial) {
  extern __shared__ __align__(16) unsigned char gram_smem[];
  double* As = reinterpret_cast<double*>(gram_smem);   // [2][GK][GP]
  double* Bs = As + 2 * GK * GP;
  int ti = 0, tj = blockIdx.x;
  while (tj > ti) tj -= ++ti;
  const int i0 = ti * GT, j0 = tj * GT, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lr = lane >> 2, lc = lane & 3;
  const int mi = (warp >> 2) * 64, nj = (warp & 3) * 32;  // the warp's rows and columns of the tile
  const bool diag = ti == tj, vec = (r & 3) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
  const int k_lo = blockIdx.y * ks, k_hi = min(m, k_lo + ks);
  double2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_double2(0.0, 0.0);
  GramRegs ra, rb;
  auto fetch = [&](int k) {
    gram_fetch(ra, Y, vec, r, i0, k, k_hi, tid);
    if (!diag) gram_fetch(rb, Y, vec, r, j0, k, k_hi, tid);
  };
  auto stash = [&](int buf) {
    gram_stash(ra, As + buf * GK * GP, tid);
    if (!diag) gram_stash(rb, Bs + buf * GK * GP, tid);
  };
  fetch(k_lo);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (int k = k_lo; k < k_hi; k += GK, buf ^= 1) {
    const bool more = k + GK < k_hi;
    if (more) fetch(k + GK);
    const double* a_s = As + buf * GK * GP + mi + lr;
    const double* b_s = (diag ? As : Bs) + buf * GK * GP + nj + lr;
#pragma unroll
    for (int k4 = 0; k4 < GK; k4 += 4) {
      double a[8], b[4];
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = a_s[(k4 + lc) * GP + 8 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = b_s[(k4 + lc) * GP + 8 * j];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_f64(acc[i][j], a[i], b[j]);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
  }
  double* out = partial + static_cast<size_t>(blockIdx.y) * r * r;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = i0 + mi + 8 * i + lr;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = j0 + nj + 8 * j + 2 * lc;
      if (row < r && col <= row) out[static_cast<size_t>(row) * r + col] = acc[i][j].x;
      if (row < r && col + 1 <= row) out[static_cast<size_t>(row) * r + col + 1] = acc[i][j].y;
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
//   all CTAs   D = G(p,p) - P(p,p-1) P(p,p-1)^T, factored by warp 0 of each and inverted by warp 4 (the same bits everywhere, which
//              saves a meeting), while the others apply panel p-1 to the rest: first to this CTA's blocks of column p, then to
//              its share of the blocks behind column p
//   each CTA   P(R,p) = B(R,p) L(p,p)^-T for its blocks R of column p: G rows below p, and X rows up to p
// and one cluster barrier.  What bounds it is the chain of r square roots with the steps between them, and a panel's round trips to
// L2: D's operands, the barrier.  The products are fp64 tensor instructions (at the fp64 units' rate, with a sixth of the
// instructions), a block's operands are asked for at the start of the panel, and the factor takes four columns a step.
// (A device that cannot hold 16 such CTAs in a cluster gets 8, 4, .. of them: what it holds at once is asked.)
// Rows and columns beyond r behave as an identity.
// At r = 512, cycles a panel: 26 000 with one column a step (12 000 in the factor, beside multiply-adds of 16 000 in warps of the same
// quarter of the SM), now 15 500 (D 1900, factor 8900, P 1500, barrier 2000 and more); 218 -> 136 us.
constexpr int NB = 32, kCluster = kOrthCluster, kCholThreads = 384, kPitch = NB + 4, kBlock = NB * kPitch;  // (conflict-free fragments)
constexpr int kMaxBlocks = 1024 / NB, kMaxOwn = kMaxBlocks / kCluster, kStep = 16 + 4 * NB, kExchange = 16 + NB / 4 * kStep;
// Warps with a part in the products: not those of the factor's quarter of the SM, which has its fp64 units alone.  The first
// kFormers form a block of column p and come last where the blocks behind it are shared out.
constexpr int kWorkers = 9, kFormers = 4;
// doubles: D, W, P(p,p-1), the factor's exchange, the CTA's blocks of column p, two operands for each worker
constexpr int kCholSmem = (3 * kBlock + kExchange + kMaxOwn * kBlock + 2 * kWorkers * kBlock) * 8;
static_assert(kCholSmem <= 232448, "shared memory budget");

struct CholView {
  double* G;   // [r, r], lower
  double* X;   // [r, r], upper
  int r, n;    // n block rows of each
  bool even;   // pairs of elements are aligned, and both inside or both outside
  // element (i, j) of block (R, c): R < n rows of G, otherwise rows of X
  __device__ __forceinline__ double* at(int R, int c, int i, int j, bool& in) const {
    const int row = (R < n ? R : R - n) * NB + i, col = c * NB + j;
    in = row < r && col < r;
    return (R < n ? G : X) + static_cast<size_t>(row) * r + col;
  }
  __device__ __forceinline__ double load(int R, int c, int i, int j) const {
    bool in;
    const double* p = at(R, c, i, j, in);
    return in ? __ldcg(p) : 0.0;
  }
  // elements (i, j) and (i, j + 1), j even
  __device__ __forceinline__ double2 load2(int R, int c, int i, int j) const {
    bool in;
    const double* p = at(R, c, i, j, in);
    double2 e = make_double2(0.0, 0.0);
    if (in && even) e = __ldcg(reinterpret_cast<const double2*>(p));
    else if (in) { e.x = __ldcg(p); if (c * NB + j + 1 < r) e.y = __ldcg(p + 1); }
    return e;
  }
  __device__ __forceinline__ void store2(int R, int c, int i, int j, double2 e) const {
    bool in;
    double* p = at(R, c, i, j, in);
    if (in && even) __stcg(reinterpret_cast<double2*>(p), e);
    else if (in) { __stcg(p, e.x); if (c * NB + j + 1 < r) __stcg(p + 1, e.y); }
  }
};
// A warp asks for block (R, c) in shared memory; the caller waits (cp_async_wait, __syncwarp).
__device__ __forceinline__ void fetch_block(const CholView& v, int R, int c, double* dst, int lane) {
  if (v.even) {
#pragma unroll
    for (int u = 0; u < NB / 2; ++u) {  // 16 lanes a row
      const int i = 2 * u + (lane >> 4), j = 2 * (lane & 15);
      bool in;
      const double* p = v.at(R, c, i, j, in);
      cp_async16(dst + i * kPitch + j, in ? p : v.G, in ? 16 : 0);
    }
    cp_async_commit();
  } else {
#pragma unroll 8
    for (int i = 0; i < NB; ++i) dst[i * kPitch + lane] = v.load(R, c, i, lane);
  }
}
// 1 / sqrt(d): the approximation of PTX (2^-20 off at most over all exponents, as measured), then one step of Householder's
// method of third order, y + y e (1/2 + 3/8 e) with e = 1 - d y^2: what is left is of the order of e^3, below 2^-56, and the
// result's error the roundings', below 2^-52 (the test's bound; CUDA's rsqrt is within 2^-52 too, and with it two rounds of the iteration at
// 8064 x 512 take 2090 us instead of 1970).  No branches, so that the steps around it overlap.  A pivot that is not positive (zero, NaN) is bad and counts as 1.
// An infinite one gives NaN, which a later pivot or the next pass meets; subnormal ones, which the approximation flushes, do not come
// from fp32 data.  (Tests for both here: the iteration at 2048 x 256 646 -> 658 us.)
__device__ __forceinline__ double root_approximation(double d) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  return y;
}
__device__ __forceinline__ double inverse_root(double d, bool& bad) {
  if (!(d > 0.0)) { bad = true; d = 1.0; }
  const double y = root_approximation(d), e = fma(-d * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__global__ void inverse_root_kernel(const double* d, int n, double* out, int32_t* dev_status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  bool bad = false;
  out[3 * i] = inverse_root(d[i], bad);
  out[3 * i + 1] = rsqrt(d[i]);
  out[3 * i + 2] = root_approximation(d[i]);
  if (bad) atomicOr(dev_status, TRANSMLA_DEV_NUMERIC);
}
// Two warps: D = L L^T and W = L^-T, four columns a step.  Lane i of the first holds row i of D; it factors each step's 4 x 4
// block (every lane, redundantly), hands the finished columns over and goes on, waiting for nobody.  Lane i of the second holds row i
// of the identity and follows a step behind.  A step's share of the exchange: l10 l20 l30 l21 l31 l32 of its block and the
// inverse roots of its diagonal, then the finished columns [32][4].
// left: rows that are there, what is behind is an identity's already.
__device__ __forceinline__ void step_done(int step) { asm volatile("bar.arrive %0, 64;" ::"r"(1 + step) : "memory"); }
__device__ __forceinline__ void step_wait(int step) { asm volatile("bar.sync %0, 64;" ::"r"(1 + step) : "memory"); }
// v, one row, times the inverse of the block's L^T
template <int k>
__device__ __forceinline__ void solve_row(double (&v)[NB], const double (&l)[6], const double (&inv)[4]) {
  v[k] *= inv[0];
  v[k + 1] = fma(-v[k], l[0], v[k + 1]) * inv[1];
  v[k + 2] = fma(-v[k + 1], l[3], fma(-v[k], l[1], v[k + 2])) * inv[2];
  v[k + 3] = fma(-v[k + 2], l[5], fma(-v[k + 1], l[4], fma(-v[k], l[2], v[k + 3]))) * inv[3];
}
template <int k>
__device__ __forceinline__ void update_row(double (&v)[NB], const double* done) {
#pragma unroll
  for (int j = k + 4; j < NB; ++j) {
    const double2 u = *reinterpret_cast<const double2*>(done + j * 4), w = *reinterpret_cast<const double2*>(done + j * 4 + 2);
    v[j] = fma(-v[k + 3], w.y, fma(-v[k + 2], w.x, fma(-v[k + 1], u.y, fma(-v[k], u.x, v[j]))));
  }
}
template <class Columns>
__device__ __forceinline__ void all_steps(Columns columns, int left) {
  columns(std::integral_constant<int, 0>());
  columns(std::integral_constant<int, 4>());
  if (left <= 8) return;
  columns(std::integral_constant<int, 8>());
  columns(std::integral_constant<int, 12>());
  if (left <= 16) return;
  columns(std::integral_constant<int, 16>());
  columns(std::integral_constant<int, 20>());
  if (left <= 24) return;
  columns(std::integral_constant<int, 24>());
  columns(std::integral_constant<int, 28>());
}
__device__ __forceinline__ void factor_block(const double* D, double* diag, double* exchange, int left, bool& bad) {
  const int lane = threadIdx.x & 31;
  double a[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) a[j] = D[lane * kPitch + j];
  all_steps([&](auto first) {
    constexpr int k = decltype(first)::value;
    double* out = exchange + k / 4 * kStep;
    if (lane >= k && lane < k + 4) {
      double2* d = reinterpret_cast<double2*>(diag + (lane - k) * 4);
      d[0] = make_double2(a[k], a[k + 1]);
      d[1] = make_double2(a[k + 2], a[k + 3]);
    }
    __syncwarp();
    double l[6], inv[4];
    inv[0] = inverse_root(diag[0], bad);
    l[0] = diag[4] * inv[0]; l[1] = diag[8] * inv[0]; l[2] = diag[12] * inv[0];
    inv[1] = inverse_root(fma(-l[0], l[0], diag[5]), bad);
    l[3] = fma(-l[1], l[0], diag[9]) * inv[1]; l[4] = fma(-l[2], l[0], diag[13]) * inv[1];
    inv[2] = inverse_root(fma(-l[3], l[3], fma(-l[1], l[1], diag[10])), bad);
    l[5] = fma(-l[4], l[3], fma(-l[2], l[1], diag[14])) * inv[2];
    inv[3] = inverse_root(fma(-l[5], l[5], fma(-l[4], l[4], fma(-l[2], l[2], diag[15]))), bad);
    solve_row<k>(a, l, inv);
    double2* mine = reinterpret_cast<double2*>(out + 16 + lane * 4);
    mine[0] = make_double2(a[k], a[k + 1]);
    mine[1] = make_double2(a[k + 2], a[k + 3]);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < 6; ++i) out[i] = l[i];
#pragma unroll
      for (int i = 0; i < 4; ++i) out[6 + i] = inv[i];
    }
    __syncwarp();
    step_done(k / 4);
    update_row<k>(a, out + 16);
  }, left);
}
__device__ __forceinline__ void inverse_block(double* W, const double* exchange, int left) {
  const int lane = threadIdx.x & 31;
  double x[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) x[j] = j == lane ? 1.0 : 0.0;
  all_steps([&](auto first) {
    constexpr int k = decltype(first)::value;
    const double* in = exchange + k / 4 * kStep;
    step_wait(k / 4);
    double l[6], inv[4];
#pragma unroll
    for (int i = 0; i < 6; ++i) l[i] = in[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) inv[i] = in[6 + i];
    solve_row<k>(x, l, inv);
    update_row<k>(x, in + 16);
  }, left);
#pragma unroll
  for (int j = 0; j < NB; ++j) W[lane * kPitch + j] = x[j];
}

__global__ void __launch_bounds__(kCholThreads, 1)
cholesky_kernel(double* G, double* X, int r, float* X32, int diagonal, int32_t* dev_status) {
  extern __shared__ __align__(16) double cs[];
  double* D = cs;                     // the panel's diagonal block
  double* W = D + kBlock;             // L(p,p)^-T
  double* Pp = W + kBlock;            // P(p,p-1)
  double* exchange = Pp + kBlock;
  double* Bs = exchange + kExchange;  // [kMaxOwn] blocks of column p
  double* ops = Bs + kMaxOwn * kBlock;  // [kWorkers][2]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x, ctas = gridDim.x;
  const int lr = lane >> 2, lc = lane & 3;
  const CholView v = {G, X, r, (r + NB - 1) / NB, (r & 1) == 0};
  const int n = v.n;
  const int worker = (warp & 3) == 0 ? -1 : (warp >> 2) * 3 + (warp & 3) - 1;  // -1: warps 0, 4 and (without work) 8
  double* opA = ops + worker * 2 * kBlock;
  double* opB = opA + kBlock;
  bool bad = false;

  // The blocks of column p of this CTA: list entry e is G row p + 1 + e, then X rows 0 .. p.  At most kMaxOwn at a time,
  // entries `first`, first + ctas ..: formed in Bs by the workers, eight rows a warp, then multiplied by W by all.
  auto entry = [&](int p, int e) { return e < n - 1 - p ? p + 1 + e : n + e - (n - 1 - p); };
  auto form_blocks = [&](int p, int first) {
    for (int item = worker; item < kMaxOwn * 4; item += kWorkers) {
      const int own = item >> 2, row = (item & 3) * 8 + lr, e = first + own * ctas;
      if (e >= n) break;
      const int R = entry(p, e), q = R - n;  // (q < 0 for G rows)
      double2 acc[4];
      double a[8];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = 8 * t + 2 * lc;
        acc[t] = make_double2(0.0, 0.0);  // nothing stored yet in X rows p - 1 (zeros) and p (the identity's block)
        if (q == p) acc[t] = make_double2(row == j ? 1.0 : 0.0, row == j + 1 ? 1.0 : 0.0);
        else if (R < n || q < p - 1) acc[t] = v.load2(R, p, row, j);
      }
      if (p > 0 && q != p) {
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = -v.load(R, p - 1, row, 4 * k + lc);
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
          for (int t = 0; t < 4; ++t) mma_f64(acc[t], a[k], Pp[(8 * t + lr) * kPitch + 4 * k + lc]);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) *reinterpret_cast<double2*>(Bs + own * kBlock + row * kPitch + 8 * t + 2 * lc) = acc[t];
    }
  };
  // P(R,p) = B W, two 8 x 8 tiles a warp
  const int tr = (warp & 3) * 8, tc = (warp >> 2) * 16;  // (D's tiles of a warp too; of warps 0-7)
  auto finish_blocks = [&](int p, int first) {
    for (int own = 0, e = first; own < kMaxOwn && e < n && warp < 8; e += ctas, ++own) {
      const int R = entry(p, e);
      const double* B = Bs + own * kBlock;
      double2 o[2] = {};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const double b = B[(tr + lr) * kPitch + 4 * k + lc];
#pragma unroll
        for (int t = 0; t < 2; ++t) mma_f64(o[t], b, W[(4 * k + lc) * kPitch + tc + 8 * t + lr]);
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) v.store2(R, p, tr + lr, tc + 8 * t + 2 * lc, o[t]);
    }
  };

  for (int p = 0; p < n; ++p) {
    // ---- the warp's first block behind column p: column j takes G rows j .. n-1 and X rows 0 .. p-1
    int t = (worker >= kFormers ? worker - kFormers : worker + kWorkers - kFormers) * ctas + cta, j = p + 1, R = 0;
    auto settle = [&] {  // t, counted from column j's first block on, to a block of a column
      for (; j < n; ++j) {
        const int count = n - j + p;
        if (t < count) { R = t < n - j ? j + t : n + t - (n - j); return true; }
        t -= count;
      }
      return false;
    };
    double2 acc[4][4];
    auto ask = [&] {
      fetch_block(v, R, p - 1, opA, lane);
      fetch_block(v, j, p - 1, opB, lane);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[i][u] = R != n + p - 1 ? v.load2(R, j, 8 * i + lr, 8 * u + 2 * lc) : make_double2(0.0, 0.0);
    };
    // ---- D: two 8 x 8 tiles a warp
    double2 d[2] = {};
    if (warp < 8) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int a = tr + lr;
        auto element = [&](int b) {
          bool in;
          const double* g = v.at(p, p, max(a, b), min(a, b), in);
          return in ? __ldcg(g) : (a == b ? 1.0 : 0.0);
        };
        d[u] = make_double2(element(tc + 8 * u + 2 * lc), element(tc + 8 * u + 2 * lc + 1));
      }
      if (p > 0) {
        double x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = v.load(p, p - 1, warp * 4 + i, lane);
#pragma unroll
        for (int i = 0; i < 4; ++i) Pp[(warp * 4 + i) * kPitch + lane] = x[i];
      }
    }
    __syncthreads();
    if (warp < 8) {
      if (p > 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const double a = -Pp[(tr + lr) * kPitch + 4 * k + lc];
#pragma unroll
          for (int u = 0; u < 2; ++u) mma_f64(d[u], a, Pp[(tc + 8 * u + lr) * kPitch + 4 * k + lc]);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) *reinterpret_cast<double2*>(D + (tr + lr) * kPitch + tc + 8 * u + 2 * lc) = d[u];
    }
    __syncthreads();
    if (warp == 0) {
      factor_block(D, exchange, exchange + 16, r - p * NB, bad);
    } else if (warp == 4) {
      inverse_block(W, exchange + 16, r - p * NB);
    } else if (worker >= 0) {
      bool more = p > 0 && settle();
      if (more) ask();
      form_blocks(p, cta);
      // ---- panel p - 1 on the blocks behind column p
      while (more) {
        cp_async_wait<0>();
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          double a[4], b[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) { a[i] = -opA[(8 * i + lr) * kPitch + 4 * k + lc]; b[i] = opB[(8 * i + lr) * kPitch + 4 * k + lc]; }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int u = 0; u < 4; ++u) mma_f64(acc[i][u], a[i], b[u]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int u = 0; u < 4; ++u) v.store2(R, j, 8 * i + lr, 8 * u + 2 * lc, acc[i][u]);
        __syncwarp();
        t += ctas * kWorkers;
        more = settle();
        if (more) ask();
      }
    }
    __syncthreads();
    finish_blocks(p, cta);
    for (int first = cta + kMaxOwn * ctas; first < n; first += kMaxOwn * ctas) {  // (a cluster below its full size)
      __syncthreads();
      if (worker >= 0) form_blocks(p, first);
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

cudaError_t inverse_roots(const double* d, int n, double* out, int32_t* dev_status, cudaStream_t stream) {
  inverse_root_kernel<<<(n + 255) / 256, 256, 0, stream>>>(d, n, out, dev_status);
  return cudaGetLastError();
}

}  // namespace conv
}  // namespace transmla

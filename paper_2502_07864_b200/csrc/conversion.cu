// Kernels of the GQA -> MLA conversion on calibration activations (Sec. 4.2, 4.3; App. B, C, D): rotations, balancing and
// eigenvectors in fp32 arithmetic.  The matrix products are in conversion_gemm.cu, the orthonormalisation of the subspace
// iteration in conversion_qr.cu.
#include "conversion.cuh"
#include "common.cuh"

namespace transmla {
namespace conv {

// ------------------------------------------------------------------------------------------------ RoRoPE helpers
// Position in the merged key of segment entry i of group G (i = p*g + j: frequency G*fold + p, head j), real part.
__device__ __forceinline__ int seg_pos(int G, int i, int g, int d, int fold) {
  const int p = i / g, j = i - p * g;
  return j * d + 2 * (G * fold + p);
}

__global__ void gather_segments_kernel(const float* K, int n, int g, int d, int fold, float* seg) {
  const int m = g * fold, G = blockIdx.y;
  const size_t total = static_cast<size_t>(2) * n * m;
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(e % m);
    const size_t row = e / m;                       // 0..2n-1
    const int t = static_cast<int>(row % n), im = static_cast<int>(row / n);
    seg[static_cast<size_t>(G) * total + e] = K[static_cast<size_t>(t) * g * d + seg_pos(G, i, g, d, fold) + im];
  }
}

cudaError_t gather_segments(const float* K, int n, int g, int d, int fold, float* seg, cudaStream_t stream) {
  const int groups = d / 2 / fold;
  dim3 grid(296, groups);
  gather_segments_kernel<<<grid, 256, 0, stream>>>(K, n, g, d, fold, seg);
  return cudaGetLastError();
}

// Y[(q / fold, 2 (G fold + q % fold) + im), c] = sum_i U_G[i, q] X[seg_pos(G, i) + im, c]   (Eq. 18)
// U_G and some columns of X's rows in shared memory, a thread has 8 values of q x 4 columns: a block of order 128 has 64
// columns, one of order 64 has 128, .. of order 8 1024, so that no thread is without values of q.  Bound by the fp32 units (32
// multiply-adds a thread and step against three 16-byte reads), small orders by memory.  d = 128, C = 4096: g = 32, fold = 4
// 1.2 ms with one column a thread and X read again for every 8 q, now 180 us; g = 8, fold = 1 16.5 us, now 7.8 (43 with 64 columns
// a block whatever the order).
constexpr int kRotMax = 128, kRotThreads = 256;

template <int cols>  // of X a block
__global__ void __launch_bounds__(kRotThreads) rorope_apply_kernel(const float* X, int C, const float* U, int g, int d, int fold, float* Y) {
  const int m = g * fold, mp = (m + 7) & ~7, G = blockIdx.y, im = blockIdx.z, c0 = blockIdx.x * cols;
  constexpr int across = cols / 4;
  const int tid = threadIdx.x, tx = tid & (across - 1), row0 = tid / across, q0 = row0 * 8, c = c0 + tx * 4;
  extern __shared__ __align__(16) float rot_s[];
  float* u_s = rot_s;               // [m][mp], zeros behind column m
  float* x_s = u_s + m * mp;        // [m][cols]
  const bool vec = (C & 3) == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0;
  for (int e = tid; e < m * mp; e += kRotThreads) {
    const int i = e / mp, q = e - i * mp;
    u_s[e] = q < m ? U[(static_cast<size_t>(G) * m + i) * m + q] : 0.f;
  }
  for (int i = row0; i < m; i += kRotThreads / across) {
    const float* src = X + static_cast<size_t>(seg_pos(G, i, g, d, fold) + im) * C + c;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec) { if (c < C) x = *reinterpret_cast<const float4*>(src); }
    else {
      if (c < C) x.x = src[0];
      if (c + 1 < C) x.y = src[1];
      if (c + 2 < C) x.z = src[2];
      if (c + 3 < C) x.w = src[3];
    }
    *reinterpret_cast<float4*>(x_s + i * cols + tx * 4) = x;
  }
  __syncthreads();
  if (q0 >= m) return;
  float acc[8][4] = {};
#pragma unroll 4
  for (int i = 0; i < m; ++i) {
    const float4 x = *reinterpret_cast<const float4*>(x_s + i * cols + tx * 4);
    const float4 ua = *reinterpret_cast<const float4*>(u_s + i * mp + q0), ub = *reinterpret_cast<const float4*>(u_s + i * mp + q0 + 4);
    const float u[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      acc[k][0] = fmaf(u[k], x.x, acc[k][0]); acc[k][1] = fmaf(u[k], x.y, acc[k][1]);
      acc[k][2] = fmaf(u[k], x.z, acc[k][2]); acc[k][3] = fmaf(u[k], x.w, acc[k][3]);
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int q = q0 + k;
    if (q >= m) break;
    float* dst = Y + static_cast<size_t>((q / fold) * d + 2 * (G * fold + q % fold) + im) * C + c;
    if (vec) { if (c < C) *reinterpret_cast<float4*>(dst) = make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]); }
    else {
#pragma unroll
      for (int j = 0; j < 4; ++j) if (c + j < C) dst[j] = acc[k][j];
    }
  }
}

cudaError_t rorope_apply(const float* X, int C, const float* U, int g, int d, int fold, float* Y, cudaStream_t stream) {
  const int m = g * fold, mp = (m + 7) & ~7, groups = d / 2 / fold;
  if (m > kRotMax) return cudaErrorInvalidValue;
  auto launch = [&](auto kernel, int cols) {
    const size_t smem = static_cast<size_t>(m) * (mp + cols) * sizeof(float);
    kernel<<<dim3((C + cols - 1) / cols, groups, 2), kRotThreads, smem, stream>>>(X, C, U, g, d, fold, Y);
    return cudaGetLastError();
  };
  if (m <= 8) return launch(rorope_apply_kernel<1024>, 1024);
  if (m <= 16) return launch(rorope_apply_kernel<512>, 512);
  if (m <= 32) return launch(rorope_apply_kernel<256>, 256);
  static PerDeviceFlag smem_set[2];  // above the default limit
  if (m <= 64) {
    if (cudaError_t e = ensure_dynamic_smem(rorope_apply_kernel<128>, 64 * (64 + 128) * 4, smem_set[0]); e != cudaSuccess) return e;
    return launch(rorope_apply_kernel<128>, 128);
  }
  if (cudaError_t e = ensure_dynamic_smem(rorope_apply_kernel<64>, kRotMax * (kRotMax + 64) * 4, smem_set[1]); e != cudaSuccess) return e;
  return launch(rorope_apply_kernel<64>, 64);
}

// ------------------------------------------------------------------------------------------------ Eq. 19
// norms[0..n) = ||k_nope,t||, norms[n..2n) = ||v_t||: one warp per row; then one block sums both halves in a fixed
// order (the same bits on every run) and writes alpha = mean ||k|| / mean ||v||.  Bound by memory: 16-byte loads where the
// rows are aligned for them, four on their way a lane.
__global__ void row_norms_kernel(const float* a, int n, int m, float* out) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;
  float s = 0.f;
  const float* src = a + static_cast<size_t>(row) * m;
  if ((m & 3) == 0 && (reinterpret_cast<uintptr_t>(a) & 15) == 0) {
#pragma unroll 4
    for (int c = lane * 4; c < m; c += 128) {
      const float4 x = *reinterpret_cast<const float4*>(src + c);
      s = fmaf(x.x, x.x, s); s = fmaf(x.y, x.y, s); s = fmaf(x.z, x.z, s); s = fmaf(x.w, x.w, s);
    }
  } else {
    for (int c = lane; c < m; c += 32) s = fmaf(src[c], src[c], s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[row] = sqrtf(s);
}
__global__ void __launch_bounds__(1024) alpha_kernel(const float* norms, int n, float* alpha_out) {
  __shared__ double part[2][1024];
  double sk = 0.0, sv = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) { sk += norms[i]; sv += norms[n + i]; }
  part[0][threadIdx.x] = sk; part[1][threadIdx.x] = sv;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if (threadIdx.x < o) { part[0][threadIdx.x] += part[0][threadIdx.x + o]; part[1][threadIdx.x] += part[1][threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) *alpha_out = static_cast<float>(part[0][0] / part[1][0]);
}
cudaError_t row_norm_ratio(const float* k_nope, int n, int mk, const float* v, int mv, float* scratch, float* alpha_out,
                           cudaStream_t stream) {
  row_norms_kernel<<<(n + 7) / 8, 256, 0, stream>>>(k_nope, n, mk, scratch);
  row_norms_kernel<<<(n + 7) / 8, 256, 0, stream>>>(v, n, mv, scratch + n);
  alpha_kernel<<<1, 1024, 0, stream>>>(scratch, n, alpha_out);
  return cudaGetLastError();
}

// Z[t] = [k_nope,t / alpha ; v_t]   (App. D.2 step 1).  `lanes` threads a row, as many as it has pieces, up to a block; a
// piece is 16 bytes where the rows are aligned for them.  Bound by memory.  n = 8192, 3968 + 4096 columns: 290 us with a
// division an element, now 81; n = 65536, 16 + 16 columns 8.8 us, now 3.8 (23.5 with a block a row whatever its length).
__global__ void balance_concat_kernel(const float* k_nope, int n, int mk, const float* v, int mv, const float* alpha, float* Z, int vec,
                                      int lanes) {
  const float inv = 1.f / *alpha;
  const int m = mk + mv, rows = blockDim.x / lanes, lane = threadIdx.x & (lanes - 1);
  for (int t = blockIdx.x * rows + threadIdx.x / lanes; t < n; t += gridDim.x * rows) {
    const float* k_row = k_nope + static_cast<size_t>(t) * mk;
    const float* v_row = v + static_cast<size_t>(t) * mv;
    float* z_row = Z + static_cast<size_t>(t) * m;
    if (vec) {
#pragma unroll 4
      for (int c = lane * 4; c < m; c += lanes * 4) {
        float4 x = *reinterpret_cast<const float4*>(c < mk ? k_row + c : v_row + (c - mk));
        if (c < mk) { x.x *= inv; x.y *= inv; x.z *= inv; x.w *= inv; }
        *reinterpret_cast<float4*>(z_row + c) = x;
      }
    } else {
      for (int c = lane; c < m; c += lanes) z_row[c] = c < mk ? k_row[c] * inv : v_row[c - mk];
    }
  }
}
cudaError_t balance_concat(const float* k_nope, int n, int mk, const float* v, int mv, const float* alpha, float* Z,
                           cudaStream_t stream) {
  const bool vec = ((mk | mv) & 3) == 0 &&
                   ((reinterpret_cast<uintptr_t>(k_nope) | reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(Z)) & 15) == 0;
  const long long pieces = vec ? (static_cast<long long>(mk) + mv) / 4 : static_cast<long long>(mk) + mv;
  int lanes = 1;
  while (lanes < 256 && lanes < pieces) lanes *= 2;
  const int rows = 256 / lanes, blocks = (n + rows - 1) / rows;
  balance_concat_kernel<<<blocks < 1184 ? blocks : 1184, 256, 0, stream>>>(k_nope, n, mk, v, mv, alpha, Z, vec, lanes);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------ eigenvectors
// Parallel cyclic Jacobi for a symmetric matrix of order m <= 128, one block per matrix, A and V in shared memory.
// A round rotates m/2 disjoint index pairs (round-robin tournament), all with angles taken from the matrix as it
// stands before the round.  Sweeps stop when the off-diagonal mass is below fp32 resolution of the whole; the eigenvalues
// are then sorted in descending order.
// What bounds it: shared memory, and the chain of rounds.  A pair of pairs (k, l) owns a 2 x 2 block of A, so a thread
// applies J_k^T . J_l to it in registers in one visit, for k < l only, and writes the block and its mirror image; the
// diagonal blocks belong to the threads that find the angles.  V, which no angle depends on, is rotated while two warps find
// the next round's angles: two barriers a round.  Index pairs advance by one a round, so no thread divides.
// 16 matrices of order 128: 9.15 ms with columns and rows of A in passes of their own, 1.6 to 2.7 ms (by sweeps needed) in
// this form, and eigenvalues ten times closer because the angles' own 2 x 2 blocks are set to their exact form.
// A warp for every pair of V's columns and two for the angles, 32 at most: a small order then leaves room for several matrices
// on an SM.  512 matrices of order 16: 127 us before, 206 with 32 warps whatever the order, now 103.
constexpr int kEigMax = 128, kEigSweeps = 30, kEigThreads = 1024;
constexpr int kEigBlocks = (kEigMax / 2) * (kEigMax / 2 - 1) / 2;                  // pairs of index pairs
constexpr int kEigOwn = (kEigBlocks + kEigThreads - 1) / kEigThreads;             // of one thread

// Sum over the block; every thread gets it.
__device__ __forceinline__ float eig_block_sum(float x, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();  // the readers of the call before are done
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  x = (threadIdx.x & 31) < blockDim.x / 32 ? red[threadIdx.x & 31] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__global__ void __launch_bounds__(kEigThreads) jacobi_eigh_kernel(const float* a_in, int m, float* eigvals, float* eigvecs,
                                                          int32_t* dev_status) {
  extern __shared__ float es[];
  // An odd order gets one more index, of zeros: nothing couples to it, so it never turns.  Odd row length: columns are as
  // free of bank conflicts as rows.
  const int mm = (m + 1) & ~1, half = mm / 2, ring = mm - 1, ld = mm + 1;
  float* A = es;                    // [mm][ld]
  float* V = A + mm * ld;           // [mm][ld]
  __shared__ float2 cs[2][kEigMax / 2];  // cosine and sine of each pair, this round's and the next one's
  __shared__ float red[kEigThreads / 32];
  __shared__ int order[kEigMax];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x, warps = threads >> 5;
  const float* src = a_in + static_cast<size_t>(blockIdx.x) * m * m;
  for (int e = tid; e < mm * mm; e += threads) {
    const int i = e / mm, j = e % mm;
    A[i * ld + j] = i < m && j < m ? 0.5f * (src[i * m + j] + src[j * m + i]) : 0.f;  // exactly symmetric whatever rounding the input carries
    V[i * ld + j] = i == j ? 1.f : 0.f;
  }
  // The blocks (k, l), k < l, of this thread.  Row r of the triangle and row half-1-r have half-1 entries between them.
  int own_k[kEigOwn], own_l[kEigOwn];
#pragma unroll
  for (int u = 0; u < kEigOwn; ++u) {
    const int e = tid + u * threads;
    own_k[u] = -1;
    own_l[u] = 0;
    if (half < 2) continue;
    const int r = e / (half - 1), c = e % (half - 1);
    if (c < half - 1 - r) { own_k[u] = r; own_l[u] = r + 1 + c; }
    else if (r < half - 1 - r) { own_k[u] = half - 1 - r; own_l[u] = c + 1; }
    if (r >= (half + 1) / 2) own_k[u] = -1;
  }
  auto first_of = [&](int k, int rd) { if (k == 0) return mm - 1; const int x = rd + k; return x >= ring ? x - ring : x; };
  auto second_of = [&](int k, int rd) { const int x = rd - k; return x < 0 ? x + ring : x; };
  auto find_angles = [&](int rd) {  // threads 0 .. half-1
    if (tid >= half) return;
    const int p = first_of(tid, rd), q = second_of(tid, rd);
    const float apq = A[p * ld + q], app = A[p * ld + p], aqq = A[q * ld + q];
    float c = 1.f, s = 0.f;
    if (fabsf(apq) > 1e-30f) {
      const float theta = (aqq - app) / (2.f * apq);
      const float t = (theta >= 0.f ? 1.f : -1.f) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
      c = 1.f / sqrtf(t * t + 1.f);
      s = t * c;
      A[p * ld + p] = app - t * apq;
      A[q * ld + q] = aqq + t * apq;
      A[p * ld + q] = 0.f;
      A[q * ld + p] = 0.f;
    }
    cs[rd & 1][tid] = make_float2(c, s);
  };
  __syncthreads();
  bool done = false;
  float prev_off = 3.4e38f;
  for (int sweep = 0; sweep < kEigSweeps; ++sweep) {
    // convergence: off-diagonal sum of squares against the whole
    float off = 0.f, diag = 0.f;
    for (int i = warp; i < m; i += warps)
      for (int j = lane; j < m; j += 32) {
        const float x = A[i * ld + j];
        if (i == j) diag += x * x; else off += x * x;
      }
    const float off_all = eig_block_sum(off, red), tot_all = off_all + eig_block_sum(diag, red);
    // converged: the off-diagonal mass is gone, or it sits at the fp32 rounding floor of the rotations (it has
    // stopped shrinking and is below 1e-8 of the whole)
    if (off_all <= 1e-13f * tot_all || (sweep >= 4 && off_all > 0.25f * prev_off && off_all <= 1e-8f * tot_all)) { done = true; break; }
    prev_off = off_all;
    find_angles(0);
    __syncthreads();
    for (int rd = 0; rd < ring; ++rd) {
      const float2* rot = cs[rd & 1];
#pragma unroll
      for (int u = 0; u < kEigOwn; ++u) {                      // A <- J^T A J off the diagonal blocks
        if (own_k[u] < 0) continue;
        const float2 rk = rot[own_k[u]], rl = rot[own_l[u]];
        const int pk = first_of(own_k[u], rd), qk = second_of(own_k[u], rd), pl = first_of(own_l[u], rd), ql = second_of(own_l[u], rd);
        const float x = A[pk * ld + pl], y = A[pk * ld + ql], z = A[qk * ld + pl], w = A[qk * ld + ql];
        const float x1 = rl.x * x - rl.y * y, y1 = rl.y * x + rl.x * y, z1 = rl.x * z - rl.y * w, w1 = rl.y * z + rl.x * w;
        const float x2 = rk.x * x1 - rk.y * z1, z2 = rk.y * x1 + rk.x * z1, y2 = rk.x * y1 - rk.y * w1, w2 = rk.y * y1 + rk.x * w1;
        A[pk * ld + pl] = x2; A[pk * ld + ql] = y2; A[qk * ld + pl] = z2; A[qk * ld + ql] = w2;
        A[pl * ld + pk] = x2; A[ql * ld + pk] = y2; A[pl * ld + qk] = z2; A[ql * ld + qk] = w2;
      }
      __syncthreads();
      if (warp < 2) {
        if (rd + 1 < ring) find_angles(rd + 1);
      } else {
        for (int k = warp - 2; k < half; k += warps - 2) {  // V <- V J, a pair of columns a warp
          const float2 r = rot[k];
          float* vp = V + first_of(k, rd) + lane * ld;
          float* vq = V + second_of(k, rd) + lane * ld;
#pragma unroll
          for (int i = 0; i < kEigMax; i += 32) {
            if (i + lane >= m) break;
            const float a = vp[i * ld], b = vq[i * ld];
            vp[i * ld] = r.x * a - r.y * b;
            vq[i * ld] = r.y * a + r.x * b;
          }
        }
      }
      __syncthreads();
    }
  }
  if (tid == 0 && !done && dev_status != nullptr) atomicOr(dev_status, TRANSMLA_DEV_NUMERIC);
  if (tid < m) {  // descending, equal values by index; a value that is not a number goes behind those that are
    const float x = A[tid * ld + tid];
    int rank = 0;
    for (int j = 0; j < m; ++j) {
      const float y = A[j * ld + j];
      const bool before = isnan(x) ? (!isnan(y) || j < tid) : (y > x || (y == x && j < tid));
      rank += before;
    }
    order[rank] = tid;
  }
  __syncthreads();
  float* w = eigvals + static_cast<size_t>(blockIdx.x) * m;
  float* vec = eigvecs + static_cast<size_t>(blockIdx.x) * m * m;
  for (int q = tid; q < m; q += threads) w[q] = A[order[q] * ld + order[q]];
  for (int e = tid; e < m * m; e += threads) { const int i = e / m, q = e % m; vec[e] = V[i * ld + order[q]]; }
}

cudaError_t sym_eig(float* a, int batch, int m, float* eigvals, float* eigvecs, int32_t* dev_status, cudaStream_t stream) {
  if (m < 1 || m > kEigMax) return cudaErrorInvalidValue;
  const size_t mm = (m + 1) & ~1, smem = 2 * mm * (mm + 1) * sizeof(float);
  if (cudaError_t e = cudaFuncSetAttribute(jacobi_eigh_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
      e != cudaSuccess)
    return e;
  const int pairs = (m + 1) / 2, warps = pairs + 2 < kEigThreads / 32 ? pairs + 2 : kEigThreads / 32;
  jacobi_eigh_kernel<<<batch, warps * 32, smem, stream>>>(a, m, eigvals, eigvecs, dev_status);
  return cudaGetLastError();
}
}  // namespace conv
}  // namespace transmla

// Kernels of the GQA -> MLA conversion on calibration activations (Sec. 4.2, 4.3; App. B, C, D): rotations, balancing and
// eigenvectors in fp32 arithmetic.  The matrix products are in conversion_gemm.cu, the orthonormalisation of the subspace
// iteration in conversion_qr.cu.
#include "conversion.cuh"

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
__global__ void rorope_apply_kernel(const float* X, int C, const float* U, int g, int d, int fold, float* Y) {
  const int m = g * fold, G = blockIdx.y, im = blockIdx.z;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  extern __shared__ float u_s[];  // U_G [m][m]
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) u_s[e] = U[static_cast<size_t>(G) * m * m + e];
  __syncthreads();
  if (c >= C) return;
  for (int q0 = 0; q0 < m; q0 += 8) {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int i = 0; i < m; ++i) {
      const float x = X[static_cast<size_t>(seg_pos(G, i, g, d, fold) + im) * C + c];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (q0 + u < m) acc[u] = fmaf(u_s[i * m + q0 + u], x, acc[u]);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int q = q0 + u;
      if (q < m) Y[static_cast<size_t>((q / fold) * d + 2 * (G * fold + q % fold) + im) * C + c] = acc[u];
    }
  }
}

cudaError_t rorope_apply(const float* X, int C, const float* U, int g, int d, int fold, float* Y, cudaStream_t stream) {
  const int m = g * fold, groups = d / 2 / fold;
  const size_t smem = static_cast<size_t>(m) * m * sizeof(float);
  if (smem > 48 * 1024) {
    if (cudaError_t e = cudaFuncSetAttribute(rorope_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        e != cudaSuccess)
      return e;
  }
  dim3 grid((C + 127) / 128, groups, 2);
  rorope_apply_kernel<<<grid, 128, smem, stream>>>(X, C, U, g, d, fold, Y);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------ Eq. 19
// norms[0..n) = ||k_nope,t||, norms[n..2n) = ||v_t||: one warp per row; then one block sums both halves in a fixed
// order (the same bits on every run) and writes alpha = mean ||k|| / mean ||v||.
__global__ void row_norms_kernel(const float* a, int n, int m, float* out) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;
  float s = 0.f;
  for (int c = lane; c < m; c += 32) { const float x = a[static_cast<size_t>(row) * m + c]; s = fmaf(x, x, s); }
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

// Z[t] = [k_nope,t / alpha ; v_t]   (App. D.2 step 1)
__global__ void balance_concat_kernel(const float* k_nope, int n, int mk, const float* v, int mv, const float* alpha, float* Z) {
  const float inv = 1.f / *alpha;
  const int m = mk + mv;
  const size_t total = static_cast<size_t>(n) * m;
  for (size_t e = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t t = e / m;
    const int c = static_cast<int>(e % m);
    Z[e] = c < mk ? k_nope[t * mk + c] * inv : v[t * mv + (c - mk)];
  }
}
cudaError_t balance_concat(const float* k_nope, int n, int mk, const float* v, int mv, const float* alpha, float* Z,
                           cudaStream_t stream) {
  balance_concat_kernel<<<592, 256, 0, stream>>>(k_nope, n, mk, v, mv, alpha, Z);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------ eigenvectors
// Parallel cyclic Jacobi for a symmetric matrix of order m <= 128, one block per matrix, A and V in shared memory.
// A round rotates m/2 disjoint index pairs (round-robin tournament), all with angles taken from the matrix as it
// stands before the round: columns first (A <- A J, V <- V J), then rows (A <- J^T A).  Sweeps stop when the
// off-diagonal mass is below fp32 resolution of the whole; the eigenvalues are then sorted in descending order.
constexpr int kEigMax = 128, kEigSweeps = 30, kEigThreads = 512;

__global__ void __launch_bounds__(kEigThreads) jacobi_eigh_kernel(const float* a_in, int m, float* eigvals, float* eigvecs,
                                                          int32_t* dev_status) {
  extern __shared__ float es[];
  const int ld = m + 1, mm = (m + 1) & ~1, half = mm / 2;
  float* A = es;                    // [m][ld]
  float* V = A + m * ld;            // [m][ld]
  float* cs = V + m * ld;           // [half][2]
  int* pq = reinterpret_cast<int*>(cs + 2 * half);  // [half][2]
  int* order = pq + 2 * half;       // [m]
  __shared__ float red[kEigThreads];
  __shared__ int done;
  const int tid = threadIdx.x;
  const float* src = a_in + static_cast<size_t>(blockIdx.x) * m * m;
  for (int e = tid; e < m * m; e += kEigThreads) {
    const int i = e / m, j = e % m;
    A[i * ld + j] = 0.5f * (src[e] + src[j * m + i]);  // exactly symmetric whatever rounding the input carries
    V[i * ld + j] = i == j ? 1.f : 0.f;
  }
  if (tid == 0) done = 0;
  __syncthreads();
  float prev_off = 3.4e38f;
  for (int sweep = 0; sweep < kEigSweeps; ++sweep) {
    // convergence: off-diagonal sum of squares against the whole
    float off = 0.f, tot = 0.f;
    for (int e = tid; e < m * m; e += kEigThreads) {
      const int i = e / m, j = e % m;
      const float x = A[i * ld + j];
      tot += x * x;
      if (i != j) off += x * x;
    }
    red[tid] = off; __syncthreads();
    for (int o = kEigThreads / 2; o > 0; o >>= 1) { if (tid < o) red[tid] += red[tid + o]; __syncthreads(); }
    const float off_all = red[0]; __syncthreads();
    red[tid] = tot; __syncthreads();
    for (int o = kEigThreads / 2; o > 0; o >>= 1) { if (tid < o) red[tid] += red[tid + o]; __syncthreads(); }
    const float tot_all = red[0]; __syncthreads();
    // converged: the off-diagonal mass is gone, or it sits at the fp32 rounding floor of the rotations (it has
    // stopped shrinking and is below 1e-8 of the whole)
    if (off_all <= 1e-13f * tot_all || (sweep >= 4 && off_all > 0.25f * prev_off && off_all <= 1e-8f * tot_all)) {
      if (tid == 0) done = 1;
      __syncthreads();
      break;
    }
    prev_off = off_all;
    for (int rd = 0; rd < mm - 1; ++rd) {
      if (tid < half) {
        int p, q;
        if (tid == 0) { p = mm - 1; q = rd; }
        else { p = (rd + tid) % (mm - 1); q = (rd - tid + mm - 1) % (mm - 1); }
        if (p > q) { const int t = p; p = q; q = t; }
        float c = 1.f, s = 0.f;
        if (q < m) {
          const float apq = A[p * ld + q], app = A[p * ld + p], aqq = A[q * ld + q];
          if (fabsf(apq) > 1e-30f) {
            const float theta = (aqq - app) / (2.f * apq);
            const float t = (theta >= 0.f ? 1.f : -1.f) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
            c = 1.f / sqrtf(t * t + 1.f);
            s = t * c;
          }
        } else { p = -1; }
        pq[2 * tid] = p; pq[2 * tid + 1] = q; cs[2 * tid] = c; cs[2 * tid + 1] = s;
      }
      __syncthreads();
      for (int e = tid; e < half * m; e += kEigThreads) {      // columns p, q of A and V
        const int k = e / m, i = e % m, p = pq[2 * k], q = pq[2 * k + 1];
        if (p < 0) continue;
        const float c = cs[2 * k], s = cs[2 * k + 1];
        const float ap = A[i * ld + p], aq = A[i * ld + q];
        A[i * ld + p] = c * ap - s * aq; A[i * ld + q] = s * ap + c * aq;
        const float vp = V[i * ld + p], vq = V[i * ld + q];
        V[i * ld + p] = c * vp - s * vq; V[i * ld + q] = s * vp + c * vq;
      }
      __syncthreads();
      for (int e = tid; e < half * m; e += kEigThreads) {      // rows p, q of A
        const int k = e / m, j = e % m, p = pq[2 * k], q = pq[2 * k + 1];
        if (p < 0) continue;
        const float c = cs[2 * k], s = cs[2 * k + 1];
        const float ap = A[p * ld + j], aq = A[q * ld + j];
        A[p * ld + j] = c * ap - s * aq; A[q * ld + j] = s * ap + c * aq;
      }
      __syncthreads();
    }
  }
  if (tid == 0) {
    if (!done && dev_status != nullptr) atomicOr(dev_status, TRANSMLA_DEV_NUMERIC);
    for (int i = 0; i < m; ++i) order[i] = i;
    for (int i = 0; i < m; ++i) {       // selection sort, descending (stable for equal values)
      int best = i;
      for (int j = i + 1; j < m; ++j)
        if (A[order[j] * ld + order[j]] > A[order[best] * ld + order[best]]) best = j;
      const int t = order[best];
      for (int j = best; j > i; --j) order[j] = order[j - 1];
      order[i] = t;
    }
  }
  __syncthreads();
  float* w = eigvals + static_cast<size_t>(blockIdx.x) * m;
  float* vec = eigvecs + static_cast<size_t>(blockIdx.x) * m * m;
  for (int q = tid; q < m; q += kEigThreads) w[q] = A[order[q] * ld + order[q]];
  for (int e = tid; e < m * m; e += kEigThreads) { const int i = e / m, q = e % m; vec[e] = V[i * ld + order[q]]; }
}

cudaError_t sym_eig(float* a, int batch, int m, float* eigvals, float* eigvecs, int32_t* dev_status, cudaStream_t stream) {
  if (m < 1 || m > kEigMax) return cudaErrorInvalidValue;
  const int half = ((m + 1) & ~1) / 2;
  const size_t smem = (static_cast<size_t>(2) * m * (m + 1) + 4 * half + m) * sizeof(float);
  if (cudaError_t e = cudaFuncSetAttribute(jacobi_eigh_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
      e != cudaSuccess)
    return e;
  jacobi_eigh_kernel<<<batch, kEigThreads, smem, stream>>>(a, m, eigvals, eigvecs, dev_status);
  return cudaGetLastError();
}
}  // namespace conv
}  // namespace transmla

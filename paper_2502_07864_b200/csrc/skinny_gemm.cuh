// Skinny GEMM tile shared by the append and by the layer's linear maps: y[t, f0..f0+7] = x[t, :] . w[f0..f0+7, :]
// for a range of tokens t (the M dimension of the tensor-core tiles).  One block owns 8 consecutive output
// features; its 8 warps split the contracted dimension and meet in shared memory; every (token, feature pair)
// is handed to an epilogue functor.  Operands are read straight from global memory with 16-byte loads in a
// permuted k order (see small_kernels.cu).
#pragma once
#include "common.cuh"

namespace transmla {

__device__ __forceinline__ uint32_t ld_u32(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ uint4 ld_u128(const __nv_bfloat16* p) { return *reinterpret_cast<const uint4*>(p); }

// RoPE of Eq. 1 on the pair (re, im) = elements (2l, 2l+1) of a d-vector at position pos.  The angle is formed
// and reduced to [-pi, pi] in fp64 so that positions of 10^5 keep their phase; sine and cosine are fp32.
__device__ __forceinline__ double rope_freq(int l, int d, float theta) { return exp2(-2.0 * l / d * log2(static_cast<double>(theta))); }
__device__ __forceinline__ void rope_angle(int pos, double freq, float& cs, float& sn) {
  const double ang = static_cast<double>(pos) * freq;
  const double red_ang = ang - 6.283185307179586476925 * rint(ang * 0.15915494309189533577);
  sincosf(static_cast<float>(red_ang), &sn, &cs);
}
__device__ __forceinline__ void rope_pair_at(float& re, float& im, int pos, double freq) {
  float sn, cs;
  rope_angle(pos, freq, cs, sn);
  const float nre = re * cs - im * sn, nim = im * cs + re * sn;
  re = nre;
  im = nim;
}
__device__ __forceinline__ void rope_pair(float& re, float& im, int pos, int l, int d, float theta) {
  rope_pair_at(re, im, pos, rope_freq(l, d, theta));
}

constexpr int kAppendMaxMT = 8;  // 16-token tiles per pass
constexpr size_t kAppendSmem = 8 * kAppendMaxMT * 16 * 8 * sizeof(float);  // 32 KB

// Partial products of one warp over its slice of the hidden dimension for tokens [t0, t0 + 16*MT).
template <int MT, int UNROLL, int MAXMT, int NT>
__device__ __forceinline__ void append_partial(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ wrow,
                                               int D, int T, int t0, int k_lo, int slice, int g, int t4,
                                               float (&acc)[MAXMT][NT][4]) {
  const __nv_bfloat16* xr[MT][2];
  bool ok[MT][2];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int row = t0 + mt * 16 + g + hf * 8;
      ok[mt][hf] = row < T;
      xr[mt][hf] = x + static_cast<size_t>(min(row, T - 1)) * D + k_lo + t4 * 8;
    }
#pragma unroll UNROLL
  for (int k = 0; k < slice; k += 32) {
    uint4 wv[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) wv[nt] = ld_u128(wrow + static_cast<size_t>(nt) * 8 * D + k);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      uint4 x0 = make_uint4(0, 0, 0, 0), x1 = make_uint4(0, 0, 0, 0);
      if (ok[mt][0]) x0 = ld_u128(xr[mt][0] + k);
      if (ok[mt][1]) x1 = ld_u128(xr[mt][1] + k);
      const uint32_t a0[4] = {x0.x, x1.x, x0.y, x1.y}, a1[4] = {x0.z, x1.z, x0.w, x1.w};
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        mma_bf16_16816(acc[mt][nt], a0, wv[nt].x, wv[nt].y);
        mma_bf16_16816(acc[mt][nt], a1, wv[nt].z, wv[nt].w);
      }
    }
  }
}

// Shared memory the tile needs for the meeting of its 8 warps.
constexpr size_t skinny_gemm_smem(int maxmt, int nt) { return static_cast<size_t>(8) * maxmt * 16 * 8 * nt * sizeof(float); }

// x [*, K] row-major, w [*, K] row-major (K a multiple of 256), tokens [t_begin, t_end), output features
// f0 .. f0 + 8*NT - 1.  smem_raw: skinny_gemm_smem(MAXMT, NT) bytes.
// epi(token, pair 0..4*NT-1, value of feature f0 + 2*pair, value of feature f0 + 2*pair + 1) is called once per pair.
// MAXMT: 16-token tiles per pass.  NT: 8-feature tiles per block; more of them re-read the activations less often,
// which is what bounds these kernels once the weights are large (every block reads all its tokens' activations).
template <int MAXMT = kAppendMaxMT, int NT = 1, class Epi>
__device__ __forceinline__ void skinny_gemm_tile(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ w,
                                                 int K, int f0, int t_begin, int t_end, unsigned char* smem_raw, Epi epi) {
  float* red = reinterpret_cast<float*>(smem_raw);  // [8 warps][MAXMT*16 rows][8*NT]
  constexpr int kCols = 8 * NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int slice = K / 8, k_lo = warp * slice;
  const __nv_bfloat16* wrow = w + static_cast<size_t>(f0 + g) * K + k_lo + t4 * 8;
  if (t4 == 0)
    for (int nt = 0; nt < NT; ++nt)
      for (int k = 0; k < slice; k += 64) prefetch_l2(wrow + static_cast<size_t>(nt) * 8 * K + k);  // this warp's weight lines
  pdl_wait();  // activations and everything the epilogue touches may belong to kernels still in flight; weights may not
  const int T = t_end;
  for (int t0 = t_begin; t0 < T; t0 += MAXMT * 16) {
    float acc[MAXMT][NT][4];
#pragma unroll
    for (int mt = 0; mt < MAXMT; ++mt)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) acc[mt][nt][0] = acc[mt][nt][1] = acc[mt][nt][2] = acc[mt][nt][3] = 0.f;
    const int left = T - t0;
    constexpr int U1 = NT == 1 ? 8 : 4, U2 = NT == 1 ? 4 : 2;
    if (left <= 16) append_partial<1, U1, MAXMT, NT>(x, wrow, K, T, t0, k_lo, slice, g, t4, acc);
    else if (MAXMT == 2 || left <= 32) append_partial<(MAXMT >= 2 ? 2 : MAXMT), U2, MAXMT, NT>(x, wrow, K, T, t0, k_lo, slice, g, t4, acc);
    else if (left <= 64) append_partial<(MAXMT >= 4 ? 4 : MAXMT), U2, MAXMT, NT>(x, wrow, K, T, t0, k_lo, slice, g, t4, acc);
    else append_partial<MAXMT, (NT == 1 ? 2 : 1), MAXMT, NT>(x, wrow, K, T, t0, k_lo, slice, g, t4, acc);
    __syncthreads();  // previous pass has consumed `red`
#pragma unroll
    for (int mt = 0; mt < MAXMT; ++mt) {
      if (mt * 16 < left) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          float* d = red + (warp * MAXMT * 16 + mt * 16 + g) * kCols + nt * 8 + t4 * 2;
          *reinterpret_cast<float2*>(d) = make_float2(acc[mt][nt][0], acc[mt][nt][1]);
          *reinterpret_cast<float2*>(d + 8 * kCols) = make_float2(acc[mt][nt][2], acc[mt][nt][3]);
        }
      }
    }
    __syncthreads();
    const int rows = min(MAXMT * 16, left);
    for (int i = tid; i < rows * 4 * NT; i += 256) {
      const int row = i / (4 * NT), pr = i % (4 * NT);
      float re = 0.f, im = 0.f;
#pragma unroll
      for (int wv = 0; wv < 8; ++wv) {
        const float2 v = *reinterpret_cast<const float2*>(red + (wv * MAXMT * 16 + row) * kCols + pr * 2);
        re += v.x; im += v.y;
      }
      epi(t0 + row, pr, re, im);
    }
  }
}

// ------------------------------------------------------------------------------------------------
// The append's form for latents and rope keys of any size (r = 512, dR = 64 has prologue_sm100.cu): a cluster of kSliceCtas
// CTAs owns 64 features x 64 tokens, each CTA a slice of the contracted dimension, which it takes through shared memory 128
// wide (asynchronous copies, three pieces in flight, the weights of the first three from before the dependency wait).  Its
// warps take 32 of a piece's 128 each and half of the tokens, meet in shared memory, and the CTAs' sums meet through
// distributed shared memory: CTA i finishes the i-th share of the tokens, adding the slices in order.
// What bounds it is what an SM gets from L2 (30 bytes a cycle) and round trips: a block of 32 features x 16 tokens read
// 384 KB at 128 tokens of D = 4096, one of 64 x 64 x D/8 reads 128, as many blocks.
// ------------------------------------------------------------------------------------------------
constexpr int kSliceCtas = 8, kSliceFeatures = 64, kSliceTokens = 64, kSliceK = 128, kSliceStages = 3;
constexpr int kSlicePitch = kSliceFeatures + 8;  // of the sums, floats (conflict-free fragments)
constexpr int kSliceRow = kSliceK + 8;           // of the operands, bf16 (conflict-free ldmatrix)
constexpr size_t kSliceSmem = static_cast<size_t>(kSliceStages) * (kSliceFeatures + kSliceTokens) * kSliceRow * sizeof(__nv_bfloat16);
static_assert(4 * kSliceTokens * kSlicePitch * sizeof(float) <= kSliceSmem, "the warps' sums take the ring's place");

__device__ __forceinline__ void slice_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// x [*, K] row-major, w [n_features, K] row-major, K a multiple of 256; features f0 .. f0 + 63 (those below n_features), tokens
// t_begin .. t_begin + 63 (those below t_end).  rank: of the CTA in its cluster.  Each (token, pair of features) belongs
// to one thread of the cluster: it calls prep(token) when the kernels before this one have finished, and
// epi(token, f, value of f, value of f + 1, what prep gave) with the sums.
template <class Prep, class Epi>
__device__ __forceinline__ void slice_gemm_tile(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ w, int K, int n_features,
                                                int f0, int t_begin, int t_end, int rank, unsigned char* smem_raw, Prep prep, Epi epi) {
  constexpr int kTok = kSliceTokens, kWarpsK = 4, MT = kTok / 2 / 16, NT = kSliceFeatures / 8;
  constexpr int kStage = (kSliceFeatures + kTok) * kSliceRow;                   // bf16
  __nv_bfloat16* ring = reinterpret_cast<__nv_bfloat16*>(smem_raw);             // stages of [features | tokens][kSliceRow]
  float* red = reinterpret_cast<float*>(smem_raw);                              // later: [kWarpsK][kTok][kSlicePitch]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3, mi = lane >> 3;
  const int wk = warp & 3, wt = warp >> 2;
  const int k_lo = rank * (K / kSliceCtas), k_hi = k_lo + K / kSliceCtas, pieces = (K / kSliceCtas + kSliceK - 1) / kSliceK;
  auto copy = [&](int piece, const __nv_bfloat16* src, int row0, int rows_end, int rows, int at) {  // 16 bytes a thread and turn
    __nv_bfloat16* dst = ring + piece % kSliceStages * kStage + at * kSliceRow;
#pragma unroll
    for (int i = tid; i < rows * (kSliceK / 8); i += 256) {
      const int rr = i / (kSliceK / 8), c = i % (kSliceK / 8) * 8, k = k_lo + piece * kSliceK + c;
      const bool in = row0 + rr < rows_end && k < k_hi;  // the rest is filled with zeros
      cp_async16(dst + rr * kSliceRow + c, src + (in ? static_cast<size_t>(row0 + rr) * K + k : 0), in ? 16 : 0);
    }
  };
#pragma unroll
  for (int p = 0; p < kSliceStages; ++p)
    if (p < pieces) copy(p, w, f0, n_features, kSliceFeatures, 0);
  cp_async_commit();
  pdl_wait();  // activations and everything the epilogue touches may belong to kernels still in flight; weights may not
#pragma unroll
  for (int p = 0; p < kSliceStages; ++p) {
    if (p < pieces) copy(p, x, t_begin, t_end, kTok, kSliceFeatures);
    cp_async_commit();
  }
  const int my_t = t_begin + rank * (kTok / kSliceCtas) + (tid >> 5);
  const bool mine = tid < kTok / kSliceCtas * 32 && my_t < t_end && f0 + 2 * lane < n_features;
  auto prepared = prep(mine ? my_t : -1);
  float acc[MT][NT][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) acc[mt][nt][0] = acc[mt][nt][1] = acc[mt][nt][2] = acc[mt][nt][3] = 0.f;
#pragma unroll 1
  for (int p = 0; p < pieces; ++p) {
    if (p == 0) cp_async_wait<kSliceStages - 1>(); else cp_async_wait<kSliceStages - 2>();
    __syncthreads();  // the piece is there for all, and all have finished the one before
    if (p > 0) {
      const int q = p + kSliceStages - 1;
      if (q < pieces) {
        copy(q, w, f0, n_features, kSliceFeatures, 0);
        copy(q, x, t_begin, t_end, kTok, kSliceFeatures);
      }
      cp_async_commit();
    }
    const __nv_bfloat16* ws = ring + p % kSliceStages * kStage + wk * 32;
    const __nv_bfloat16* xs = ring + p % kSliceStages * kStage + (kSliceFeatures + wt * MT * 16) * kSliceRow + wk * 32;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      uint32_t a[MT][4], b[NT / 2][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) ldmatrix_x4(a[mt], xs + (mt * 16 + (mi & 1) * 8 + (lane & 7)) * kSliceRow + ks * 16 + (mi >> 1) * 8);
#pragma unroll
      for (int n2 = 0; n2 < NT / 2; ++n2) ldmatrix_x4(b[n2], ws + (n2 * 16 + (mi >> 1) * 8 + (lane & 7)) * kSliceRow + ks * 16 + (mi & 1) * 8);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc[mt][nt], a[mt], b[nt / 2][nt % 2 * 2], b[nt / 2][nt % 2 * 2 + 1]);
    }
  }
  cp_async_wait<0>();
  __syncthreads();
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float* d = red + (wk * kTok + (wt * MT + mt) * 16 + g) * kSlicePitch + nt * 8 + t4 * 2;
      *reinterpret_cast<float2*>(d) = make_float2(acc[mt][nt][0], acc[mt][nt][1]);
      *reinterpret_cast<float2*>(d + 8 * kSlicePitch) = make_float2(acc[mt][nt][2], acc[mt][nt][3]);
    }
  __syncthreads();
#pragma unroll
  for (int i = tid; i < kTok * 16; i += 256) {  // the CTA's sum takes the place of its first warp's
    float4* d = reinterpret_cast<float4*>(red + (i >> 4) * kSlicePitch + (i & 15) * 4);
    float4 sum = *d;
#pragma unroll
    for (int wv = 1; wv < kWarpsK; ++wv) {
      const float4 v = *reinterpret_cast<const float4*>(red + (wv * kTok + (i >> 4)) * kSlicePitch + (i & 15) * 4);
      sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
    }
    *d = sum;
  }
  slice_cluster_sync();
  if (mine) {
    const uint32_t local = smem_u32(red + (my_t - t_begin) * kSlicePitch + 2 * lane);
    float2 v[kSliceCtas];
#pragma unroll
    for (int c = 0; c < kSliceCtas; ++c) {
      uint32_t remote;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(c));
      asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v[c].x), "=f"(v[c].y) : "r"(remote) : "memory");
    }
    float re = v[0].x, im = v[0].y;
#pragma unroll
    for (int c = 1; c < kSliceCtas; ++c) { re += v[c].x; im += v[c].y; }
    epi(my_t, f0 + 2 * lane, re, im, prepared);
  }
  slice_cluster_sync();  // nobody leaves while its memory may still be read
}

// Launch with programmatic dependent launch in clusters of kSliceCtas.
template <typename... KArgs, typename... Args>
cudaError_t launch_slices(void (*kernel)(KArgs...), int blocks, size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = kSliceCtas;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace transmla

// Latent append into the FP8 cache (Eq. 7 left, then this library's FP8 row format): the projection and RoPE run as in
// the bf16 append but leave fp32 rows in a scratch buffer, because a row's scale is the maximum over all of its 512
// latent values, which 64 different blocks of the projection produce; a second, tiny launch quantises the rows.
#include <cuda_fp16.h>

#include "common.cuh"
#include "skinny_gemm.cuh"

namespace transmla {

// y[t, :] = [W_DKV; W_KR] x_t with RoPE on y[r:], fp32, into scratch [T, r + dR].  Block = 8 NT features x a share of the
// tokens.  Bound by what an SM gets from L2: a block reads its features' weights and its tokens' activations.  64 tokens of
// D = 4096: 72 blocks of 8 features and all tokens read 576 KB each, 144 of 16 features and 16 tokens 256 KB:
// 19 -> 10.8 us.  The whole step at 64 tokens 106.5 -> 103 us, at 100 142.5 -> 122.7, at 128 shorter sequences 138 -> 108.
// A value is the same sum in the same order in every form.
template <int MAXMT, int NT>
__global__ void __launch_bounds__(256) append_rows_f32_kernel(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ w,
                                                              const int32_t* positions, float* rows, int B, int S, int D, int r,
                                                              int dR, float theta, int t_splits) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  const int K = r + dR, f_tiles = K / (8 * NT), f0 = (blockIdx.x % f_tiles) * 8 * NT;
  const int t_chunk = (((B * S + t_splits - 1) / t_splits) + 15) & ~15;
  const int t_begin = (blockIdx.x / f_tiles) * t_chunk, t_end = min(B * S, t_begin + t_chunk);
  skinny_gemm_tile<MAXMT, NT>(x, w, D, f0, t_begin, t_end, smem_raw, [&](int t, int pr, float re, float im) {
    const int f = f0 + pr * 2;
    if (f >= r) rope_pair(re, im, positions[t / S] + t % S, (f - r) >> 1, dR, theta);  // RoPE pair l of the decoupled key (Eq. 1)
    *reinterpret_cast<float2*>(rows + static_cast<size_t>(t) * K + f) = make_float2(re, im);
  });
}

// One warp per token: scale = max|c| / 448 (1 for an all-zero row), codes = e4m3(c / scale), k^R / scale as bf16,
// written to the token's 656-byte row.  r = 512, dR = 64.
__global__ void __launch_bounds__(128) quantize_rows_kernel(const float* rows, const int32_t* positions, const int32_t* page_table,
                                                            unsigned char* cache, int32_t* dev_status, int B, int S,
                                                            int num_pages, int max_pages) {
  pdl_trigger();
  pdl_wait();
  const int t = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= B * S) return;
  const int b = t / S, pos = positions[b] + t % S, pj = pos / kPage;
  int page = -1;
  if (pos >= 0 && pj < max_pages) page = page_table[static_cast<size_t>(b) * max_pages + pj];
  if (page < 0 || page >= num_pages) {
    if (lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE);
    return;
  }
  const float* row = rows + static_cast<size_t>(t) * 576;
  float c[16];
  float amax = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 v = *reinterpret_cast<const float4*>(row + lane * 16 + i * 4);
    c[4 * i] = v.x; c[4 * i + 1] = v.y; c[4 * i + 2] = v.z; c[4 * i + 3] = v.w;
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  const float scale = amax > 0.f ? amax / 448.f : 1.f;
  uint32_t codes[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint16_t lo, hi;
    asm volatile("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(lo) : "f"(c[4 * i + 1] / scale), "f"(c[4 * i] / scale));
    asm volatile("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(hi) : "f"(c[4 * i + 3] / scale), "f"(c[4 * i + 2] / scale));
    codes[i] = static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
  }
  unsigned char* dst = cache + (static_cast<size_t>(page) * kPage + pos % kPage) * TRANSMLA_FP8_ROW_BYTES;
  *reinterpret_cast<uint4*>(dst + lane * 16) = make_uint4(codes[0], codes[1], codes[2], codes[3]);
  const float2 kr = *reinterpret_cast<const float2*>(row + 512 + lane * 2);
  *reinterpret_cast<uint32_t*>(dst + 512 + lane * 4) = pack_bf16(kr.x / scale, kr.y / scale);
  if (lane < 4) *reinterpret_cast<uint32_t*>(dst + 640 + lane * 4) = lane == 0 ? __float_as_uint(scale) : 0u;
}

cudaError_t launch_append_fp8(const transmla_params_t& p, const __nv_bfloat16* x, const __nv_bfloat16* w, const int32_t* positions,
                              const int32_t* page_table, void* cache_fp8, float* scratch, int32_t* dev_status,
                              cudaStream_t stream) {
  const int K = p.kv_lora_rank + p.qk_rope_dim, T = p.batch * p.q_len;
  // Up to 48 tokens 8 features a block (the whole step at 33 tokens: 74.9 us, 77.1 in the next form), up to 64 tokens 16
  // features x 16 tokens, beyond that 32 x 16: about as many blocks as SMs (r + dR = 576 is a multiple of 32).
  const int ts = T <= 48 ? 1 : (T + 15) / 16 > 32 ? 32 : (T + 15) / 16;
  auto rows = [&](auto kernel, int features) {
    return launch_pdl(kernel, dim3(K / features * ts), dim3(256), kAppendSmem, stream, x, w, positions, scratch, p.batch, p.q_len,
                      p.hidden_dim, p.kv_lora_rank, p.qk_rope_dim, p.rope_theta, ts);
  };
  static_assert(skinny_gemm_smem(1, 4) <= kAppendSmem && skinny_gemm_smem(1, 2) <= kAppendSmem, "shared memory of the wide forms");
  cudaError_t e = T <= 48 ? rows(append_rows_f32_kernel<kAppendMaxMT, 1>, 8)
                          : T <= 64 ? rows(append_rows_f32_kernel<1, 2>, 16) : rows(append_rows_f32_kernel<1, 4>, 32);
  if (e != cudaSuccess) return e;
  return launch_pdl(quantize_rows_kernel, dim3((T + 3) / 4), dim3(128), static_cast<size_t>(0), stream,
                    static_cast<const float*>(scratch), positions, page_table, static_cast<unsigned char*>(cache_fp8), dev_status,
                    p.batch, p.q_len, p.num_pages, p.max_pages_per_seq);
}

}  // namespace transmla

// The merge of split partials by their lse (Eq. 9's softmax over a sequence's partitions), shared by the combine kernels.
#pragma once
#include "common.cuh"

namespace transmla {

struct MergeArgs {
  const int32_t* cum;        // the plan's prefix sums, then first and last partition of each sequence
  const int32_t* plan;
  const float* partial_o;    // segments of sequence b live in slots i + b for the partitions i that overlap its pages
  const float* partial_lse;
  int B, S, H, r, G;
};
// A warp merges rows bs_first, bs_first + bs_step .. (kAtOnce of them side by side) of head h: each lane kChunks pieces of four latents,
// 128 apart from c0 on.  kSegs partials of each row are in flight.  Rows beyond the last, and rows with nothing to merge, are 0.
template <int kAtOnce, int kChunks, int kSegs>
__device__ __forceinline__ void merge_rows(const MergeArgs& a, int h, int bs_first, int bs_step, int c0, float (&acc)[kAtOnce][kChunks][4],
                                           float (&lse)[kAtOnce]) {
  const int S = a.S, H = a.H, r = a.r, SH = S * H, BS = a.B * S, lane = threadIdx.x & 31;
  const int32_t* plan = a.plan;
  const float* partial_o = a.partial_o;
  const float* partial_lse = a.partial_lse;
  const long long T = a.cum[a.B];
  const bool dense = T >= a.G;  // then every partition owns at least one slot (of G at most)
  const int32_t* seq_parts = a.cum + a.B + 1;  // only 4-byte aligned: B + 1 may be odd
  int nseg[kAtOnce], i_first[kAtOnce], batch[kAtOnce], row[kAtOnce];
#pragma unroll
  for (int u = 0; u < kAtOnce; ++u) {
    const int bs = bs_first + bs_step * u;
    batch[u] = bs / S;
    row[u] = bs % S * H + h;
    i_first[u] = nseg[u] = 0;
    if (bs < BS) {
      i_first[u] = seq_parts[2 * batch[u]];
      nseg[u] = seq_parts[2 * batch[u] + 1] - i_first[u] + 1;
    }
  }
  auto seg_lse = [&](int u, int j) -> float {  // lse of the j-th candidate partition, -inf if it is empty or absent
    if (j >= nseg[u]) return -INFINITY;
    const int pi = i_first[u] + j;
    const float l = partial_lse[static_cast<size_t>(pi + batch[u]) * SH + row[u]];
    if (!dense) {
      const int2 range = *reinterpret_cast<const int2*>(plan + 4 * pi);
      if (range.y <= range.x) return -INFINITY;
    }
    return l;
  };
  float l_first[kAtOnce], m[kAtOnce], den[kAtOnce];
#pragma unroll
  for (int u = 0; u < kAtOnce; ++u) l_first[u] = seg_lse(u, lane);
  int most = 0;
#pragma unroll
  for (int u = 0; u < kAtOnce; ++u) {
    m[u] = l_first[u];
    for (int base = 32; base < nseg[u]; base += 32) m[u] = fmaxf(m[u], seg_lse(u, base + lane));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m[u] = fmaxf(m[u], __shfl_xor_sync(0xffffffffu, m[u], o));
    if (m[u] == -INFINITY) nseg[u] = 0;  // nothing to merge
    most = max(most, nseg[u]);
    den[u] = 0.f;
#pragma unroll
    for (int c = 0; c < kChunks; ++c) acc[u][c][0] = acc[u][c][1] = acc[u][c][2] = acc[u][c][3] = 0.f;
  }
  const size_t seg_stride = static_cast<size_t>(SH) * r;
#pragma unroll 1
  for (int base = 0; base < most; base += 32) {
    float wgt[kAtOnce];
    const float* po[kAtOnce];
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      const float l = base == 0 ? l_first[u] : seg_lse(u, base + lane);
      wgt[u] = nseg[u] > 0 && l > -INFINITY ? __expf(l - m[u]) : 0.f;
      den[u] += wgt[u];
      po[u] = partial_o + (static_cast<size_t>(i_first[u] + base + batch[u]) * SH + row[u]) * r + c0;
    }
    const int cnt = min(32, most - base);
    // the loads of a round overlap; a zero weight skips the (unwritten) slot
#pragma unroll 1
    for (int j0 = 0; j0 < cnt; j0 += kSegs) {
      float wj[kAtOnce][kSegs];
      float4 v[kAtOnce][kSegs][kChunks];
#pragma unroll
      for (int u = 0; u < kAtOnce; ++u)
#pragma unroll
        for (int q = 0; q < kSegs; ++q) {
          wj[u][q] = (j0 + q < cnt) ? __shfl_sync(0xffffffffu, wgt[u], (j0 + q) & 31) : 0.f;
#pragma unroll
          for (int c = 0; c < kChunks; ++c) {
            v[u][q][c] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (wj[u][q] != 0.f && c * 128 + c0 < r)
              v[u][q][c] = *reinterpret_cast<const float4*>(po[u] + (j0 + q) * seg_stride + c * 128);
          }
        }
#pragma unroll
      for (int u = 0; u < kAtOnce; ++u)
#pragma unroll
        for (int q = 0; q < kSegs; ++q)
#pragma unroll
          for (int c = 0; c < kChunks; ++c) {
            acc[u][c][0] = fmaf(wj[u][q], v[u][q][c].x, acc[u][c][0]); acc[u][c][1] = fmaf(wj[u][q], v[u][q][c].y, acc[u][c][1]);
            acc[u][c][2] = fmaf(wj[u][q], v[u][q][c].z, acc[u][c][2]); acc[u][c][3] = fmaf(wj[u][q], v[u][q][c].w, acc[u][c][3]);
          }
    }
  }
#pragma unroll
  for (int u = 0; u < kAtOnce; ++u) {
    float inv = 0.f;
    lse[u] = -INFINITY;
    if (nseg[u] > 0) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) den[u] += __shfl_xor_sync(0xffffffffu, den[u], o);
      inv = 1.f / den[u];
      lse[u] = m[u] + __logf(den[u]);
    }
#pragma unroll
    for (int c = 0; c < kChunks; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[u][c][e] *= inv;
  }
}

// The combine on the Blackwell tensor path (combine_sm100.cu).
bool combine_sm100_supported(const transmla_params_t& p);
cudaError_t launch_combine_sm100(const transmla_params_t& p, int G, const int32_t* cum, const int32_t* plan, const float* partial_o,
                                 const float* partial_lse, const __nv_bfloat16* w_uv, __nv_bfloat16* out, float* lse_out,
                                 int32_t* dev_status, cudaStream_t stream, bool give_up = false);

}  // namespace transmla

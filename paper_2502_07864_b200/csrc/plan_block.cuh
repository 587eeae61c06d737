// The split plan's block routine, shared by the kernels that hold a plan block.
#pragma once
#include "common.cuh"

namespace transmla {

// ------------------------------------------------------------------------------------------------
// Split plan.  Every non-empty sequence owns ceil(L_b/P) page slots preceded by kSegCost virtual slots (the
// price of opening a sequence); cum[b] = slots before sequence b; partition i owns slots
// [floor(i*T/G), floor((i+1)*T/G)), of the G that are planned (see plan_block); plan row = (begin, end, sequence of first slot, of last slot).
// One block of 256 threads; the scan runs in chunks of 256 sequences; the prefix sums are kept in
// shared memory (when they fit) for the binary searches.
// ------------------------------------------------------------------------------------------------
constexpr int kPlanSmemSeqs = 4096;

__device__ __forceinline__ int seq_of_page(const int32_t* cum, int B, int x) {
  // the b in [0, B) with cum[b] <= x < cum[b+1]  ==  (first index with cum > x) - 1
  int lo = 0, hi = B + 1;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (cum[mid] > x) hi = mid; else lo = mid + 1;
  }
  return lo - 1;
}

__device__ __forceinline__ void plan_block(const int32_t* seqlens, int B, Partitioning parts, int RB, int max_pages, int32_t* cum, int32_t* plan,
                           int32_t* dev_status, unsigned char* smem_raw) {
  __shared__ int warp_sums[8];
  __shared__ int carry;
  int32_t* cum_s = reinterpret_cast<int32_t*>(smem_raw);  // [B+1] when B < kPlanSmemSeqs
  const bool in_smem = B < kPlanSmemSeqs;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int sequences = 0;  // that are not empty
  pdl_wait();
  if (tid == 0) { carry = 0; cum[0] = 0; if (in_smem) cum_s[0] = 0; }
  __syncthreads();
  for (int base = 0; base < B; base += 256) {
    const int b = base + tid;
    int n = 0;
    if (b < B) { const int L = clamped_len(seqlens[b], max_pages, dev_status); n = L > 0 ? (L + kPage - 1) / kPage + kSegCost : 0; }
    int v = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { int t = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += t; }
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    int before = carry;
    for (int w = 0; w < warp; ++w) before += warp_sums[w];
    const int incl = v + before;
    if (b < B) { cum[b + 1] = incl; if (in_smem) cum_s[b + 1] = incl; }
    sequences += __syncthreads_count(n > 0);
    if (tid == 255) carry = incl;
    __syncthreads();
  }
  const int32_t* cs = in_smem ? cum_s : cum;
  const long long T = cs[B];
  const int G = parts.count(static_cast<int>(T) - kSegCost * sequences, sequences);
  for (int i = G + tid; i < parts.most; i += 256) reinterpret_cast<int4*>(plan)[i] = make_int4(0, 0, -1, -1);
  for (int i = tid; i < G; i += 256) {
    const int p0 = static_cast<int>((static_cast<long long>(i) * T) / G);
    const int p1 = static_cast<int>((static_cast<long long>(i + 1) * T) / G);
    int b0 = -1, b1 = -1;
    if (p1 > p0) { b0 = seq_of_page(cs, B, p0); b1 = seq_of_page(cs, B, p1 - 1); }
    reinterpret_cast<int4*>(plan)[i] = make_int4(p0, p1, b0, b1);
  }
  // Partitions that hold pages of sequence b: first and last index (0, -1 for an empty sequence), stored behind
  // the prefix sums so that the combine does not repeat the 64-bit divisions for every row and head.
  int32_t* seq_parts = cum + B + 1;
  for (int b = tid; b < B; b += 256) {
    const long long c0 = static_cast<long long>(cs[b]) + kSegCost, c1 = cs[b + 1];
    int i_first = 0, i_last = -1;
    if (c1 > c0) {
      i_first = static_cast<int>(((c0 + 1) * G - 1) / T);
      i_last = static_cast<int>((c1 * G - 1) / T);
    }
    seq_parts[2 * b] = i_first;
    seq_parts[2 * b + 1] = i_last;
  }
  // The page counters of the split-KV kernel start at zero.  Every earlier kernel of the stream has completed
  // here (the dependency wait above), so nobody is still counting.
  int32_t* next = cum + 3 * B + 1;
  for (int i = tid; i < RB * B; i += 256) next[i] = 0;
}

}  // namespace transmla

// Plan, absorb, append and combine kernels of the absorbed-MLA decode step.
//
// These touch a few MB (weights, queries, split partials) against the hundreds of MB the split-KV
// kernel streams.  They are small GEMMs with M = number of query rows or new tokens, latency bound
// rather than bandwidth bound, so they run on mma.sync tensor-core tiles, keep many independent
// 16-byte loads in flight, and are fused into as few launches as the data dependencies allow: one
// "prologue" launch holds the append blocks, the absorb blocks and the plan block.
//
// 16-byte operand loads: a lane (g, t) of an m16n8k16 tile needs k = 2t, 2t+1, 2t+8, 2t+9 of its row.
// A dot product does not care in which order k is visited as long as both operands agree, so both
// sides load the 8 consecutive elements 8t .. 8t+7 of a 32-wide k window with one uint4 and feed words
// (x, y) to one MMA and (z, w) to the next.  Where one operand comes from shared memory instead, it
// is stored there in the matching order (kperm below).
#include "append_block.cuh"
#include "combine.cuh"
#include "common.cuh"
#include "plan_block.cuh"
#include "skinny_gemm.cuh"

namespace transmla {

// Position, inside its 32-wide window, at which element p must sit in shared memory so that ldmatrix
// hands out the fragment that pairs with a uint4 global load of the other operand.
__device__ __forceinline__ int kperm(int p) { return ((p & 7) >> 1) * 8 + (p >> 3) * 2 + (p & 1); }

// ------------------------------------------------------------------------------------------------
// Absorb (Eq. 9 right, first line): q_hat[bs,h,:r] = W_UK_h^T q_nope[bs,h,:], q_hat[bs,h,r:] = q_pe[bs,h,:].
// A block owns nt consecutive 128-column tiles of one head's latent columns (nt = 1, or 2 when that brings the
// launch down to one wave): it stages W_UK_h[:, tiles] and the head's query rows (128 at a time) in shared
// memory with asynchronous 16-byte copies, all in flight together, and walks the rows in 16-row tiles, so W_UK
// is read once.  The block that owns a head's first tile also copies the rope part of the rows.
// ------------------------------------------------------------------------------------------------
constexpr int kAbsorbRows = 128;  // query rows staged per pass

template <int nt>
__device__ __forceinline__ void absorb_block(const __nv_bfloat16* q_nope, const __nv_bfloat16* q_pe,
                             const __nv_bfloat16* __restrict__ w_uk, __nv_bfloat16* q_hat, int BS, int H,
                             int dn, int dR, int r, int h, int rt0, unsigned char* smem_raw) {
  constexpr int wpitch = nt * 128 + 8, vec_per_row = nt * 16;
  const int apitch = dn + 8;
  __nv_bfloat16* w_s = reinterpret_cast<__nv_bfloat16*>(smem_raw);  // [dn][wpitch]
  __nv_bfloat16* a_s = w_s + dn * wpitch;                            // [kAbsorbRows][dn + 8]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3, mi = lane >> 3;
  const int n0 = rt0 * 128, K = r + dR;
  for (int i = tid; i < dn * vec_per_row; i += 256) {  // columns beyond r are zero-filled
    const int k = i / vec_per_row, c = i % vec_per_row;
    const bool in = n0 + c * 8 < r;
    cp_async16(w_s + k * wpitch + c * 8, w_uk + (static_cast<size_t>(h) * dn + k) * r + (in ? n0 + c * 8 : 0), in ? 16 : 0);
  }
  cp_async_commit();
  pdl_wait();  // the queries may come from the kernel before this one; the weights above may not
  const int chunks = dn / 8;
  for (int p0 = 0; p0 < BS; p0 += kAbsorbRows) {
    const int rows = min(kAbsorbRows, BS - p0);
    const int rows16 = (rows + 15) & ~15;
    if (p0 > 0) __syncthreads();  // previous pass has consumed a_s
    for (int i = tid; i < rows16 * chunks; i += 256) {  // rows beyond the last one are zero-filled
      const int rr = i / chunks, c = i % chunks;
      cp_async16(a_s + rr * apitch + c * 8, q_nope + (static_cast<size_t>(p0 + min(rr, rows - 1)) * H + h) * dn + c * 8,
                 rr < rows ? 16 : 0);
    }
    cp_async_commit();
    if (p0 == 0 && rt0 == 0 && dR > 0) {
      // the rope part is a plain copy, made while the operands of the first products are on their way
      if (dR % 8 == 0 && r % 8 == 0) {  // 16 bytes at a time, four copies in flight
        const int vecs = dR / 8;
        for (int i0 = tid; i0 < BS * vecs; i0 += 256 * 4) {
          uint4 v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 256, row = i / vecs, c = (i % vecs) * 8;
            v[u] = make_uint4(0, 0, 0, 0);
            if (i < BS * vecs) v[u] = ld_u128(q_pe + (static_cast<size_t>(row) * H + h) * dR + c);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 256, row = i / vecs, c = (i % vecs) * 8;
            if (i < BS * vecs) *reinterpret_cast<uint4*>(q_hat + (static_cast<size_t>(row) * H + h) * K + r + c) = v[u];
          }
        }
      } else {
        const int pairs = dR / 2;
        for (int i = tid; i < BS * pairs; i += 256) {
          const int row = i / pairs, c = (i % pairs) * 2;
          *reinterpret_cast<uint32_t*>(q_hat + (static_cast<size_t>(row) * H + h) * K + r + c) =
              ld_u32(q_pe + (static_cast<size_t>(row) * H + h) * dR + c);
        }
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    for (int m0 = 0; m0 < rows16; m0 += 16) {
#pragma unroll 1
      for (int wc = warp * 16 * nt; wc < (warp + 1) * 16 * nt; wc += 16) {  // this warp's 16-column steps
        float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 4
        for (int ks = 0; ks < dn / 16; ++ks) {
          uint32_t a[4], bf[4];
          ldmatrix_x4(a, a_s + (m0 + (mi & 1) * 8 + (lane & 7)) * apitch + ks * 16 + (mi >> 1) * 8);
          ldmatrix_x4_trans(bf, w_s + (ks * 16 + (mi & 1) * 8 + (lane & 7)) * wpitch + wc + (mi >> 1) * 8);
          mma_bf16_16816(acc[0], a, bf[0], bf[1]);
          mma_bf16_16816(acc[1], a, bf[2], bf[3]);
        }
        const int r0 = p0 + m0 + g, r1 = r0 + 8;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int col = n0 + wc + j * 8 + t4 * 2;
          if (col < r) {
            if (r0 < BS) *reinterpret_cast<uint32_t*>(q_hat + (static_cast<size_t>(r0) * H + h) * K + col) = pack_bf16(acc[j][0], acc[j][1]);
            if (r1 < BS) *reinterpret_cast<uint32_t*>(q_hat + (static_cast<size_t>(r1) * H + h) * K + col) = pack_bf16(acc[j][2], acc[j][3]);
          }
        }
      }
    }
  }
}

static size_t absorb_smem(int dn, int nt) {
  return (static_cast<size_t>(dn) * (nt * 128 + 8) + static_cast<size_t>(kAbsorbRows) * (dn + 8)) * sizeof(__nv_bfloat16);
}

// Tiles per absorb block: two when the prologue launch would otherwise not fit the device in one wave of one block
// per SM (the append's accumulators allow no more), the tile count is even and the pair's weights fit.
static int absorb_tiles_per_block(const transmla_params_t& p, int other_blocks) {
  static PerDeviceFlag sms_of;  // SM count per device, asked once
  const int slot = current_device_slot();
  int sms = slot >= 0 ? sms_of.value[slot].load(std::memory_order_acquire) : 0;
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return 1;
    }
    if (slot >= 0) sms_of.value[slot].store(sms, std::memory_order_release);
  }
  const int r_tiles = (p.kv_lora_rank + 127) / 128;
  const bool fits_one = other_blocks + p.num_heads * r_tiles <= sms;
  return (!fits_one && r_tiles % 2 == 0 && p.qk_nope_dim <= 128) ? 2 : 1;
}

// The append of sizes that prologue_sm100.cu does not take goes by clusters (see slice_gemm_tile) or by blocks.
__global__ void __launch_bounds__(256, 2) append_cluster_kernel(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ w,
                                                                const int32_t* positions, const int32_t* page_table,
                                                                __nv_bfloat16* cache, int32_t* dev_status, int B, int S, int D,
                                                                int r, int dR, int num_pages, int max_pages, float theta) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  append_cluster(x, w, positions, 0, page_table, cache, dev_status, B, S, D, r, dR, num_pages, max_pages, theta,
                 blockIdx.x / kSliceCtas, blockIdx.x % kSliceCtas, smem_raw);
}
__global__ void __launch_bounds__(256) append_kernel(const __nv_bfloat16* x,
                                                     const __nv_bfloat16* __restrict__ w,
                                                     const int32_t* positions,
                                                     const int32_t* page_table,
                                                     __nv_bfloat16* cache, int32_t* dev_status, int B,
                                                     int S, int D, int r, int dR, int num_pages, int max_pages,
                                                     float theta, int t_splits, int wide) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  if (wide)
    append_block<1, 4>(x, w, positions, 0, page_table, cache, dev_status, B, S, D, r, dR, num_pages, max_pages, theta,
                       blockIdx.x, t_splits, smem_raw);
  else
    append_block<kAppendMaxMT, 1>(x, w, positions, 0, page_table, cache, dev_status, B, S, D, r, dR, num_pages, max_pages,
                                  theta, blockIdx.x, t_splits, smem_raw);
}

// Absorb blocks followed by one plan block: everything transmla_mla_decode needs before the split-KV kernel.
template <int nt>
__global__ void __launch_bounds__(256) absorb_plan_kernel(const __nv_bfloat16* q_nope,
                                                          const __nv_bfloat16* q_pe,
                                                          const __nv_bfloat16* __restrict__ w_uk,
                                                          __nv_bfloat16* q_hat,
                                                          const int32_t* seqlens, int32_t* cum,
                                                          int32_t* plan, int32_t* dev_status, int B, int S, int H,
                                                          int dn, int dR, int r, Partitioning parts, int max_pages) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  const int per_head = (r + 127) / 128 / nt;  // absorb blocks per head, nt tiles each
  const int n_absorb = H * per_head;
  if (static_cast<int>(blockIdx.x) < n_absorb) {
    absorb_block<nt>(q_nope, q_pe, w_uk, q_hat, B * S, H, dn, dR, r, blockIdx.x / per_head, blockIdx.x % per_head * nt, smem_raw);
  } else {
    plan_block(seqlens, B, parts, (S * H + kRowBlock - 1) / kRowBlock, max_pages, cum, plan, dev_status, smem_raw);
  }
}

// The whole prologue of a decode step in one launch: append clusters or blocks, plan block, absorb blocks.
// The appended token of sequence b sits at seqlens[b] - S + s.  n_append: clusters, or blocks of t_splits token splits.
template <bool kClusters, int nt>
__global__ void __launch_bounds__(256, kClusters ? 2 : 1) prologue_kernel(
    const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ w_dkv_kr,
    const int32_t* page_table, __nv_bfloat16* cache, const __nv_bfloat16* q_nope,
    const __nv_bfloat16* q_pe, const __nv_bfloat16* __restrict__ w_uk, __nv_bfloat16* q_hat,
    const int32_t* seqlens, int32_t* cum, int32_t* plan, int32_t* dev_status, int B, int S, int H, int D,
    int dn, int dR, int r, int num_pages, int max_pages, float theta, Partitioning parts, int n_append, int t_splits, int wide) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  const int per_head = (r + 127) / 128 / nt;  // absorb blocks per head, nt tiles each
  const int bid = static_cast<int>(blockIdx.x) - n_append * (kClusters ? kSliceCtas : 1);
  if (bid < 0) {
    if (kClusters)
      append_cluster(x, w_dkv_kr, seqlens, -S, page_table, cache, dev_status, B, S, D, r, dR, num_pages, max_pages, theta,
                     blockIdx.x / kSliceCtas, blockIdx.x % kSliceCtas, smem_raw);
    else if (wide)
      append_block<1, 4>(x, w_dkv_kr, seqlens, -S, page_table, cache, dev_status, B, S, D, r, dR, num_pages, max_pages,
                         theta, blockIdx.x, t_splits, smem_raw);
    else
      append_block<kAppendMaxMT, 1>(x, w_dkv_kr, seqlens, -S, page_table, cache, dev_status, B, S, D, r, dR, num_pages,
                                    max_pages, theta, blockIdx.x, t_splits, smem_raw);
  } else if (bid == 0) {
    plan_block(seqlens, B, parts, (S * H + kRowBlock - 1) / kRowBlock, max_pages, cum, plan, dev_status, smem_raw);
  } else if (bid <= H * per_head) {  // (a grid of clusters is whole: a few blocks at its end have nothing to do)
    absorb_block<nt>(q_nope, q_pe, w_uk, q_hat, B * S, H, dn, dR, r, (bid - 1) / per_head, (bid - 1) % per_head * nt, smem_raw);
  }
}

constexpr int kPrologueMaxSmem = 144 * 1024;

// Token splits of the append's blocks.  With many new tokens a block takes 32 output features and 16 tokens (activations re-read
// a quarter as often per feature, weights four times as often per token: 384 KB per block instead of 576 KB at 128 tokens).
// Otherwise 8 features: one split per 64 tokens, at most 4.
bool append_wide(const transmla_params_t& p) {
  return p.batch * p.q_len > 32 && (p.kv_lora_rank + p.qk_rope_dim) % 32 == 0 && p.kv_lora_rank % 2 == 0;
}
int append_token_splits(const transmla_params_t& p) {
  const int T = p.batch * p.q_len;
  if (append_wide(p)) return (T + 15) / 16 > 32 ? 32 : (T + 15) / 16;
  return T <= 64 ? 1 : (T + 63) / 64 > 4 ? 4 : (T + 63) / 64;
}
// Clusters read the operands a quarter as often but take 2 to 3 us more to start and to meet.  The decode step, blocks / clusters:
// r = 64, dR = 16, D = 256 1 sequence 14.0 / 15.2 us, 16 (64 heads) 16.6 / 19.0, 64 18.0 to 23.2 / 19.3 to 25.3; the same with D = 4096 16
// 20.6 / 21.9, 64 27.7 / 21.2; r = 512, dR = 64, dn = 64 1 20.6 / 22.2, 16 22.2 / 24.6, 160 46.1 / 39.5 and (64 heads) 75.4 / 69.8.  With
// r = 128, dR = 0 blocks of 32 features x 16 tokens are as many as clusters have CTAs: 16 19.1 / 22.2, 64 22.5 / 22.9, 160 23.8 / 26.3.
// An append call is followed by the decode's absorb, which starts earlier beside clusters: with it and the combine, 100 cached tokens,
// blocks / clusters: r = 512, dn = 64 16 tokens 25.7 / 30.7, 32 31.2 / 30.2, 128 51.2 / 46.2; r = 128 16 21.1 / 23.7, 32 26.3 / 24.2; r = 64, D = 4096
// 16 20.1 / 23.4, 32 26.9 / 23.4; D = 256 16 18.9 / 19.7, 32 19.4 / 20.0.  (By themselves blocks stay ahead up to 256 tokens of r = 512: 128
// tokens 6.8 / 10.0.  The two forms add a value's products in other orders, both in fp32.)
static bool append_in_clusters(const transmla_params_t& p, bool alone) {
  const int T = p.batch * p.q_len;
  return alone ? T > 16 : T > 32 && (p.kv_lora_rank + p.qk_rope_dim) % 128 != 0;
}

cudaError_t launch_append(const transmla_params_t& p, const __nv_bfloat16* x, const __nv_bfloat16* w,
                          const int32_t* positions, const int32_t* page_table, __nv_bfloat16* cache,
                          int32_t* dev_status, cudaStream_t stream) {
  const int K = p.kv_lora_rank + p.qk_rope_dim;
  if (prologue_sm100_supported(p))
    return launch_append_sm100(p, x, w, positions, page_table, cache, nullptr, dev_status, stream);
  if (append_in_clusters(p, true)) {
    static PerDeviceFlag smem_set;
    if (cudaError_t e = ensure_dynamic_smem(append_cluster_kernel, static_cast<int>(kSliceSmem), smem_set); e != cudaSuccess) return e;
    return launch_slices(append_cluster_kernel, append_clusters(p) * kSliceCtas, kSliceSmem, stream, x, w, positions, page_table, cache,
                         dev_status, p.batch, p.q_len, p.hidden_dim, p.kv_lora_rank, p.qk_rope_dim, p.num_pages,
                         p.max_pages_per_seq, p.rope_theta);
  }
  const int ts = append_token_splits(p);
  const int wide = append_wide(p) ? 1 : 0;
  return launch_pdl(append_kernel, dim3(K / (wide ? 32 : 8) * ts), dim3(256), kAppendSmem, stream, x, w, positions, page_table,
                    cache, dev_status, p.batch, p.q_len, p.hidden_dim, p.kv_lora_rank, p.qk_rope_dim, p.num_pages,
                    p.max_pages_per_seq, p.rope_theta, ts, wide);
}

cudaError_t launch_absorb_plan(const transmla_params_t& p, const Partitioning& parts, const __nv_bfloat16* q_nope,
                               const __nv_bfloat16* q_pe, const __nv_bfloat16* w_uk, __nv_bfloat16* q_hat,
                               const int32_t* seqlens, int32_t* cum, int32_t* plan, int32_t* dev_status,
                               bool behind_maps, cudaStream_t stream) {
  // Few rows behind a launch of linear maps: the maps' CTAs leave some SMs free, where more and shorter blocks end sooner
  // (layer step, mma.sync / tcgen05: 1 token 47.1 / 47.6 us, 16 70.5 / 71.9, 32 75.6 / 76.0, 48 91.1 / 90.1, 64 91.0 / 85.1; 64
  // heads: 8 99.6 / 101.3, 32 118.2 / 118.5, 64 145.4 / 143.2; behind the FP8 append: 4 35.7 / 35.6, 16 55.2 / 52.0).
  const bool sm100 = prologue_sm100_supported(p);
  if (sm100 && !(behind_maps && p.batch * p.q_len <= 32))
    return launch_absorb_sm100(p, parts, nullptr, nullptr, nullptr, nullptr, q_nope, q_pe, w_uk, q_hat, seqlens, cum, plan, dev_status, stream);
  const int nt = sm100 ? 1 : absorb_tiles_per_block(p, 1);
  size_t smem = absorb_smem(p.qk_nope_dim, nt);
  if (smem < kPlanSmemSeqs * sizeof(int32_t)) smem = kPlanSmemSeqs * sizeof(int32_t);
  static PerDeviceFlag smem_set[2];  // zero-initialised; one slot per device
  auto kernel = nt == 2 ? absorb_plan_kernel<2> : absorb_plan_kernel<1>;
  if (cudaError_t e = ensure_dynamic_smem(kernel, kPrologueMaxSmem, smem_set[nt - 1]); e != cudaSuccess) return e;
  const int blocks = p.num_heads * ((p.kv_lora_rank + 127) / 128 / nt) + 1;
  return launch_pdl(kernel, dim3(blocks), dim3(256), smem, stream, q_nope, q_pe, w_uk, q_hat, seqlens, cum,
                    plan, dev_status, p.batch, p.q_len, p.num_heads, p.qk_nope_dim, p.qk_rope_dim, p.kv_lora_rank, parts,
                    p.max_pages_per_seq);
}

cudaError_t launch_prologue(const transmla_params_t& p, const Partitioning& parts, const __nv_bfloat16* x, const __nv_bfloat16* w_dkv_kr,
                            const int32_t* page_table, __nv_bfloat16* cache, const __nv_bfloat16* q_nope,
                            const __nv_bfloat16* q_pe, const __nv_bfloat16* w_uk, __nv_bfloat16* q_hat,
                            const int32_t* seqlens, int32_t* cum, int32_t* plan, int32_t* dev_status,
                            cudaStream_t stream) {
  if (prologue_sm100_supported(p))
    return launch_absorb_sm100(p, parts, x, w_dkv_kr, page_table, cache, q_nope, q_pe, w_uk, q_hat, seqlens, cum, plan, dev_status, stream);
  const bool clusters = append_in_clusters(p, false);
  const int ts = append_token_splits(p), wide = append_wide(p) ? 1 : 0;
  const int n_append = clusters ? append_clusters(p) : (p.kv_lora_rank + p.qk_rope_dim) / (wide ? 32 : 8) * ts;
  const int nt = clusters ? 1 : absorb_tiles_per_block(p, 1 + n_append);
  const int others = 1 + p.num_heads * ((p.kv_lora_rank + 127) / 128 / nt);
  const size_t smem_append = clusters ? kSliceSmem : kAppendSmem;
  size_t smem = absorb_smem(p.qk_nope_dim, nt);
  if (smem < smem_append) smem = smem_append;
  static PerDeviceFlag smem_set[3];  // zero-initialised; one slot per device
  auto kernel = clusters ? prologue_kernel<true, 1> : nt == 2 ? prologue_kernel<false, 2> : prologue_kernel<false, 1>;
  if (cudaError_t e = ensure_dynamic_smem(kernel, kPrologueMaxSmem, smem_set[clusters ? 2 : nt - 1]); e != cudaSuccess) return e;
  auto with_args = [&](auto launch) {
    return launch(x, w_dkv_kr, page_table, cache, q_nope, q_pe, w_uk, q_hat, seqlens, cum, plan, dev_status, p.batch, p.q_len,
                  p.num_heads, p.hidden_dim, p.qk_nope_dim, p.qk_rope_dim, p.kv_lora_rank, p.num_pages, p.max_pages_per_seq,
                  p.rope_theta, parts, n_append, ts, wide);
  };
  if (clusters)
    return with_args([&](auto... a) { return launch_slices(kernel, (n_append + (others + kSliceCtas - 1) / kSliceCtas) * kSliceCtas, smem, stream, a...); });
  return with_args([&](auto... a) { return launch_pdl(kernel, dim3(n_append + others), dim3(256), smem, stream, a...); });
}

// ------------------------------------------------------------------------------------------------
// Combine + up-projection (Eq. 9 right, last line before W_O).  Block = one head x kRows query rows
// x (optionally) one half of the dv output columns.
// Phase 1: each warp merges the split partials of its rows (or of half a row's latents) by their lse (segments of sequence b
// live in slots i + b for the partitions i that overlap its pages) into shared memory as a bf16 hi/lo
// pair, so that the tensor-core product of phase 2 carries fp32-like precision of o_hat.  The merged
// rows are stored in kperm order.
// Phase 2: out[rows, h, :]^T = W_UV_h o_hat^T with W_UV_h read straight from global memory, 16 bytes per lane: 16 output
// columns a warp are the M of its products, 8 query rows the N.
// What bounds it is a chain of round trips to L2 (look-ups of the row's partitions, their lse, the partials, the weights; a
// partial's is 2000 to 3000 cycles with all blocks asking), then the mma.sync products, 16 cycles each on an SM's quarter:
// with the rows as M, 16 of which 4 to 8 were there, and one accumulator for all, they took 3000 to 6400 cycles a tile.
// ------------------------------------------------------------------------------------------------
// kPrefetch: hold the weights in registers from before the dependency wait, one block per SM; otherwise load them
// between the phases and keep the register count low enough for two blocks per SM.
template <int kRows, int kHalves, bool kPrefetch>
__global__ void __launch_bounds__(256, kPrefetch ? 1 : 2) combine_kernel(const int32_t* cum,
                                                      const int32_t* plan,
                                                      const float* partial_o,
                                                      const float* partial_lse,
                                                      const __nv_bfloat16* __restrict__ w_uv,
                                                      __nv_bfloat16* out, float* lse_out,
                                                      int B, int S, int H, int r, int dv, int G) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kWarpsPerRow = kRows < 8 ? 8 / kRows : 1;
  constexpr int kAtOnce = kRows > 8 ? 2 : 1;                    // rows a warp merges side by side
  constexpr int kChunks = 4 / kWarpsPerRow;                     // 128-latent chunks of a row a warp merges
  constexpr int kSegs = (kPrefetch ? 20 : 16) / (kAtOnce * kChunks);  // partials of each row in flight
  constexpr int kWin = kPrefetch ? 16 : 16 / kHalves;           // windows of 32 latents whose weights are in registers at once
  constexpr int kRowTiles = (kRows + 7) / 8;
  const int pitch = r + 8;
  __nv_bfloat16* o_hi = reinterpret_cast<__nv_bfloat16*>(smem_raw);                 // [kRows, 8 at least][pitch]
  __nv_bfloat16* o_lo = o_hi + (kRows < 8 ? 8 : kRows) * pitch;
  pdl_trigger();
  const int h = blockIdx.x, bs0 = blockIdx.y * kRows;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int SH = S * H, BS = B * S;
  const int g = lane >> 2, t4 = lane & 3, mi = lane >> 3;
  // kHalves = 2: tiles of 16 output columns, the block has all of them; 1: of 8 (M is half empty), it has half of them.
  const int tiles = dv / 8, tiles_per_z = (tiles + gridDim.z - 1) / gridDim.z;
  const int nt_lo = blockIdx.z * tiles_per_z, nt_hi = min(tiles, nt_lo + tiles_per_z);
  uint4 wv[kHalves][kWin];
  auto load_weights = [&](int nt, int w0) {
#pragma unroll
    for (int j = 0; j < kHalves; ++j) {
      const __nv_bfloat16* wrow = w_uv + (static_cast<size_t>(h) * dv + min(nt + j, tiles - 1) * 8 + g) * r + t4 * 8;
#pragma unroll
      for (int u = 0; u < kWin; ++u)
        wv[j][u] = (nt + j < nt_hi && w0 + u * 32 < r) ? ld_u128(wrow + w0 + u * 32) : make_uint4(0, 0, 0, 0);
    }
  };
  const int nt_first = nt_lo + warp * kHalves;
  // The weights do not depend on the merge: they are asked for now and land while the partials are merged.
  if (kPrefetch) load_weights(nt_first, 0);
  else {
    const __nv_bfloat16* w = w_uv + (static_cast<size_t>(h) * dv + nt_lo * 8) * r;
    for (int i = tid * 64; i < (nt_hi - nt_lo) * 8 * r; i += 256 * 64) prefetch_l2(w + i);
  }
  pdl_wait();  // the partials and the prefix sums come from the kernels before this one
  const long long T = cum[B];
  const bool dense = T >= G;  // then every partition owns at least one slot (of G at most)
  const int32_t* seq_parts = cum + B + 1;  // only 4-byte aligned: B + 1 may be odd

  // (The merge is merge_rows of combine.cuh written out, and what changes in one changes in both.  As one routine, with the sums handed
  // back or taken by a callback, the compiler's schedule costs 2 to 10 % of the launch: the step of 16 x 8192 45.7 -> 46.0 and 46.1 us, of 32
  // ragged sequences 127.2 -> 128.9 and 128.5.)
#pragma unroll 1
  for (int r0 = warp / kWarpsPerRow; r0 < kRows; r0 += 8 * kAtOnce) {
    const int c0 = kWarpsPerRow > 1 ? warp % kWarpsPerRow * (kChunks * 128) + lane * 4 : lane * 4;  // the lane's first latent
    int nseg[kAtOnce], i_first[kAtOnce], batch[kAtOnce], row[kAtOnce];
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      const int bs = bs0 + r0 + 8 * u;
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
    float l_first[kAtOnce], m[kAtOnce], den[kAtOnce], acc[kAtOnce][kChunks][4];
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
      float inv = 0.f, lse = -INFINITY;
      if (nseg[u] > 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) den[u] += __shfl_xor_sync(0xffffffffu, den[u], o);
        inv = 1.f / den[u];
        lse = m[u] + __logf(den[u]);
      }
      const int rr = r0 + 8 * u;
      if (lse_out != nullptr && lane == 0 && warp % kWarpsPerRow == 0 && blockIdx.z == 0 && bs0 + rr < BS)
        lse_out[static_cast<size_t>(bs0 + rr) * H + h] = lse;
#pragma unroll
      for (int c = 0; c < kChunks; ++c) {
        const int k = c * 128 + c0;
        if (k < r) {
          float v[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            v[e] = acc[u][c][e] * inv;
            lo[e] = v[e] - __bfloat162float(__float2bfloat16_rn(v[e]));
          }
          const int win = k & ~31, p = k & 31;  // elements p..p+3 of the window: two pairs, each stays adjacent
          const int q0 = win + kperm(p), q1 = win + kperm(p + 2);
          *reinterpret_cast<uint32_t*>(o_hi + rr * pitch + q0) = pack_bf16(v[0], v[1]);
          *reinterpret_cast<uint32_t*>(o_hi + rr * pitch + q1) = pack_bf16(v[2], v[3]);
          *reinterpret_cast<uint32_t*>(o_lo + rr * pitch + q0) = pack_bf16(lo[0], lo[1]);
          *reinterpret_cast<uint32_t*>(o_lo + rr * pitch + q1) = pack_bf16(lo[2], lo[3]);
        }
      }
    }
  }
  if (!kPrefetch) load_weights(nt_first, 0);
  __syncthreads();

  // (Rows 4 to 7 of a block that has 4 are whatever is there: nothing of them is stored, and a product's rows do not mix.)
  for (int nt = nt_first; nt < nt_hi; nt += 8 * kHalves) {
    float acc[kRowTiles][2][4];  // high and low part apart: two chains
#pragma unroll
    for (int n = 0; n < kRowTiles; ++n)
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[n][e >> 2][e & 3] = 0.f;
#pragma unroll 1
    for (int w0 = 0; w0 < r; w0 += kWin * 32) {
      if (nt != nt_first || w0 != 0) load_weights(nt, w0);
#pragma unroll
      for (int u = 0; u < kWin; ++u) {
        if (w0 + u * 32 < r) {
          const uint4 wa = wv[0][u], wb = kHalves == 2 ? wv[kHalves - 1][u] : make_uint4(0, 0, 0, 0);
          const uint32_t a0[4] = {wa.x, wb.x, wa.y, wb.y}, a1[4] = {wa.z, wb.z, wa.w, wb.w};
#pragma unroll
          for (int n = 0; n < kRowTiles; ++n) {
            uint32_t hi[4], lo[4];
            const int off = (n * 8 + (lane & 7)) * pitch + w0 + u * 32 + mi * 8;
            ldmatrix_x4(hi, o_hi + off);
            ldmatrix_x4(lo, o_lo + off);
            mma_bf16_16816(acc[n][0], a0, hi[0], hi[1]);
            mma_bf16_16816(acc[n][1], a0, lo[0], lo[1]);
            mma_bf16_16816(acc[n][0], a1, hi[2], hi[3]);
            mma_bf16_16816(acc[n][1], a1, lo[2], lo[3]);
          }
        }
      }
    }
    // A lane has columns g and (second half) g + 8 of rows 2 t4 and 2 t4 + 1: neighbouring columns meet by an exchange.
#pragma unroll
    for (int n = 0; n < kRowTiles; ++n) {
#pragma unroll
      for (int j = 0; j < kHalves; ++j) {
        const float v0 = acc[n][0][2 * j] + acc[n][1][2 * j], v1 = acc[n][0][2 * j + 1] + acc[n][1][2 * j + 1];
        // even g keeps row 2 t4, odd g row 2 t4 + 1, each of columns g & ~1 and g | 1
        const float got = __shfl_xor_sync(0xffffffffu, g & 1 ? v0 : v1, 4);
        const int rr = n * 8 + 2 * t4 + (g & 1), col = (nt + j) * 8 + (g & ~1);
        if (nt + j < nt_hi && rr < kRows && bs0 + rr < BS)
          *reinterpret_cast<uint32_t*>(out + (static_cast<size_t>(bs0 + rr) * H + h) * dv + col) =
              g & 1 ? pack_bf16(got, v1) : pack_bf16(v0, got);
      }
    }
  }
}

cudaError_t launch_combine(const transmla_params_t& p, int G, const int32_t* cum, const int32_t* plan, const float* partial_o,
                           const float* partial_lse, const __nv_bfloat16* w_uv, __nv_bfloat16* out, float* lse_out,
                           int32_t* dev_status, cudaStream_t stream) {
  const int BS = p.batch * p.q_len, H = p.num_heads;
  constexpr int kSms = 148;
  auto blocks = [&](int rows) { return static_cast<long long>(H) * ((BS + rows - 1) / rows); };
  auto launch = [&](auto kernel, int rows, int halves) {
    const size_t smem = 2 * (rows < 8 ? 8 : rows) * (p.kv_lora_rank + 8) * sizeof(__nv_bfloat16);
    return launch_pdl(kernel, dim3(H, (BS + rows - 1) / rows, halves), dim3(256), smem, stream, cum, plan, partial_o, partial_lse, w_uv,
                      out, lse_out, p.batch, p.q_len, H, p.kv_lora_rank, p.v_dim, G);
  };
  // Up to one wave of blocks.  Four rows a block, two warps a row, merge sooner than eight; two halves of dv read half of W_UV_h each,
  // which is what is left to wait for where the merge is short.  Both while twice the blocks of four fit; beyond that eight rows and
  // halves where a row has few partials, otherwise four rows and all of dv.  The step of 32 heads, dv = 128, 4 rows / 8 rows: 9
  // sequences (at most G / batch = 4, 8, 16, 16 partials) of 1000 25.3 / 22.4 us, 2000 23.4 / 23.2, 4000 25.6 / 26.1, 16384 44.4 / 45.1; 13 (3, 11) of 300
  // 26.6 / 25.1, 16384 55.0 / 55.0; 16 (9) of 8192 46.5 / 45.8; S = 2, 5 sequences (4, 30) of 1000 25.4 / 22.5, 16384 39.3 / 41.1; 64 heads, 8 of 300 (1)
  // 26.7 / 25.4, 40000 (18) 77.1 / 77.8.  (The table's room stands for the lengths: with room for 128K 9 x 300 takes 23.2 where 8 rows
  // would take 21.6.)  With dv <= 64 a warp has one tile of columns as it is, and few rows leave more SMs to the launches either
  // side: dv = 64, append + decode + combine of 4 sequences of 100 27.8 us (4 rows, all of dv), 26.7 (halves), 25.2.
  if (p.v_dim >= 128 && 2 * blocks(4) <= kSms) return launch(combine_kernel<4, 1, true>, 4, 2);
  if (p.v_dim <= 64 && BS <= 32 && blocks(8) <= kSms) return launch(combine_kernel<8, 1, true>, 8, 1);
  if (2 * blocks(8) <= kSms && (G <= 12LL * p.batch || blocks(4) > kSms)) return launch(combine_kernel<8, 1, true>, 8, 2);
  if (blocks(4) <= kSms) return launch(combine_kernel<4, 2, true>, 4, 1);
  if (blocks(8) <= kSms) return launch(combine_kernel<8, 2, true>, 8, 1);
  if (combine_sm100_supported(p)) return launch_combine_sm100(p, G, cum, plan, partial_o, partial_lse, w_uv, out, lse_out, dev_status, stream);
  // (8 warps x 16 columns are 128 of dv: while a wave of two blocks an SM has room, dv = 256 goes in halves.  32 heads x 64 rows, the
  // step of 300 and 4000 cached tokens: 40.4 and 79.6 us -> 32.4 and 72.6; with more blocks it costs: x 128 rows 17.3 -> 21.1 alone.)
  return launch(combine_kernel<16, 2, false>, 16, p.v_dim > 128 && blocks(16) <= kSms ? 2 : 1);
}

}  // namespace transmla

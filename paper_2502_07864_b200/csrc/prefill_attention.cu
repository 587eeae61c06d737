// Causal attention of a chunk of query positions over the decompressed keys and values (Eq. 9 left): prefill in
// the MHA form, per head  z = q_nope . k^C + q_pe . k^R,  softmax,  sum p v.
//
// One CTA = two tiles of 128 query positions (or one, see the launch) x one head x one sequence.  Per 64-token page and tile
//   S [128 x 64]  = Q x [k^C | k^R]^T, K = 192 (a third of Q from tensor memory, the rest and the page from shared memory)
//   O [128 x 128] += P (tensor memory, bf16) x V (shared memory, MN-major)
// What bounds it: the products need 640 cycles a tile and page, 780 with two thirds of Q from shared memory, and the
// exponentials 512 (16 a cycle); softmax of one tile runs beside the products of the other and the scores of its own next
// page.  Eight softmax warps a tile: a thread has half a row, 32 scores.  One tile of four softmax warps took
// 1620 cycles a page; now two tiles take 2100 together (the chain scores, softmax 1250, products): 64 pages x 256 CTAs of
// the S = 512 chunk over 4 x 8192 tokens 400 -> 287 us, 12 sequences of 1900 positions 2000 -> 1383 us.
// Tensor memory: Q 2 x 32 columns, S 2 x 64, P 2 x 32, O 2 x 128 = 512, which is why most of Q is not there.
// The pair of threads that share a row use one reference maximum, which moves only when a score exceeds it by 2^8: a vote
// of the two warps per page, values exchanged only then.
// Each tile has a warp that issues its scores and products; what it issues the tensor pipe works in that order.
// k^C and v come from the decompressed store (row page*64 + slot, columns h*256 ..), k^R from the latent cache
// itself (columns 512..575 of the same row), all through the page table.
// Warps 0-15 softmax + write-out (tile w / 8, half w / 4 % 2, tensor-memory lanes 32 (w % 4)..), 16 TMA, 17 and 18 products.
// Bounded waits throughout.
#include "prefill.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace prefill {

using namespace sm100;

constexpr int R_ = 512, DR_ = 64, DN_ = 128, DV_ = 128;
constexpr int kQRows = 128, kTiles = 2;
constexpr int kSub64 = kPage * 128;                // 8192: 64 tokens x 128 bytes
constexpr int kQSub = kQRows * 128;                // 16384: 128 query rows x 128 bytes
constexpr int kKvStage = 5 * kSub64;               // k^C (2) | k^R (1) | v (2) = 40960
constexpr int kKvStages = 4;
constexpr int kSoftmaxWarps = 16, kAttnThreads = (kSoftmaxWarps + 3) * 32;
// Q's sub-tiles: columns 0-63 of q_nope pass through ring stage 0 into tensor memory, 64-127 and q_pe stay in shared memory
constexpr int kOffQ = 0, kOffKv = kTiles * 2 * kQSub, kOffBarA = kOffKv + kKvStages * kKvStage, kOffMiscA = kOffBarA + 256;
constexpr int kAttnSmem = kOffMiscA + 2048 + 64;  // misc: row maxima [tile][half][128] f32, tensor-memory base, abort
static_assert(kOffBarA % 256 == 0 && kAttnSmem <= 232448, "shared memory map");
static_assert(kTiles * kQSub <= kKvStage, "q_nope staging");
constexpr uint32_t kColQ = 0, kColS = 64, kColP = 192, kColO = 256;  // Q 2 x 32, S 2 x 64, P 2 x 32, O 2 x 128
enum { A_KV_FULL = 0, A_KV_EMPTY = A_KV_FULL + kKvStages, A_Q_READY = A_KV_EMPTY + kKvStages, A_S_FULL, A_S_FREE = A_S_FULL + kTiles,
       A_P_READY = A_S_FREE + kTiles, A_PV_DONE = A_P_READY + kTiles };

__host__ __device__ constexpr uint32_t idesc_attn(int m, int n, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn ? 1u : 0u) << 16) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(m >> 4) << 24);
}
__global__ void __launch_bounds__(kAttnThreads, 1)
prefill_attention_kernel(const __grid_constant__ CUtensorMap qn_map, const __grid_constant__ CUtensorMap qr_map,
                         const __grid_constant__ CUtensorMap kv_map, const __grid_constant__ CUtensorMap cache_map,
                         const int32_t* page_table, const int32_t* seqlens, __nv_bfloat16* out, float* lse_out,
                         int32_t* dev_status, int S, int H, int num_pages, int max_pages, float scale_log2, int cta_tiles) {
  extern __shared__ __align__(1024) unsigned char smem_aligned[];  // no room to align by hand
  unsigned char* sm = smem_aligned;
  const uint32_t base = smem_u32(sm);
  if ((base & 1023u) != 0) { set_status(dev_status, TRANSMLA_DEV_TIMEOUT); return; }
  float* row_s = reinterpret_cast<float*>(sm + kOffMiscA);   // [tile][half][128]
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(sm + kOffMiscA + 2048);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  auto bar = [&](int i) -> uint32_t { return base + kOffBarA + 8 * i; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int qt = gridDim.x - 1 - blockIdx.x, h = blockIdx.y, b = blockIdx.z;   // the tiles that see most first
  pdl_trigger();
  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&qn_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&qr_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&kv_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&cache_map)) : "memory");
    for (int i = 0; i < kKvStages; ++i) { mbar_init(bar(A_KV_FULL + i), 1); mbar_init(bar(A_KV_EMPTY + i), kTiles); }
    mbar_init(bar(A_Q_READY), kSoftmaxWarps);
    for (int i = 0; i < kTiles; ++i) {
      mbar_init(bar(A_S_FULL + i), 1);
      mbar_init(bar(A_S_FREE + i), kSoftmaxWarps / kTiles);
      mbar_init(bar(A_P_READY + i), kSoftmaxWarps / kTiles);
      mbar_init(bar(A_PV_DONE + i), 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  pdl_wait();
  const int L = clamped_len(seqlens[b], max_pages, (tid == 0 && blockIdx.x == 0 && h == 0) ? dev_status : nullptr);
  // Query position s of the chunk sees tokens [0, L - (S - 1 - s)); a tile's last position sees the most.
  auto tile_pages = [&](int t) -> int {  // pages that tile t of this CTA looks at (0: nothing to see, or no rows)
    const int s_first = (qt * cta_tiles + t) * kQRows;
    if (t >= cta_tiles || s_first >= S) return 0;
    return (max(0, L - (S - 1 - (min(S, s_first + kQRows) - 1))) + kPage - 1) / kPage;
  };
  const int nt0 = tile_pages(0), nt1 = tile_pages(1), n_pages = max(nt0, nt1);  // block-uniform

  if (warp == kSoftmaxWarps && n_pages > 0) {
    // ======================================================================== TMA producer
    // Page n uses stage (n + 1) % 4; the first use of stage 0 is q_nope's.
    if (elect_one()) {
      const int tiles = cta_tiles == 2 && (qt * 2 + 1) * kQRows < S ? 2 : 1;
      mbar_arrive_expect_tx(bar(A_KV_FULL), tiles * 3 * kQSub);
      for (int t = 0; t < tiles; ++t) {
        const int row0 = b * S + (qt * cta_tiles + t) * kQRows;
        tma_load_2d(base + kOffKv + t * kQSub, &qn_map, h * DN_, row0, bar(A_KV_FULL));
        tma_load_2d(base + kOffQ + 2 * t * kQSub, &qn_map, h * DN_ + 64, row0, bar(A_KV_FULL));
        tma_load_2d(base + kOffQ + (2 * t + 1) * kQSub, &qr_map, h * DR_, row0, bar(A_KV_FULL));
      }
    }
    __syncwarp();
    const int32_t* row = page_table + static_cast<size_t>(b) * max_pages;
    for (int n = 0; n < n_pages; ++n) {
      int idx = row[n];
      const bool ok = idx >= 0 && idx < num_pages;
      if (!ok) { if (lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE); idx = 0; }
      const int g = n + 1, stage = g % kKvStages, use = g / kKvStages;
      mbar_wait(bar(A_KV_EMPTY + stage), (use & 1) ^ 1, abort_flag, dev_status);
      if (!*abort_flag && elect_one()) {
        mbar_arrive_expect_tx(bar(A_KV_FULL + stage), kKvStage);
        const uint32_t dst = base + kOffKv + stage * kKvStage;
        const int x = h * (DN_ + DV_), y = idx * kPage;
        tma_load_2d(dst, &kv_map, x, y, bar(A_KV_FULL + stage));
        tma_load_2d(dst + kSub64, &kv_map, x + 64, y, bar(A_KV_FULL + stage));
        tma_load_2d(dst + 2 * kSub64, &cache_map, R_, y, bar(A_KV_FULL + stage));
        tma_load_2d(dst + 3 * kSub64, &kv_map, x + DN_, y, bar(A_KV_FULL + stage));
        tma_load_2d(dst + 4 * kSub64, &kv_map, x + DN_ + 64, y, bar(A_KV_FULL + stage));
      }
      __syncwarp();
    }
  } else if (warp > kSoftmaxWarps && n_pages > 0) {
    // ======================================================================== MMA issuers, one per tile
    constexpr uint32_t idesc_qk = idesc_attn(kQRows, kPage, false), idesc_pv = idesc_attn(kQRows, DV_, true);
    const int t = warp - kSoftmaxWarps - 1, nt = t ? nt1 : nt0;
    const uint32_t s_col = tmem + kColS + t * 64, q_col = tmem + kColQ + t * 32, p_col = tmem + kColP + t * 32, o_col = tmem + kColO + t * DV_;
    const uint64_t q0 = smem_desc(base + kOffQ + 2 * t * kQSub, 16, 1024);
    mbar_wait(bar(A_Q_READY), 0, abort_flag, dev_status);
    if (elect_one()) mbar_arrive(bar(A_KV_EMPTY));   // its share of handing stage 0 to the pages
    __syncwarp();
    auto scores = [&](int n) {
      const int g = n + 1, stage = g % kKvStages;
      mbar_wait(bar(A_KV_FULL + stage), (g / kKvStages) & 1, abort_flag, dev_status);
      tc_fence_after();
      const uint64_t k0 = smem_desc(base + kOffKv + stage * kKvStage, 16, 1024);
      if (elect_one()) {
#pragma unroll
        for (int i = 0; i < 4; ++i) mma_ts(s_col, q_col + i * 8, desc_advance(k0, i * 32), idesc_qk, i != 0);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          mma_ss(s_col, desc_advance(q0, (i >> 2) * kQSub + (i & 3) * 32), desc_advance(k0, (1 + (i >> 2)) * kSub64 + (i & 3) * 32), idesc_qk, 1u);
        tc_commit(bar(A_S_FULL + t));
      }
      __syncwarp();
    };
    if (nt > 0) scores(0);
    for (int n = 0; n < nt; ++n) {
      if (n + 1 < nt) {
        mbar_wait(bar(A_S_FREE + t), n & 1, abort_flag, dev_status);
        scores(n + 1);
      }
      const int stage = (n + 1) % kKvStages;
      mbar_wait(bar(A_P_READY + t), n & 1, abort_flag, dev_status);
      tc_fence_after();
      const uint64_t v0 = smem_desc(base + kOffKv + stage * kKvStage + 3 * kSub64, kSub64, 1024);
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) mma_ts(o_col, p_col + kk * 8, desc_advance(v0, kk * 2048), idesc_pv, (n | kk) ? 1u : 0u);
        tc_commit(bar(A_KV_EMPTY + stage));
        tc_commit(bar(A_PV_DONE + t));
      }
      __syncwarp();
    }
    for (int n = nt; n < n_pages; ++n) {  // pages that only the other tile looks at
      const int g = n + 1, stage = g % kKvStages;
      mbar_wait(bar(A_KV_FULL + stage), (g / kKvStages) & 1, abort_flag, dev_status);
      if (elect_one()) mbar_arrive(bar(A_KV_EMPTY + stage));
      __syncwarp();
    }
  } else if (warp < kSoftmaxWarps) {
    // ======================================================================== softmax + write-out
    const int tile = warp >> 3, half = (warp >> 2) & 1, quad = warp & 3;
    const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
    const int row = quad * 32 + lane, s = (qt * cta_tiles + tile) * kQRows + row;
    const bool in_chunk = s < S && tile < cta_tiles;
    const int nt = tile ? nt1 : nt0;
    if (n_pages > 0) {
      // a quarter of this row of q_nope: shared memory (swizzled sub-tile of 128 rows x 128 bytes) -> tensor memory
      mbar_wait(bar(A_KV_FULL), 0, abort_flag, dev_status);
      const unsigned char* qrow = sm + kOffKv + tile * kQSub + row * 128;
      uint32_t v[16];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint4 x = *reinterpret_cast<const uint4*>(qrow + (((4 * half + j) ^ (row & 7)) << 4));
        v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
      }
      tmem_st16(tmem + lane_base + kColQ + tile * 32 + half * 16, v);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(A_Q_READY));
    }
    if (nt > 0) {
      // rows of the tile beyond the chunk are computed unmasked and never stored
      const int n_vis = in_chunk ? max(0, L - (S - 1 - s)) : 0x3fffffff;
      const bool pos_scale = scale_log2 >= 0.f;
      const uint32_t s_addr = tmem + lane_base + kColS + tile * 64 + half * 32;
      const uint32_t o_addr = tmem + lane_base + kColO + tile * DV_ + half * 64;
      const uint32_t p_addr = tmem + lane_base + kColP + tile * 32 + half * 16;
      float* my_max = row_s + (tile * 2 + half) * kQRows + row;
      const float* other_max = row_s + (tile * 2 + (half ^ 1)) * kQRows + row;
      const int pair_bar = 1 + tile * 4 + quad;   // the two warps that share these rows
      float m_used = -INFINITY, l_run = 0.f;
      for (int n = 0; n < nt; ++n) {
        mbar_wait(bar(A_S_FULL + tile), n & 1, abort_flag, dev_status);
        tc_fence_after();
        uint32_t sq[32];
        tmem_ld32(s_addr, sq);
        tc_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(A_S_FREE + tile));
        const int tok_end = n_vis - n * kPage - half * 32;  // of this thread's 32 tokens, [0, tok_end) are visible
        const bool full = __all_sync(0xffffffffu, tok_end >= 32) && pos_scale;
        float rowmax = -INFINITY;
        if (full) {
          float a = __uint_as_float(sq[0]), c2 = __uint_as_float(sq[1]);
#pragma unroll
          for (int j = 2; j < 32; j += 2) { a = fmaxf(a, __uint_as_float(sq[j])); c2 = fmaxf(c2, __uint_as_float(sq[j + 1])); }
          rowmax = fmaxf(a, c2) * scale_log2;
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) rowmax = fmaxf(rowmax, j < tok_end ? __uint_as_float(sq[j]) * scale_log2 : -INFINITY);
        }
        int move;  // does the reference maximum of any of the 32 rows have to move?
        asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, %2, 64, q;\nselp.s32 %0, 1, 0, p;\n}"
                     : "=r"(move) : "r"(static_cast<int>(n == 0 || rowmax > m_used + 8.f)), "r"(pair_bar) : "memory");
        if (move) {
          *my_max = rowmax;
          asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
          const float m_new = fmaxf(m_used, fmaxf(rowmax, *other_max));
          const float alpha = (m_new == -INFINITY) ? 1.f : exp2f(m_used - m_new);
          m_used = m_new;
          l_run *= alpha;
          if (n > 0) {
            mbar_wait(bar(A_PV_DONE + tile), (n - 1) & 1, abort_flag, dev_status);  // O is at rest
            tc_fence_after();
#pragma unroll 1
            for (int g = 0; g < 4; ++g) {
              uint32_t ov[16];
              tmem_ld16(o_addr + g * 16, ov);
              tc_wait_ld();
#pragma unroll
              for (int j = 0; j < 16; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * alpha);
              tmem_st16(o_addr + g * 16, ov);
            }
          }
        }
        const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used;
        uint32_t pk[16];
        float ps0 = 0.f, ps1 = 0.f;
        if (full) {
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float p0 = ex2_approx(fmaf(__uint_as_float(sq[j]), scale_log2, neg_m));
            const float p1 = ex2_approx(fmaf(__uint_as_float(sq[j + 1]), scale_log2, neg_m));
            ps0 += p0; ps1 += p1;
            pk[j >> 1] = pack_bf16(p0, p1);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float p0 = j < tok_end ? ex2_approx(fmaf(__uint_as_float(sq[j]), scale_log2, neg_m)) : 0.f;
            const float p1 = j + 1 < tok_end ? ex2_approx(fmaf(__uint_as_float(sq[j + 1]), scale_log2, neg_m)) : 0.f;
            ps0 += p0; ps1 += p1;
            pk[j >> 1] = pack_bf16(p0, p1);
          }
        }
        l_run += ps0 + ps1;
        if (n > 0) mbar_wait(bar(A_PV_DONE + tile), (n - 1) & 1, abort_flag, dev_status);  // P has been read
        tmem_st16(p_addr, pk);
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(A_P_READY + tile));
      }
      // ---- write-out: wait for the last PV; the two halves of the row's sum meet where the tile's queries were; normalise,
      // store half the row
      mbar_wait(bar(A_PV_DONE + tile), (nt - 1) & 1, abort_flag, dev_status);
      tc_fence_after();
      float* sums = reinterpret_cast<float*>(sm + kOffQ + 2 * tile * kQSub);  // [half][128]
      sums[half * kQRows + row] = l_run;
      asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
      const float l_tot = l_run + sums[(half ^ 1) * kQRows + row];
      const float inv = l_tot > 0.f ? 1.f / l_tot : 0.f;
      __nv_bfloat16* dst = out + ((static_cast<size_t>(b) * S + s) * H + h) * DV_ + half * 64;
#pragma unroll 1
      for (int g = 0; g < 2; ++g) {
        uint32_t ov[32];
        tmem_ld32(o_addr + g * 32, ov);
        tc_wait_ld();
        if (in_chunk) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint4 o;
            o.x = pack_bf16(__uint_as_float(ov[8 * q]) * inv, __uint_as_float(ov[8 * q + 1]) * inv);
            o.y = pack_bf16(__uint_as_float(ov[8 * q + 2]) * inv, __uint_as_float(ov[8 * q + 3]) * inv);
            o.z = pack_bf16(__uint_as_float(ov[8 * q + 4]) * inv, __uint_as_float(ov[8 * q + 5]) * inv);
            o.w = pack_bf16(__uint_as_float(ov[8 * q + 6]) * inv, __uint_as_float(ov[8 * q + 7]) * inv);
            reinterpret_cast<uint4*>(dst + g * 32)[q] = o;
          }
        }
      }
      if (in_chunk && half == 0 && lse_out != nullptr)
        lse_out[(static_cast<size_t>(b) * S + s) * H + h] = l_tot > 0.f ? (m_used + log2f(l_tot)) * kLn2 : -INFINITY;
      tc_fence_before();
    } else if (in_chunk) {
      // nothing visible to any row of the tile (L < S): zeros and lse = -inf
      uint4* dst = reinterpret_cast<uint4*>(out + ((static_cast<size_t>(b) * S + s) * H + h) * DV_ + half * 64);
      for (int q = 0; q < 8; ++q) dst[q] = make_uint4(0, 0, 0, 0);
      if (half == 0 && lse_out != nullptr) lse_out[(static_cast<size_t>(b) * S + s) * H + h] = -INFINITY;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace prefill

cudaError_t launch_prefill_attention(const transmla_params_t& p, const __nv_bfloat16* q_nope, const __nv_bfloat16* q_pe,
                                     const __nv_bfloat16* cache, const __nv_bfloat16* kv_dec, const int32_t* page_table,
                                     const int32_t* seqlens, __nv_bfloat16* out, float* lse, int32_t* dev_status,
                                     cudaStream_t stream) {
  using namespace prefill;
  // q_nope as [B*S rows, H*dn], q_pe as [B*S, H*dR]: a box is 128 rows (positions) x 64 columns of one head.
  CUtensorMap qn, qr, kv, cm;
  const uint64_t rows = static_cast<uint64_t>(p.batch) * p.q_len;
  if (!sm100::tensor_map_2d(&qn, q_nope, rows, p.num_heads * DN_, kQRows) ||
      !sm100::tensor_map_2d(&qr, q_pe, rows, p.num_heads * DR_, kQRows) ||
      !sm100::tensor_map_2d(&kv, kv_dec, static_cast<uint64_t>(p.num_pages) * kPage, p.num_heads * (DN_ + DV_), kPage) ||
      !sm100::tensor_map_2d(&cm, cache, static_cast<uint64_t>(p.num_pages) * kPage, R_ + DR_, kPage))
    return cudaErrorInvalidValue;
  static PerDeviceFlag smem_set;
  if (cudaError_t e = ensure_dynamic_smem(prefill_attention_kernel, kAttnSmem, smem_set); e != cudaSuccess) return e;
  // Two tiles a CTA take about 1.3 times as long as one, so that one is better where the device then needs no more waves than
  // 1.3 times those of CTAs with two (32 heads over 8192 tokens: 1 x 256 positions 100 us with one, 126 with two; 3 x 300 over
  // 16384 397 and 464; 4 x 256 200 and 155, 6 x 256 306 and 268).
  constexpr long long kSms = 148;
  const long long heads = static_cast<long long>(p.num_heads) * p.batch;
  auto waves = [&](int tiles) { return ((p.q_len + tiles * kQRows - 1) / (tiles * kQRows) * heads + kSms - 1) / kSms; };
  const int cta_tiles = 10 * waves(1) < 13 * waves(2) ? 1 : 2;
  dim3 grid((p.q_len + cta_tiles * kQRows - 1) / (cta_tiles * kQRows), p.num_heads, p.batch);
  return launch_pdl(prefill_attention_kernel, grid, dim3(kAttnThreads), static_cast<size_t>(kAttnSmem), stream, qn, qr, kv, cm, page_table,
                    seqlens, out, lse, dev_status, p.q_len, p.num_heads, p.num_pages, p.max_pages_per_seq,
                    p.softmax_scale * kLog2e, cta_tiles);
}
}  // namespace transmla

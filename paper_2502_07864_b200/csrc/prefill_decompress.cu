// Decompression of the latent cache for prefill in the MHA form (Eq. 8): k^C_{j,h} = W_UK_h c_j, v_{j,h} = W_UV_h c_j.
//
// A GEMM [tokens x 512] x [512 x H*256] on the Blackwell tensor path, by CTA pairs (cta_group::2) that stay resident.  A unit
// of work is 256 tokens (four pages of one sequence, fetched through the page table, 128 tokens in each CTA) x one head;
// the units of the whole batch are cut into equal runs, one per pair, so that no wave is left half empty.  The latent tile
// stays in shared memory for the run's heads; the head's weights stream through a four-stage ring 64 columns at a time, the
// first CTA loading W_UK_h and the second W_UV_h: each is read once per pair.  D [128 x 256] per CTA, two of them in tensor
// memory, so that the write-out of one head runs beside the next one's products.
// What bounds it: the tensor pipe, 32 products of 130 cycles a unit.  With one CTA per tile the weights, 256 KB a head and
// CTA, came from L2 at 30 bytes a cycle and SM, about what it gives: a head took 8400 cycles; now 5000,
// 26 bytes a cycle and SM of weights and 13 of stores.  32 768 tokens x 32 heads: 288 -> 229 us (1.2 PFLOP/s); 12 ragged
// sequences of 3 to 30 thousand: 412 -> 383 us.
// Write-out: D passes as bf16 through a staging tile in shared memory (the layout of the store's tensor map) to the store by
// TMA, whole 128-byte lines at a time, 64 columns of the 128 tokens per half of the warps and round.
// Rows of tokens at or beyond the sequence length are stored as zeros: a probability of zero times such a value
// row must stay zero in the attention kernel.
// Warps 0-7 write out (warp w: tensor-memory lanes 32 (w % 4).., columns 128 (w / 4)..), warp 8 issues TMA, warp 9 of the
// pair's first CTA issues the products.  Bounded waits.
#include "prefill.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace prefill {

using namespace sm100;

constexpr int R = 512, DR = 64, DN = 128, DV = 128;
constexpr int kTok = 128;                       // tokens per CTA
constexpr int kHeadCols = DN + DV;              // 256
constexpr int kSub = kPage * 128;               // 8192: 64 rows x 64 columns
constexpr int kASub = kTok * 128;               // 16384: 128 tokens x 64 latent columns
constexpr int kABytes = R / 64 * kASub;         // 131072: the latent tile
constexpr int kBStage = DN * 128;               // 16384: this CTA's 128 of the 256 weight rows x 64 columns
constexpr int kBStages = 4;
constexpr int kOutHalf = kTok * 128;            // 16384: staging of one half of the warps, 2 pages x 64 rows x 128 bytes
constexpr int kOffA = 0, kOffB = kABytes, kOffOut = kOffB + kBStages * kBStage, kOffBar = kOffOut + 2 * kOutHalf, kOffMisc = kOffBar + 256;
constexpr int kDecompSmem = kOffMisc + 64;
constexpr int kDecompThreads = 320;
static_assert(kOffBar % 256 == 0 && kDecompSmem <= 232448, "shared memory map");
enum { BAR_B_FULL = 0, BAR_B_EMPTY = kBStages, BAR_A_FULL = 2 * kBStages, BAR_A_EMPTY, BAR_D_FULL, BAR_D_FREE = BAR_D_FULL + 2,
       BAR_D_FREE2 = BAR_D_FREE + 2 };  // ..2: the second CTA's word

__host__ __device__ constexpr uint32_t instr_desc_pair(int n) {  // bf16, fp32 accumulator, both operands K-major, M = 256
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);
}
__device__ __forceinline__ uint32_t first_cta(uint32_t bar) {  // the barrier at this offset in the pair's first CTA
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(bar));
  return a;
}
// A load into this CTA that reports to a barrier of the pair's first CTA.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(d), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void commit_pair(uint32_t bar) {  // arrives on the barrier at this offset in both CTAs
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(static_cast<uint16_t>(3)) : "memory");
}
// Arrival on a barrier of the pair's first CTA that hands over tensor memory and nothing in memory: it needs no release, because
// tcgen05.wait::ld has completed the reads before it is issued.
__device__ __forceinline__ void arrive_first(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(first_cta(bar)) : "memory");
}

// Tile pairs (256 tokens) of sequences before b, and which sequence holds tile pair `want`: all lanes of a warp together.
struct TileAt { int b, tile, L; };
__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int seq_tiles(const int32_t* seqlens, int b, int B, int max_pages) {
  if (b >= B) return 0;
  return (clamped_len(seqlens[b], max_pages, nullptr) + 2 * kTok - 1) / (2 * kTok);
}
__device__ TileAt find_tile(const int32_t* seqlens, int B, int max_pages, int want, int lane) {
  for (int b0 = 0; b0 < B; b0 += 32) {
    const int mine = seq_tiles(seqlens, b0 + lane, B, max_pages);
    int before = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, before, o); if (lane >= o) before += t; }
    const int total = __shfl_sync(0xffffffffu, before, 31);
    if (want < total) {
      const int owner = __ffs(__ballot_sync(0xffffffffu, want < before)) - 1;
      const int b = b0 + owner;
      return {b, want - __shfl_sync(0xffffffffu, before - mine, owner), clamped_len(seqlens[b], max_pages, nullptr)};
    }
    want -= total;
  }
  return {0, 0, 0};
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kDecompThreads, 1)
decompress_kernel(const __grid_constant__ CUtensorMap cache_map, const __grid_constant__ CUtensorMap wuk_map,
                  const __grid_constant__ CUtensorMap wuv_map, const __grid_constant__ CUtensorMap out_map,
                  const int32_t* page_table, const int32_t* seqlens, int32_t* dev_status, int B, int H, int num_pages,
                  int max_pages) {
  extern __shared__ __align__(1024) unsigned char smem_aligned[];  // no room to align by hand
  unsigned char* sm = smem_aligned;
  const uint32_t base = smem_u32(sm);
  if ((base & 1023u) != 0) { set_status(dev_status, TRANSMLA_DEV_TIMEOUT); return; }
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(sm + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  auto bar = [&](int i) -> uint32_t { return base + kOffBar + 8 * i; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  pdl_trigger();
  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&cache_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(rank ? &wuv_map : &wuk_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&out_map)) : "memory");
    for (int i = 0; i < kBStages; ++i) { mbar_init(bar(BAR_B_FULL + i), 1); mbar_init(bar(BAR_B_EMPTY + i), 1); }
    mbar_init(bar(BAR_A_FULL), 1);
    mbar_init(bar(BAR_A_EMPTY), 1);
    for (int i = 0; i < 2; ++i) { mbar_init(bar(BAR_D_FULL + i), 1); mbar_init(bar(BAR_D_FREE + i), 8); mbar_init(bar(BAR_D_FREE2 + i), 8); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  auto sync_pair = [] { asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory"); };
  tc_fence_before();
  __syncthreads();
  sync_pair();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  pdl_wait();
  int tiles = 0;
  for (int b0 = 0; b0 < B; b0 += 32) {
    if (pair == 0 && rank == 0 && warp == 0 && b0 + lane < B) clamped_len(seqlens[b0 + lane], max_pages, dev_status);  // reports a bad length
    tiles += warp_sum(seq_tiles(seqlens, b0 + lane, B, max_pages));
  }
  const long long units = static_cast<long long>(tiles) * H;
  const int u0 = static_cast<int>(units * pair / pairs), u1 = static_cast<int>(units * (pair + 1) / pairs);  // this pair's run

  // The run, tile by tile: this CTA's two pages of the tile (page -1: none, or not valid), and the heads h0 .. h1-1.
  struct Segment { int b, first_page, L, page[2], pages_here, pages_pair, h0, h1; };
  auto segment_at = [&](int u, bool report) -> Segment {
    const int tile_pair = u / H;
    const TileAt at = find_tile(seqlens, B, max_pages, tile_pair, lane);
    Segment s;
    s.b = at.b;
    s.L = at.L;
    s.first_page = at.tile * 4 + rank * 2;
    const int n_pages = (at.L + kPage - 1) / kPage;
    s.pages_here = max(0, min(2, n_pages - s.first_page));
    s.pages_pair = min(4, n_pages - at.tile * 4);
    for (int i = 0; i < 2; ++i) {
      s.page[i] = -1;
      if (i >= s.pages_here) continue;
      const int p = page_table[static_cast<size_t>(at.b) * max_pages + s.first_page + i];
      if (p >= 0 && p < num_pages) s.page[i] = p;
      else if (report && lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE);
    }
    s.h0 = u - tile_pair * H;
    s.h1 = min(H, s.h0 + u1 - u);
    return s;
  };

  if (warp == 8) {
    // ---------------------------------------------------------------------- TMA: the tile, then the heads' weights
    const uint32_t a_full = first_cta(bar(BAR_A_FULL));
    const CUtensorMap* w_map = rank ? &wuv_map : &wuk_map;
    int g = 0, segs = 0;
    for (int u = u0; u < u1; ++segs) {
      const Segment s = segment_at(u, true);
      mbar_wait(bar(BAR_A_EMPTY), (segs & 1) ^ 1, abort_flag, dev_status);
      if (!*abort_flag && elect_one()) {
        if (rank == 0) mbar_arrive_expect_tx(bar(BAR_A_FULL), s.pages_pair * (R / 64) * kSub);
        for (int i = 0; i < s.pages_here; ++i) {
#pragma unroll
          for (int c = 0; c < R / 64; ++c)
            tma_load_pair(base + kOffA + c * kASub + i * kSub, &cache_map, c * 64, max(0, s.page[i]) * kPage, a_full);
        }
      }
      __syncwarp();
      for (int h = s.h0; h < s.h1; ++h) {
        for (int kc = 0; kc < R / 64; ++kc, ++g) {
          const int stage = g % kBStages, use = g / kBStages;
          mbar_wait(bar(BAR_B_EMPTY + stage), (use & 1) ^ 1, abort_flag, dev_status);
          if (!*abort_flag && elect_one()) {
            if (rank == 0) mbar_arrive_expect_tx(bar(BAR_B_FULL + stage), 2 * kBStage);
            tma_load_pair(base + kOffB + stage * kBStage, w_map, kc * 64, h * DN, first_cta(bar(BAR_B_FULL + stage)));
          }
          __syncwarp();
        }
      }
      u += s.h1 - s.h0;
    }
  } else if (warp == 9) {
    // ---------------------------------------------------------------------- products, for both CTAs
    if (rank == 0) {
      constexpr uint32_t idesc = instr_desc_pair(kHeadCols);
      int g = 0, d = 0, segs = 0;
      for (int u = u0; u < u1; ++segs) {
        const int h0 = u % H, h1 = min(H, h0 + u1 - u);
        mbar_wait(bar(BAR_A_FULL), segs & 1, abort_flag, dev_status);
        tc_fence_after();
        const uint64_t a0 = smem_desc(base + kOffA, 16, 1024);
        for (int h = h0; h < h1; ++h, ++d) {
          const int buf = d & 1;
          if (d >= 2) {
            mbar_wait(bar(BAR_D_FREE + buf), ((d >> 1) - 1) & 1, abort_flag, dev_status);
            mbar_wait(bar(BAR_D_FREE2 + buf), ((d >> 1) - 1) & 1, abort_flag, dev_status);
          }
#pragma unroll 1
          for (int kc = 0; kc < R / 64; ++kc, ++g) {
            const int stage = g % kBStages;
            mbar_wait(bar(BAR_B_FULL + stage), (g / kBStages) & 1, abort_flag, dev_status);
            tc_fence_after();
            const uint64_t b0 = smem_desc(base + kOffB + stage * kBStage, 16, 1024);
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                mma_pair(tmem + buf * kHeadCols, desc_advance(a0, kc * kASub + kk * 32), desc_advance(b0, kk * 32), idesc, (kc | kk) ? 1u : 0u);
              commit_pair(bar(BAR_B_EMPTY + stage));
              if (kc == R / 64 - 1) {
                commit_pair(bar(BAR_D_FULL + buf));
                if (h == h1 - 1) commit_pair(bar(BAR_A_EMPTY));
              }
            }
            __syncwarp();
          }
        }
        u += h1 - h0;
      }
    }
  } else {
    // ---------------------------------------------------------------------- warps 0-7: thread = token row
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t d_addr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + half * 128;
    const int row = quarter * 32 + lane, slot = row & (kPage - 1), half_bar = 1 + half;
    unsigned char* stage_row = sm + kOffOut + half * kOutHalf + (row >> 6) * kSub + slot * 128;
    const bool issuer = (tid & 127) == 0;
    int d = 0;
    for (int u = u0; u < u1;) {
      const Segment s = segment_at(u, false);
      const bool real = s.first_page * kPage + row < s.L;  // otherwise zeros
      for (int h = s.h0; h < s.h1; ++h, ++d) {
        const int buf = d & 1;
        mbar_wait(bar(BAR_D_FULL + buf), (d >> 1) & 1, abort_flag, dev_status);
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          uint32_t v[64];
          tmem_ld32(d_addr + buf * kHeadCols + c * 64, v);
          tmem_ld32(d_addr + buf * kHeadCols + c * 64 + 32, v + 32);
          tc_wait_ld();
          if (c == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { if (rank == 0) mbar_arrive(bar(BAR_D_FREE + buf)); else arrive_first(bar(BAR_D_FREE2 + buf)); }
          }
          // the TMA store of the round before must have finished reading the staging tile
          if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          asm volatile("bar.sync %0, 128;" ::"r"(half_bar) : "memory");
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t* x = v + j * 8;
            uint4 o;
            o.x = real ? pack_bf16(__uint_as_float(x[0]), __uint_as_float(x[1])) : 0u;
            o.y = real ? pack_bf16(__uint_as_float(x[2]), __uint_as_float(x[3])) : 0u;
            o.z = real ? pack_bf16(__uint_as_float(x[4]), __uint_as_float(x[5])) : 0u;
            o.w = real ? pack_bf16(__uint_as_float(x[6]), __uint_as_float(x[7])) : 0u;
            *reinterpret_cast<uint4*>(stage_row + ((j ^ (slot & 7)) << 4)) = o;
          }
          fence_proxy_async();
          asm volatile("bar.sync %0, 128;" ::"r"(half_bar) : "memory");
          if (issuer) {
            for (int i = 0; i < 2; ++i) {
              if (s.page[i] < 0) continue;   // none, or a page the table does not name validly: reported, not written
              asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                           ::"l"(reinterpret_cast<uint64_t>(&out_map)), "r"(h * kHeadCols + half * 128 + c * 64), "r"(s.page[i] * kPage),
                             "r"(base + kOffOut + half * kOutHalf + i * kSub)
                           : "memory");
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        }
      }
      u += s.h1 - s.h0;
    }
    if (issuer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // the last stores have left shared memory and landed
  }
  tc_fence_before();
  __syncthreads();
  sync_pair();  // neither CTA leaves while the other may still reach its barriers
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace prefill

bool prefill_supported(const transmla_params_t& p) {
  return p.kv_lora_rank == prefill::R && p.qk_rope_dim == prefill::DR && p.qk_nope_dim == prefill::DN && p.v_dim == prefill::DV;
}

cudaError_t launch_prefill_decompress(const transmla_params_t& p, const __nv_bfloat16* cache, const int32_t* page_table,
                                      const int32_t* seqlens, const __nv_bfloat16* w_uk, const __nv_bfloat16* w_uv,
                                      __nv_bfloat16* kv_dec, int32_t* dev_status, cudaStream_t stream) {
  using namespace prefill;
  CUtensorMap cmap, kmap, vmap, omap;
  if (!sm100::tensor_map_2d(&cmap, cache, static_cast<uint64_t>(p.num_pages) * kPage, R + DR, kPage) ||
      !sm100::tensor_map_2d(&kmap, w_uk, static_cast<uint64_t>(p.num_heads) * DN, R, DN) ||
      !sm100::tensor_map_2d(&vmap, w_uv, static_cast<uint64_t>(p.num_heads) * DV, R, DV) ||
      !sm100::tensor_map_2d(&omap, kv_dec, static_cast<uint64_t>(p.num_pages) * kPage, p.num_heads * kHeadCols, kPage))
    return cudaErrorInvalidValue;
  static PerDeviceFlag smem_set;
  if (cudaError_t e = ensure_dynamic_smem(decompress_kernel, kDecompSmem, smem_set); e != cudaSuccess) return e;
  // As many pairs as the device holds at once (a pair lives inside one GPC), or fewer when the page table has no room for
  // that many units.
  static PerDeviceFlag pairs_of;  // asked once per device
  const int dev = current_device_slot();
  int pairs = dev >= 0 ? pairs_of.value[dev].load(std::memory_order_acquire) : 0;
  if (pairs == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kDecompThreads);
    cfg.dynamicSmemBytes = kDecompSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaError_t e = cudaOccupancyMaxActiveClusters(&pairs, decompress_kernel, &cfg); e != cudaSuccess) return e;
    if (pairs < 1) return cudaErrorInvalidConfiguration;
    if (dev >= 0) pairs_of.value[dev].store(pairs, std::memory_order_release);
  }
  const long long most = static_cast<long long>(p.batch) * ((p.max_pages_per_seq + 3) / 4) * p.num_heads;
  if (most < pairs) pairs = static_cast<int>(most);
  return launch_pdl(decompress_kernel, dim3(2 * pairs), dim3(kDecompThreads), static_cast<size_t>(kDecompSmem), stream, cmap, kmap, vmap, omap,
                    page_table, seqlens, dev_status, p.batch, p.num_heads, p.num_pages, p.max_pages_per_seq);
}

}  // namespace transmla

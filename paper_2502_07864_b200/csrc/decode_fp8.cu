// Split-KV absorbed-MLA decode (Eq. 9 right, second line) over an FP8 latent cache, r = 512, dR = 64.
//
// Stored row of a token (656 bytes instead of 1152): 512 e4m3 codes of c / scale, 64 bf16 values k^R / scale,
// the fp32 scale, 12 bytes of padding.  (The paper only names FP8; the format is this library's own.)  The kernel
// is the bf16 split-KV kernel with three differences:
//   - scores: the page's codes are the B operand of native FP8 products (kind::f8f6f4, K = 32).  The absorbed
//     queries are split, row by row, into two e4m3 terms q ~ sq * (hi + lo) when they are moved into tensor memory
//     (two terms carry about the 8 bits a bf16 query has), and the 32 high and 32 low rows are the 64 rows of one
//     weight-stationary product, so that a page's codes are read once; the rope part runs as bf16 products on
//     k^R / scale and (q^R / sq, 0).  A score is sq * scale_j times the sum of its high and its low row.
//   - products: eight more warps transpose the codes of a page on their way (ldmatrix) and put them into tensor memory
//     as fp16 (exactly), latents on the lanes: the A operand of O^T += V^T P'^T.  A token's scale goes into its
//     probability instead: P' = scale_j * p_j in fp16 (operands of one product must agree in type), with the reference
//     maximum taken over score + log2 scale so that P' keeps the range p had.
//   - a page's stage goes back to the TMA warp when three parties are done with it: the scores, the converters,
//     and the softmax warps (they read the scales).
// Tensor-memory map: Q 0-127 (four codes a column; high rows in quadrants 0 and 2, low rows in 1 and 3), q^R / sq 128-159,
// S 160-191, O^T 192-319, V^T 320-511 (three buffers of half a page: 4 tiles of 128 latents x 32 tokens, two a column).
// Lane i of a group of 16 holds latent 2 i (i < 8) or 2 (i - 8) + 1 of its 16: ldmatrix hands out pairs.
//
// What bounds it: HBM, 1800 cycles a page at 148 SMs (a TMA-only loop over such pages reaches 6.1 TB/s whatever the stage
// count).  The codes as fp16 in shared memory (written by the converters, read again by the products) cost 1000 cycles
// of its 128 bytes a page and held a page at 2500 cycles; now about 1000 are left in all and a page
// takes 2100, of which the converters are busy 1700.  B=64 x 4K-8K: kernel 110 -> 66 us (4.0 TB/s), step 145 -> 112 us;
// S=2 B=30 x 11K-20K: step 266 -> 180 us.
//
// Warp roles: warps 0-3 softmax + epilogue, warp 4 TMA, warp 5 score products, warp 6 PV products, warps 8-15
// converters.  All waits are bounded as in the bf16 kernel.
#include <cuda_fp16.h>

#include "common.cuh"
#include "partition_walk.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace fp8 {

using namespace sm100;

constexpr int R = 512, DR = 64, K = R + DR;
constexpr int kRowBytes = TRANSMLA_FP8_ROW_BYTES;     // 656
constexpr int kCodeTiles = R / 128;                   // 4 sub-tiles of 64 tokens x 128 codes
constexpr int kSubTileBytes = kPage * 128;            // 8192
constexpr int kOffRope = kCodeTiles * kSubTileBytes;  // 32768: 64 tokens x 64 bf16
constexpr int kOffScale = kOffRope + kSubTileBytes;   // 40960: 64 tokens x 16 bytes (the scale is the first 4)
constexpr int kStageBytes = kOffScale + kPage * 16;   // 41984
constexpr int kStages = 4;
constexpr int kPBytes = kRowBlock * 128;              // 4096: P[32 rows][64 tokens] fp16
constexpr int kQTileBytes = kRowBlock * 128;          // 4096: one 64-column sub-tile of the 32 query rows (bf16)
constexpr int kQChunks = K / 64;                      // 9
constexpr int kThreads = 512, kConverters = 256;
constexpr int kVBufs = 3;                             // V^T buffers, half a page each
constexpr uint32_t kTmemCols = 512;
constexpr int kMetaRing = 16;
enum { ITEM_QUERIES = 1, ITEM_PAGE = 2, ITEM_END = 3 };
constexpr uint32_t kColQ = 0, kColQr = 128, kColS = 160, kColO = 192, kColV = 320;

// shared-memory map (offsets from a 1024-byte aligned base)
constexpr int kOffStage = 0;
constexpr int kOffP = kStages * kStageBytes;      // 167936 (a multiple of 1024), 2 buffers
constexpr int kOffX = kOffP + 2 * kPBytes;        // halves of the scores on their way between warps: [4][16][32] f32
constexpr int kOffBar = kOffX + 8192;             // mbarriers (8 bytes each)
constexpr int kOffMisc = kOffBar + 256;
// misc: pmax_s[2][4][32] f32, alpha_s[32], inv_l[32], qmax_s[4][32] f32, meta[16] int4, tmem base, abort, ring_done, v_flags[3]
constexpr int kMiscBytes = 1024 + 128 + 128 + 512 + 16 * kMetaRing + 32;
constexpr int kSmemBytes = kOffMisc + kMiscBytes + 1024;  // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 232448, "shared memory budget");
static_assert(kStageBytes % 1024 == 0 && kQChunks * kQTileBytes <= kStageBytes, "stage layout");

enum { BAR_KV_FULL = 0, BAR_KV_EMPTY = kStages, BAR_Q_READY = 2 * kStages, BAR_S_FULL, BAR_S_FREE, BAR_P_READY0,
       BAR_P_READY1, BAR_PV_DONE0, BAR_PV_DONE1, BAR_V_FULL, BAR_V_EMPTY = BAR_V_FULL + kVBufs, BAR_COUNT = BAR_V_EMPTY + kVBufs };
static_assert(BAR_COUNT <= 24 && kOffBar % 256 == 0, "barrier block");

// D[tmem] (+)= A[tmem] * B[smem desc], both operands e4m3 (K = 32 per instruction), weight-stationary, M = 64 (layout of
// A and D as for mma_ws_ss; A replicated in the two halves of the lanes)
__device__ __forceinline__ void mma_ws_ts_f8(uint32_t d, uint32_t a, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.ws.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n}"
      ::"r"(d), "r"(a), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Instruction descriptors, fp32 accumulator: e4m3 x e4m3 (both K-major), M = 64; fp16 x fp16, M = 128.
__host__ __device__ constexpr uint32_t instr_desc_e4m3(int n) {
  return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(64 >> 4) << 24);
}
__host__ __device__ constexpr uint32_t instr_desc_f16(int n) {
  return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(128 >> 4) << 24);
}
// Two floats -> two e4m3 codes (nearest, ties to even, saturating), first argument in the low byte.
__device__ __forceinline__ uint32_t pack_e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}
// Two e4m3 codes (low 16 bits) -> two fp16 values, exactly.
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t v) {
  uint32_t r;
  asm("{\n.reg .b16 t;\nmov.b32 {t, _}, %1;\ncvt.rn.f16x2.e4m3x2 %0, t;\n}" : "=r"(r) : "r"(v));
  return r;
}
__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// 16 lanes x 16 columns: thread 4 i + k of the warp gives column 4 j + k of lanes i (v[2 j]) and i + 8 (v[2 j + 1]), j = 0..3.
__device__ __forceinline__ void tmem_st_16x128b_x4(uint32_t taddr, const uint32_t* v) {
  asm volatile("tcgen05.st.sync.aligned.16x128b.x4.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"
               ::TM_W4(v, 0), TM_W4(v, 4), "r"(taddr)
               : "memory");
}

// An all-zero row adds nothing to O, but its scale is 1 by definition and may be far above its neighbours': if the reference
// maximum followed it, their P' would leave fp16's range.  So whenever the reference is about to move (rarely: a segment's
// first page, a new maximum far above) the softmax warps look for such rows and leave them out.  In functions of their own:
// the same code inside the page loop cost 240 cycles a page.
// Which of the warp's 16 tokens have all-zero rows; rows with a scale of exactly 1 are rare, and only their codes are read.
__device__ __noinline__ uint32_t find_zero_rows(const unsigned char* page_s, int warp, int lane) {
  uint32_t zero = 0;
  uint32_t ones = __ballot_sync(0xffffffffu, lane < 16 && *reinterpret_cast<const uint32_t*>(page_s + kOffScale + (warp * 16 + (lane & 15)) * 16) == 0x3f800000u);
#pragma unroll 1
  for (; ones != 0; ones &= ones - 1) {
    const int j = __ffs(ones) - 1;
    const uint4 c = *reinterpret_cast<const uint4*>(page_s + (lane >> 3) * kSubTileBytes + (warp * 16 + j) * 128 + (lane & 7) * 16);
    if (!__any_sync(0xffffffffu, ((c.x | c.y | c.z | c.w) & 0x7f7f7f7fu) != 0)) zero |= 1u << j;
  }
  return zero;
}
// The row's maximum of score + log2 scale over the warp's 16 tokens (scores in `x`, 32 apart; tokens from `seen` on do not
// count), a zero row's scale taken as the smallest there is.
__device__ __noinline__ float maximum_without(uint32_t zero, const float* x, const unsigned char* scl, int seen) {
  float pmax = -INFINITY;
#pragma unroll 1
  for (int j = 0; j < seen && j < 16; ++j) {
    const int e = static_cast<int>(*reinterpret_cast<const uint32_t*>(scl + j * 16) >> 23) - 127;
    pmax = fmaxf(pmax, x[j * 32] + static_cast<float>(zero >> j & 1u ? -60 : max(e, -60)));
  }
  return pmax;
}
// Zero rows' probabilities become zeros in this row of P (they may be beyond fp16's range, and infinity times zero is not zero).
__device__ __noinline__ void clear_zero_rows(uint32_t zero, unsigned char* prow, int warp, int sw) {
#pragma unroll 1
  for (; zero != 0; zero &= zero - 1) {
    const int t = warp * 16 + __ffs(zero) - 1;
    *reinterpret_cast<uint16_t*>(prow + (((t >> 3) ^ sw) << 4) + (t & 7) * 2) = 0;
  }
}

// ---------------------------------------------------------------------------------------------- kernel
__global__ void __launch_bounds__(kThreads, 1)
decode_fp8_kernel(const __grid_constant__ CUtensorMap cache_map, const __grid_constant__ CUtensorMap scale_map,
                  const __grid_constant__ CUtensorMap q_map, const unsigned char* cache,
                    const int32_t* page_table, const int32_t* seqlens,
                    const int32_t* cum, const int32_t* plan, float* partial_o,
                    float* partial_lse, int32_t* dev_status, int S, int H, int num_pages, int max_pages,
                    float scale_log2, int B, int dynamic, int32_t* next) {
  extern __shared__ unsigned char smem_unaligned[];
  const uint32_t raw = smem_u32(smem_unaligned);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_unaligned + (base - raw);
  float* pmax_s = reinterpret_cast<float*>(sm + kOffMisc);         // [2][4][32]: per page parity, warp, row
  float* alpha_s = pmax_s + 256;                                   // [32]
  float* inv_l = alpha_s + 32;                                     // [32]
  float* qmax_s = inv_l + 32;                                    // [4][32]: parts of the query rows' maxima
  int4* meta = reinterpret_cast<int4*>(qmax_s + 128);            // [kMetaRing]: what each ring item is
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(meta + kMetaRing);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  volatile int* ring_done = abort_flag + 1;
  volatile int* v_flags = ring_done + 1;  // [3]: what the converters put into each V buffer
  auto bar = [&](int i) -> uint32_t { return base + kOffBar + 8 * i; };

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rb = blockIdx.y;
  const int SH = S * H;
  pdl_trigger();

  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&cache_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&q_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&scale_map)) : "memory");
    for (int i = 0; i < kStages; ++i) { mbar_init(bar(BAR_KV_FULL + i), 1); mbar_init(bar(BAR_KV_EMPTY + i), 2 + kConverters); }
    for (int i = 0; i < kVBufs; ++i) { mbar_init(bar(BAR_V_FULL + i), kConverters); mbar_init(bar(BAR_V_EMPTY + i), 1); }
    mbar_init(bar(BAR_S_FULL), 1);
    mbar_init(bar(BAR_S_FREE), 128);
    mbar_init(bar(BAR_Q_READY), 128);
    mbar_init(bar(BAR_P_READY0), 128);
    mbar_init(bar(BAR_P_READY1), 128);
    mbar_init(bar(BAR_PV_DONE0), 1);
    mbar_init(bar(BAR_PV_DONE1), 1);
    *abort_flag = 0;
    *ring_done = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  pdl_wait();  // the plan, the absorbed queries and the appended cache rows come from the kernel before this one
  const int part = blockIdx.x;
  const int4 pl = reinterpret_cast<const int4*>(plan)[part];
  const bool has_home = pl.y > pl.x;

  if (has_home) {
    if (warp == 4) {
      // ======================================================================== TMA producer
      // The ring carries, per segment, one item with the 32 absorbed query rows followed by the segment's pages,
      // and one closing item when the CTA has nothing more to do.  What an item is goes into `meta`.
      int g = 0;  // ring items issued by this CTA so far
      const uint64_t stream_policy = l2_evict_first_policy();
      auto acquire = [&](int gi) -> uint32_t {  // waits for the stage of ring item gi; returns its index
        const int stage = gi % kStages, use = gi / kStages;
        mbar_wait(bar(BAR_KV_EMPTY + stage), (use & 1) ^ 1, abort_flag, dev_status);
        return stage;
      };
      auto issue_queries = [&](int b, int slot_code, int L) {
        const uint32_t stage = acquire(g);
        if (!*abort_flag && elect_one()) {
          meta[g & (kMetaRing - 1)] = make_int4(ITEM_QUERIES, b, slot_code, L);
          mbar_arrive_expect_tx(bar(BAR_KV_FULL + stage), kQChunks * kQTileBytes);
          const uint32_t dst = base + kOffStage + stage * kStageBytes;
#pragma unroll
          for (int c = 0; c < kQChunks; ++c)
            tma_load_2d(dst + c * kQTileBytes, &q_map, c * 64, b * SH + rb * kRowBlock, bar(BAR_KV_FULL + stage));
        }
        __syncwarp();
        ++g;
      };
      auto issue_page = [&](int b, int pj, bool first, bool last) {
        int idx = page_table[static_cast<size_t>(b) * max_pages + pj];
        const bool ok = idx >= 0 && idx < num_pages;
        if (!ok) { if (lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE); idx = 0; }
        // A page is one contiguous piece of memory: it is asked into L2 while its stage is still in use.
        if (elect_one())
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(cache + static_cast<size_t>(idx) * (kPage * kRowBytes)),
                       "r"(kPage * kRowBytes) : "memory");
        const uint32_t stage = acquire(g);
        if (!*abort_flag && elect_one()) {
          meta[g & (kMetaRing - 1)] = make_int4(ITEM_PAGE, pj, ok ? 1 : 0, (first ? 1 : 0) | (last ? 2 : 0));
          // the pool as bytes [num_pages * 64 rows, 656]: four boxes of 128 codes, one of 128 bytes (64 bf16) and,
          // through a map without swizzle, one of 16 bytes that holds the scale
          mbar_arrive_expect_tx(bar(BAR_KV_FULL + stage), kStageBytes);
          const uint32_t dst = base + kOffStage + stage * kStageBytes;
#pragma unroll
          for (int c = 0; c <= kCodeTiles; ++c)
            tma_load_2d_hint(dst + c * kSubTileBytes, &cache_map, c * 128, idx * kPage, bar(BAR_KV_FULL + stage), stream_policy);
          tma_load_2d_hint(dst + kOffScale, &scale_map, R + 2 * DR, idx * kPage, bar(BAR_KV_FULL + stage), stream_policy);
        }
        __syncwarp();
        ++g;
      };
      const PartitionWalk walk = {page_table, seqlens, cum, next + static_cast<size_t>(rb) * B, partial_lse, part, rb * kRowBlock,
                                  kRowBlock, SH, max_pages, dynamic};
      walk_partition(walk, pl, lane, issue_queries, issue_page);
      {  // closing item
        const uint32_t stage = acquire(g);
        if (elect_one()) {
          meta[g & (kMetaRing - 1)] = make_int4(ITEM_END, 0, 0, 0);
          mbar_arrive(bar(BAR_KV_FULL + stage));
        }
        __syncwarp();
      }
    } else if (warp == 5) {
      // ======================================================================== MMA issuer, scores
      // Follows the ring: skips query items (the softmax warps move them to tensor memory and report through
      // Q_READY, which also tells when the ring has ended) and runs the score products of a page as soon as it has
      // landed: one e4m3 product per 32 codes on the page's codes as they came from memory, then four bf16 products on
      // the rope part, all into one accumulator.
      constexpr uint32_t idesc_f8 = instr_desc_e4m3(kPage);
      constexpr uint32_t idesc_rope = instr_desc(kPage, false, 64);
      int g = 0, n = 0, seg = 0;  // ring items, pages, segments handled so far
      while (true) {
        // a segment begins (or the ring ends): the softmax warps say which
        mbar_wait(bar(BAR_Q_READY), seg & 1, abort_flag, dev_status);
        ++seg;
        if (__any_sync(0xffffffffu, *abort_flag != 0) || *ring_done != 0) break;
        if (elect_one()) mbar_arrive(bar(BAR_KV_EMPTY + g % kStages));  // this warp's share of handing the query item back
        __syncwarp();
        ++g;
        while (true) {
          const int stage = g % kStages, use = g / kStages;
          mbar_wait(bar(BAR_KV_FULL + stage), use & 1, abort_flag, dev_status);
          const int4 m = meta[g & (kMetaRing - 1)];
          if (n > 0) mbar_wait(bar(BAR_S_FREE), (n - 1) & 1, abort_flag, dev_status);
          tc_fence_after();
          const uint64_t k0 = smem_desc(base + kOffStage + stage * kStageBytes, 16, 1024);
          if (elect_one()) {
#pragma unroll
            for (int c = 0; c < kCodeTiles; ++c) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                mma_ws_ts_f8(tmem + kColS, tmem + kColQ + c * 32 + kk * 8, desc_advance(k0, c * kSubTileBytes + kk * 32), idesc_f8,
                             (c | kk) ? 1u : 0u);
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_ws_ts(tmem + kColS, tmem + kColQr + kk * 8, desc_advance(k0, kOffRope + kk * 32), idesc_rope, 1u);
            tc_commit(bar(BAR_KV_EMPTY + stage));  // one of the three parties that hand the stage back
            tc_commit(bar(BAR_S_FULL));
          }
          __syncwarp();
          ++g; ++n;
          if ((m.w & 2) != 0 || m.x != ITEM_PAGE || __any_sync(0xffffffffu, *abort_flag != 0)) break;
        }
      }
    } else if (warp == 6) {
      // ======================================================================== MMA issuer, products
      // O^T += V^T P'^T, half a page (32 tokens) at a time, as soon as the page's probabilities and the half's V^T are
      // there.  V^T comes with the half's place in its segment (1 = the segment starts here, 4 = nothing more): this warp
      // does not look at the ring, whose stages may be pages further.
      constexpr uint32_t idesc_pv = instr_desc_f16(kRowBlock);
      for (int h = 0;; ++h) {
        const int vb = h % kVBufs, n = h >> 1;
        mbar_wait(bar(BAR_V_FULL + vb), (h / kVBufs) & 1, abort_flag, dev_status);
        const int flags = v_flags[vb];
        if (__any_sync(0xffffffffu, *abort_flag != 0) || (flags & 4) != 0) break;
        if ((h & 1) == 0) mbar_wait(bar(BAR_P_READY0 + (n & 1)), (n >> 1) & 1, abort_flag, dev_status);
        tc_fence_after();
        const uint64_t b0 = smem_desc(base + kOffP + (n & 1) * kPBytes + (h & 1) * 64, 16, 1024);
        const uint32_t v0 = tmem + kColV + vb * 64;
        const uint32_t acc0 = (flags & 1) != 0 ? 0u : 1u;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
            for (int t = 0; t < 4; ++t)
              mma_ts(tmem + kColO + t * 32, v0 + t * 16 + kk * 8, desc_advance(b0, kk * 32), idesc_pv, kk == 0 ? acc0 : 1u);
          }
          tc_commit(bar(BAR_V_EMPTY + vb));
          if (h & 1) tc_commit(bar(BAR_PV_DONE0 + (n & 1)));
        }
        __syncwarp();
      }
    } else if (warp >= 8) {
      // ======================================================================== converters (warps 8-15)
      // Per half page (32 tokens): the codes of quadrant `quad`'s latents, transposed by ldmatrix (8 tokens x 8 pairs of
      // codes a matrix; a thread gets a pair of latents for two tokens), as fp16 into that quadrant's lanes of a V^T
      // buffer; tokens beyond the sequence become zeros.  They hand a query item back too, so that no stage can be used
      // twice before they have seen it.
      const int quad = warp & 3, t0 = (warp - 8) >> 2 << 1;   // a quadrant's two warps take two tiles of 128 latents each
      const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
      int g = 0, h = 0, L_seg = 0;
      bool run = true;
      while (run) {
        const int stage = g % kStages, use = g / kStages;
        mbar_wait(bar(BAR_KV_FULL + stage), use & 1, abort_flag, dev_status);
        const int4 m = meta[g & (kMetaRing - 1)];
        if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
        if (m.x == ITEM_QUERIES) {
          L_seg = m.w;  // the sequence's length, for the pages that follow
          mbar_arrive(bar(BAR_KV_EMPTY + stage));
          ++g;
          continue;
        }
        run = m.x == ITEM_PAGE;
        const uint32_t st = base + kOffStage + stage * kStageBytes;
        const int valid = m.z != 0 ? min(kPage, L_seg - m.y * kPage) : 0;  // tokens [valid, 64) must read as zero
#pragma unroll 1
        for (int half = 0; half < (run ? 2 : 1); ++half, ++h) {
          const int vb = h % kVBufs;
          if (h >= kVBufs) mbar_wait(bar(BAR_V_EMPTY + vb), (h / kVBufs - 1) & 1, abort_flag, dev_status);
          if (tid == 256) v_flags[vb] = !run ? 4 : half == 0 ? (m.w & 1) : 0;
          if (run) {
            tc_fence_after();
            const int tok = half * 32 + lane;
            const int left = valid - half * 32 - 2 * (lane & 3);  // of this thread's token pairs 8 j + (0, 1): visible if 8 j (+ 1) < left
            uint32_t x[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {  // tile t0 + i / 2, 16 of this quadrant's latents: one 16-byte chunk of the token rows
              const uint32_t addr = st + (t0 + (i >> 1)) * kSubTileBytes + tok * 128 + (((quad * 2 + (i & 1)) ^ (tok & 7)) << 4);
              asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                           : "=r"(x[i][0]), "=r"(x[i][1]), "=r"(x[i][2]), "=r"(x[i][3]) : "r"(addr) : "memory");
            }
            if (valid < kPage) {
#pragma unroll
              for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) x[i][j] = 8 * j + 1 < left ? x[i][j] : 8 * j < left ? x[i][j] & 0xffffu : 0u;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint32_t o[8];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                o[2 * j] = e4m3x2_to_f16x2(__byte_perm(x[i][j], 0, 0x4420));      // the even latent, tokens 2 k and 2 k + 1
                o[2 * j + 1] = e4m3x2_to_f16x2(__byte_perm(x[i][j], 0, 0x4431));  // the odd one
              }
              tmem_st_16x128b_x4(tmem + lane_base + (static_cast<uint32_t>((i & 1) * 16) << 16) + kColV + vb * 64 + (t0 + (i >> 1)) * 16, o);
            }
            tc_wait_st();
            tc_fence_before();
          }
          mbar_arrive(bar(BAR_V_FULL + vb));
        }
        mbar_arrive(bar(BAR_KV_EMPTY + stage));
        ++g;
      }
    } else if (warp < 4) {
      // ======================================================================== softmax + epilogue (warps 0-3)
      const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
      const int my_row = rb * kRowBlock + lane;  // query row of this thread (same in all four replicas)
      int g = 0, n = 0;  // ring items and pages handled so far
      float sq_row = 1.f;  // scale of this thread's query row (see open_segment)
      // Looks at ring item g.  Queries: moves the 32 rows from shared memory (swizzled sub-tiles of 32 rows x
      // 128 bytes) to this warp's replica in tensor memory, 32 columns (64 elements) at a time, hands the stage
      // back and returns the item's description.  Closing item: marks the ring as ended.  Either way the MMA
      // warp is told through Q_READY.  All 128 threads take the same path (the description is the same for all).
      auto open_segment = [&]() -> int4 {
        const int stage = g % kStages, use = g / kStages;
        mbar_wait(bar(BAR_KV_FULL + stage), use & 1, abort_flag, dev_status);
        int4 m = meta[g & (kMetaRing - 1)];
        int aborted;
        asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, 1, 128, q;\nselp.s32 %0, 1, 0, p;\n}"
                     : "=r"(aborted) : "r"(*abort_flag) : "memory");
        if (aborted || m.x != ITEM_QUERIES) {
          m.x = ITEM_END;
          if (tid == 0) *ring_done = 1;
          asm volatile("bar.sync 1, 128;" ::: "memory");
          mbar_arrive(bar(BAR_Q_READY));
          return m;
        }
        unsigned char* qrow = sm + kOffStage + stage * kStageBytes + lane * 128;
        // This row's absorbed query q (512 bf16): q ~ sq * (hi + lo) with hi, lo e4m3 and sq = max|q| / 448.  All four
        // warps need all of it in their quadrant, so each works out a quarter (two sub-tiles of 64 values) and leaves the
        // codes where the bf16 values were: 64 bytes of high terms, then 64 bytes of low terms.
        float amax = 0.f;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 x = *reinterpret_cast<const uint4*>(qrow + (2 * warp + c) * kQTileBytes + ((j ^ (lane & 7)) << 4));
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) amax = fmaxf(amax, fmaxf(fabsf(bf16_lo(w[k])), fabsf(bf16_hi(w[k]))));
          }
        }
        qmax_s[warp * 32 + lane] = amax;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        amax = fmaxf(fmaxf(qmax_s[lane], qmax_s[32 + lane]), fmaxf(qmax_s[64 + lane], qmax_s[96 + lane]));
        sq_row = amax > 0.f ? amax * (1.f / 448.f) : 1.f;
        const float inv_sq = 1.f / sq_row;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          unsigned char* tile = qrow + (2 * warp + c) * kQTileBytes;
          uint32_t qv[32];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 x = *reinterpret_cast<const uint4*>(tile + ((j ^ (lane & 7)) << 4));
            qv[4 * j] = x.x; qv[4 * j + 1] = x.y; qv[4 * j + 2] = x.z; qv[4 * j + 3] = x.w;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {  // 16 values -> 16 bytes of each term
            uint32_t h[4], l[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t w0 = qv[8 * j + 2 * k], w1 = qv[8 * j + 2 * k + 1];
              const float a0 = bf16_lo(w0) * inv_sq, a1 = bf16_hi(w0) * inv_sq, a2 = bf16_lo(w1) * inv_sq, a3 = bf16_hi(w1) * inv_sq;
              const uint32_t h0 = pack_e4m3x2(a0, a1), h1 = pack_e4m3x2(a2, a3);
              const float2 b0 = __half22float2(as_half2(e4m3x2_to_f16x2(h0))), b1 = __half22float2(as_half2(e4m3x2_to_f16x2(h1)));
              h[k] = h0 | (h1 << 16);
              l[k] = pack_e4m3x2(a0 - b0.x, a1 - b0.y) | (pack_e4m3x2(a2 - b1.x, a3 - b1.y) << 16);
            }
            *reinterpret_cast<uint4*>(tile + ((j ^ (lane & 7)) << 4)) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(tile + (((j + 4) ^ (lane & 7)) << 4)) = make_uint4(l[0], l[1], l[2], l[3]);
          }
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll 1
        for (int c = 0; c < kCodeTiles * 2; ++c) {  // 64 query values -> 16 columns of four codes, this quadrant's term
          uint32_t v[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint4 x = *reinterpret_cast<const uint4*>(qrow + c * kQTileBytes + (((j + 4 * (warp & 1)) ^ (lane & 7)) << 4));
            v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
          }
          tmem_st16(tmem + lane_base + kColQ + c * 16, v);
        }
        {  // the rope part, divided by sq, stays bf16; the low rows have none
          uint32_t v[32];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 x = *reinterpret_cast<const uint4*>(qrow + 8 * kQTileBytes + ((j ^ (lane & 7)) << 4));
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) v[4 * j + k] = (warp & 1) ? 0u : pack_bf16(bf16_lo(w[k]) * inv_sq, bf16_hi(w[k]) * inv_sq);
          }
          tmem_st32(tmem + lane_base + kColQr, v);
        }
        tc_wait_st();
        tc_fence_before();
        mbar_arrive(bar(BAR_Q_READY));
        fence_proxy_async();  // the stage was written here; its next contents come through the async proxy
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (tid == 0) mbar_arrive(bar(BAR_KV_EMPTY + stage));  // one of three: the score warp and the converters see it too
        ++g;
        return m;
      };
      int4 seg_meta = open_segment();
      while (seg_meta.x == ITEM_QUERIES) {
        const int L = seg_meta.w;
        float* o_rows = partial_o + (static_cast<size_t>(seg_meta.z) * SH + rb * kRowBlock) * R;
        float* lse_rows = partial_lse + static_cast<size_t>(seg_meta.z) * SH + rb * kRowBlock;
        const int n_vis = my_row < SH ? L - (S - 1 - my_row / H) : 0;

        float m_used = -INFINITY, l_run = 0.f;
        bool more = true;
        while (more) {
          const int stage = g % kStages;
          mbar_wait(bar(BAR_KV_FULL + stage), (g / kStages) & 1, abort_flag, dev_status);
          const int4 pm = meta[g & (kMetaRing - 1)];
          const int pj = pm.y;
          const bool page_ok = pm.z != 0;
          const int tok_end = page_ok ? n_vis - pj * kPage : 0;           // tokens [0, tok_end) of the page are visible
          const bool first = (pm.w & 1) != 0;
          const int buf = n & 1;

          // Quadrants 0 and 2 hold the high rows' sums for 32 tokens, 1 and 3 the low rows' for the same: each warp keeps
          // 16 of them (even warps the first), gets the other row's for those from its neighbour and adds.
          mbar_wait(bar(BAR_S_FULL), n & 1, abort_flag, dev_status);
          tc_fence_after();
          uint32_t sq[16];  // this warp's 16 tokens of its row
          {
            uint32_t other[16];
            tmem_ld16(tmem + lane_base + kColS + (warp & 1) * 16, sq);
            tmem_ld16(tmem + lane_base + kColS + (~warp & 1) * 16, other);
            tc_wait_ld();
            tc_fence_before();
            mbar_arrive(bar(BAR_S_FREE));
            float* mine = reinterpret_cast<float*>(sm + kOffX) + warp * 512 + lane;
            const float* theirs = reinterpret_cast<const float*>(sm + kOffX) + (warp ^ 1) * 512 + lane;
#pragma unroll
            for (int j = 0; j < 16; ++j) mine[j * 32] = __uint_as_float(other[j]);
            asm volatile("bar.sync %0, 64;" ::"r"(2 + (warp >> 1)) : "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) sq[j] = __float_as_uint(__uint_as_float(sq[j]) + theirs[j * 32]);
          }
          float sc[16];
          {
            // a score is sq (row) * scale_j (token) * the accumulated sum; tokens beyond the visible range are dropped
            // by selection, so whatever their scale holds does not matter.  The reference maximum is that of score +
            // log2 scale (its whole part, from the exponent bits; not below -60, so that exp2 of the rest stays finite).
            const unsigned char* scl = sm + kOffStage + stage * kStageBytes + kOffScale + warp * 16 * 16;
            const float row_factor = sq_row * scale_log2;
            float pmax = -INFINITY;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const bool seen = warp * 16 + j < tok_end;
              sc[j] = *reinterpret_cast<const float*>(scl + j * 16);
              const float x = seen ? __uint_as_float(sq[j]) * (row_factor * sc[j]) : -INFINITY;
              sc[j] = seen ? sc[j] : 0.f;
              sq[j] = __float_as_uint(x);
              pmax = fmaxf(pmax, x + static_cast<float>(max(static_cast<int>(__float_as_uint(sc[j]) >> 23) - 127, -60)));
            }
            pmax_s[(buf * 4 + warp) * 32 + lane] = pmax;
          }
          // one barrier per page: the row maxima meet, and all 128 threads learn together whether the CTA gave up
          int aborted;
          asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, 1, 128, q;\nselp.s32 %0, 1, 0, p;\n}"
                       : "=r"(aborted) : "r"(*abort_flag) : "memory");
          more = (pm.w & 2) == 0 && pm.x == ITEM_PAGE && !aborted;
          float rowmax = fmaxf(fmaxf(pmax_s[(buf * 4 + 0) * 32 + lane], pmax_s[(buf * 4 + 1) * 32 + lane]),
                                     fmaxf(pmax_s[(buf * 4 + 2) * 32 + lane], pmax_s[(buf * 4 + 3) * 32 + lane]));
          // Lazy rescale: the reference maximum only moves when some row's new maximum exceeds it by 2^8.  Every
          // warp holds all 32 rows, so the four warps take the same decision without talking to each other.
          float alpha = 1.f;
          // (Not after a give-up: what the warps then see may differ, and there are barriers below.)
          // (a segment's first page moves it from -infinity)
          bool rescale = __any_sync(0xffffffffu, rowmax > m_used + 8.f) && !aborted;
          uint32_t zero_rows = 0;
          if (rescale) {
            const unsigned char* page_s = sm + kOffStage + stage * kStageBytes;
            zero_rows = find_zero_rows(page_s, warp, lane);
            int again;
            asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, 1, 128, q;\nselp.s32 %0, 1, 0, p;\n}"
                         : "=r"(again) : "r"(static_cast<int>(zero_rows)) : "memory");
            if (again) {
              float* x = reinterpret_cast<float*>(sm + kOffX) + warp * 512 + lane;  // the neighbour has read its halves
#pragma unroll
              for (int j = 0; j < 16; ++j) x[j * 32] = __uint_as_float(sq[j]);
              pmax_s[(buf * 4 + warp) * 32 + lane] = maximum_without(zero_rows, x, page_s + kOffScale + warp * 16 * 16, tok_end - warp * 16);
              asm volatile("bar.sync 1, 128;" ::: "memory");
              rowmax = fmaxf(fmaxf(pmax_s[(buf * 4 + 0) * 32 + lane], pmax_s[(buf * 4 + 1) * 32 + lane]),
                             fmaxf(pmax_s[(buf * 4 + 2) * 32 + lane], pmax_s[(buf * 4 + 3) * 32 + lane]));
              rescale = __any_sync(0xffffffffu, rowmax > m_used + 8.f);
            }
          }
          if (tid == 0) mbar_arrive(bar(BAR_KV_EMPTY + stage));  // scales (and codes) have been read: the softmax warps' share
          if (first) {
            m_used = rowmax;
            rescale = false;
          } else {
            if (rescale) {
              const float m_new = fmaxf(m_used, rowmax);
              alpha = (m_new == -INFINITY) ? 1.f : exp2f(m_used - m_new);
              m_used = m_new;
              l_run *= alpha;
            }
          }
          const float m_ref = m_used == -INFINITY ? 0.f : m_used;

          // ---- probabilities of tokens 16*warp .. 16*warp+15
          uint32_t pk[8];
          float psum = 0.f;
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const float p0 = ex2_approx(__uint_as_float(sq[j]) - m_ref), p1 = ex2_approx(__uint_as_float(sq[j + 1]) - m_ref);
            psum += p0 + p1;
            pk[j >> 1] = pack_f16(p0 * sc[j], p1 * sc[j + 1]);
          }
          l_run += psum;

          // ---- P buffer `buf` is free once PV of CTA page n-2 is done
          if (n >= 2) mbar_wait(bar(BAR_PV_DONE0 + buf), ((n >> 1) - 1) & 1, abort_flag, dev_status);
          {
            unsigned char* prow = sm + kOffP + buf * kPBytes + lane * 128;
            const int c0w = 2 * warp, sw = lane & 7;
            *reinterpret_cast<uint4*>(prow + ((c0w ^ sw) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *reinterpret_cast<uint4*>(prow + (((c0w + 1) ^ sw) << 4)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            if (zero_rows != 0) clear_zero_rows(zero_rows, prow, warp, sw);
          }
          // ---- rescale O^T by alpha (columns = query rows) once the previous PV has landed
          if (rescale) {
            if (warp == 0) alpha_s[lane] = alpha;
            asm volatile("bar.sync 1, 128;" ::: "memory");  // a later rescale is at least one page barrier away
            if (n >= 1) mbar_wait(bar(BAR_PV_DONE0 + ((n - 1) & 1)), ((n - 1) >> 1) & 1, abort_flag, dev_status);
            tc_fence_after();
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
              uint32_t ov[32];
              tmem_ld32(tmem + lane_base + kColO + t * 32, ov);
              tc_wait_ld();
#pragma unroll
              for (int j = 0; j < 32; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * alpha_s[j]);
              tmem_st32(tmem + lane_base + kColO + t * 32, ov);
            }
            tc_wait_st();
          }
          fence_proxy_async();
          tc_fence_before();
          mbar_arrive(bar(BAR_P_READY0 + buf));
          ++g; ++n;
        }

        // ---- epilogue of the segment: wait for the last PV, normalise, store O (transposed back) and lse.
        // The row sums meet in the half of pmax_s that the last page did not use (its readers are behind the
        // last page's barrier; the next page writes it only after the barrier at the end of this epilogue).
        float* l_part = pmax_s + (n & 1) * 128;
        l_part[warp * 32 + lane] = l_run;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const float l_tot = l_part[lane] + l_part[32 + lane] + l_part[64 + lane] + l_part[96 + lane];
        if (warp == 0) {
          inv_l[lane] = l_tot > 0.f ? 1.f / l_tot : 0.f;
          if (my_row < SH) lse_rows[lane] = l_tot > 0.f ? (m_used + log2f(l_tot)) * kLn2 : -INFINITY;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        // The queries of the next segment go to tensor memory now (every QK^T of this segment has completed), so
        // that its first QK^T runs while this segment's result is written out.
        seg_meta = open_segment();
        const int n_last = n - 1;
        mbar_wait(bar(BAR_PV_DONE0 + (n_last & 1)), (n_last >> 1) & 1, abort_flag, dev_status);
        tc_fence_after();
        // lane -> latent, see the tensor-memory map
        float* dst = o_rows + warp * 32 + (lane & 16) + ((lane & 15) < 8 ? 2 * (lane & 15) : 2 * (lane & 7) + 1);
#pragma unroll 1
        for (int t = 0; t < 4; ++t) {
          uint32_t ov[32];
          tmem_ld32(tmem + lane_base + kColO + t * 32, ov);
          tc_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (rb * kRowBlock + j < SH) dst[static_cast<size_t>(j) * R + t * 128] = __uint_as_float(ov[j]) * inv_l[j];
        }
        tc_fence_before();
        asm volatile("bar.sync 1, 128;" ::: "memory");  // inv_l and the row sums are reused by the next segment
      }
    }
  }

  // ---- teardown: everyone arrives, tensor memory is returned
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------- host
}  // namespace fp8

bool decode_fp8_supported(const transmla_params_t& p) {
  return p.kv_lora_rank == fp8::R && p.qk_rope_dim == fp8::DR && p.q_len * p.num_heads <= 1024;
}

// The workspace's own partition count suits the bf16 kernels, which may take 64 query rows a CTA; here a CTA takes 32, and the
// batch is planned for as many partitions as bring the grid to one wave (two waves measured 290 us a step instead of 267 at
// B=30, S=2, 11K to 20K tokens).
Partitioning decode_fp8_partitioning(const transmla_params_t& p, int G) {
  if (p.num_partitions == 0 && library_partitions(p, kRowBlock, &G) != TRANSMLA_OK) G = 1;
  return {G, p.num_partitions == 0 ? 16 : 0};
}

cudaError_t launch_decode_fp8(const transmla_params_t& p, int G, const __nv_bfloat16* q_hat, const void* cache_fp8,
                              const int32_t* page_table, const int32_t* seqlens, const int32_t* cum, const int32_t* plan,
                              float* partial_o, float* partial_lse, int32_t* dev_status, cudaStream_t stream) {
  using namespace fp8;
  // The pool as bytes [num_pages * 64 rows, 656]: boxes of 64 rows x 128 bytes with the 128-byte swizzle (codes and
  // rope part), and of 64 rows x 16 bytes without swizzle (scales).  The absorbed queries as in the bf16 kernel.
  CUtensorMap map, smap, qmap;
  const int SH = p.q_len * p.num_heads;
  const uint64_t rows = static_cast<uint64_t>(p.num_pages) * kPage;
  if (!tensor_map_2d(&map, cache_fp8, rows, kRowBytes, kPage, 128, TMAP_U8_SW128) ||
      !tensor_map_2d(&smap, cache_fp8, rows, kRowBytes, kPage, 16, TMAP_U8_PLAIN) ||
      !tensor_map_2d(&qmap, q_hat, static_cast<uint64_t>(p.batch) * SH, K, kRowBlock))
    return cudaErrorInvalidValue;
  static PerDeviceFlag smem_set;
  if (cudaError_t e = ensure_dynamic_smem(decode_fp8_kernel, kSmemBytes, smem_set); e != cudaSuccess) return e;
  dim3 grid(G, (SH + kRowBlock - 1) / kRowBlock);
  int32_t* next = const_cast<int32_t*>(cum) + 3 * p.batch + 1;  // page counters, zeroed by the plan
  return launch_pdl(decode_fp8_kernel, grid, dim3(kThreads), static_cast<size_t>(kSmemBytes), stream, map, smap, qmap,
                    static_cast<const unsigned char*>(cache_fp8), page_table, seqlens, cum, plan, partial_o, partial_lse, dev_status, p.q_len, p.num_heads,
                    p.num_pages, p.max_pages_per_seq, p.softmax_scale * kLog2e, p.batch, dynamic_claims(p, G) ? 1 : 0, next);
}

}  // namespace transmla

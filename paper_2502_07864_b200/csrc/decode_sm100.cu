// Split-KV absorbed-MLA decode (Eq. 9 right, second line) on the Blackwell tensor path:
// TMA page loads -> shared memory -> tcgen05.mma with accumulators in tensor memory.
//
// Specialised for the production latent shape r = 512, dR = 64 (a cache row is 576 bf16 = 1152 B).
// One CTA = one (partition, block of 32 query rows); it walks its segments page by page.
//
// Tile plan per 64-token page
//   S  [32 x 64]    = Q_hat (tensor memory, the 32 rows replicated into the four 32-lane quadrants)
//                     x K_hat^T (the page in shared memory, K-major, 128-byte swizzle), K = 576, by
//                     tcgen05.mma.ws with M = 32, whose accumulator puts tokens 16w..16w+15 of the 32 rows in
//                     quadrant w (16 columns).  The M = 128 form on the replicated rows gives the same values and
//                     takes about as many cycles (34 against 31 an instruction), but it multiplies every row four
//                     times: at the 1000 W limit that energy was what bound long steps (SM clock 1.4 GHz at
//                     B = 128 x 8192 cached tokens; step 274 us, with M = 32 at 1.9 GHz 239 us).
//   O^T[512 x 32]  += C^T (the same shared-memory page read MN-major, four 128-row tiles)
//                     x P^T (32 rows x 64 tokens, bf16, shared memory, K-major)
// O is kept transposed (latent index on the tensor-memory lanes, query rows on the columns) so that
// the accumulator costs 4 x 32 columns instead of 512, which leaves room for Q_hat (288 columns) and
// S (16 columns) in the 512-column tensor memory, and so that no padded query row costs PV work.
//
// Warp roles: warps 0-3 softmax + epilogue (warp w owns tensor-memory lanes 32w..32w+31, i.e. replica w
// of the 32 query rows, and the probabilities of tokens 16w..16w+15 of every page); warp 4 lane 0
// issues TMA; warp 5 issues the QK^T instructions and warp 6 the PV instructions (warp-uniform control flow, one
// elected lane per instruction; two warps because issuing costs a warp about 45 cycles per instruction, more than
// the 20 to 36 cycles these small instructions occupy the pipe).  All waits are bounded: on expiry the CTA raises
// TRANSMLA_DEV_TIMEOUT, every later wait returns at once, and control flow stays identical, so the CTA
// still reaches its teardown and frees its tensor memory.
#include "common.cuh"
#include "partition_walk.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace sm100 {

constexpr int R = 512, DR = 64, K = R + DR;
constexpr int kChunks = K / 64;                       // 9 sub-tiles of 64 columns (128 bytes) per page
constexpr int kSubTileBytes = kPage * 128;            // 8192
constexpr int kStageBytes = kChunks * kSubTileBytes;  // 73728
constexpr int kStages = 3;
constexpr int kPBytes = kRowBlock * 128;              // 4096: P[32 rows][64 tokens] bf16
constexpr int kQTileBytes = kRowBlock * 128;          // 4096: one 64-column sub-tile of the 32 query rows
constexpr int kThreads = 224;
constexpr uint32_t kTmemCols = 512;
constexpr int kMetaRing = 16;            // descriptions of the ring items in flight (a power of two >= 2 * kStages)
enum { ITEM_QUERIES = 1, ITEM_PAGE = 2, ITEM_END = 3 };
constexpr uint32_t kColQ = 0, kColS = 288, kColO = 352;  // tensor-memory column map: Q_hat, S, O^T (4 x 32)

// shared-memory map (offsets from a 1024-byte aligned base)
constexpr int kOffStage = 0;
constexpr int kOffP = kStages * kStageBytes;      // 2 buffers
constexpr int kOffBar = kOffP + 2 * kPBytes;      // mbarriers (8 bytes each)
constexpr int kOffMisc = kOffBar + 128;
// misc: pmax_s[2][4][32] f32, alpha_s[32] f32, inv_l[32] f32, meta[16] int4, tmem base, abort, ring_done
constexpr int kMiscBytes = 1024 + 128 + 128 + 16 * kMetaRing + 16;
constexpr int kSmemBytes = kOffMisc + kMiscBytes + 1024;  // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 232448, "shared memory budget");

enum { BAR_KV_FULL = 0, BAR_KV_EMPTY = kStages, BAR_Q_READY = 2 * kStages, BAR_S_FULL, BAR_S_FREE, BAR_P_READY0, BAR_P_READY1,
       BAR_PV_DONE0, BAR_PV_DONE1 };

// ---------------------------------------------------------------------------------------------- kernel
__global__ void __launch_bounds__(kThreads, 1)
decode_sm100_kernel(const __grid_constant__ CUtensorMap cache_map, const __grid_constant__ CUtensorMap q_map,
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
  int4* meta = reinterpret_cast<int4*>(inv_l + 32);                // [kMetaRing]: what each ring item is
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(meta + kMetaRing);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  volatile int* ring_done = abort_flag + 1;
  auto bar = [&](int i) -> uint32_t { return base + kOffBar + 8 * i; };

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int part = blockIdx.x, rb = blockIdx.y;
  const int SH = S * H;
  pdl_trigger();

  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&cache_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&q_map)) : "memory");
    for (int i = 0; i < kStages; ++i) { mbar_init(bar(BAR_KV_FULL + i), 1); mbar_init(bar(BAR_KV_EMPTY + i), 1); }
    mbar_init(bar(BAR_Q_READY), 128);
    mbar_init(bar(BAR_S_FULL), 1);
    mbar_init(bar(BAR_S_FREE), 128);
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
          mbar_arrive_expect_tx(bar(BAR_KV_FULL + stage), kChunks * kQTileBytes);
          const uint32_t dst = base + kOffStage + stage * kStageBytes;
#pragma unroll
          for (int c = 0; c < kChunks; ++c)
            tma_load_2d(dst + c * kQTileBytes, &q_map, c * 64, b * SH + rb * kRowBlock, bar(BAR_KV_FULL + stage));
        }
        __syncwarp();
        ++g;
      };
      auto issue_page = [&](int b, int pj, bool first, bool last) {
        int idx = page_table[static_cast<size_t>(b) * max_pages + pj];
        const bool ok = idx >= 0 && idx < num_pages;
        if (!ok) { if (lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE); idx = 0; }
        const uint32_t stage = acquire(g);
        if (!*abort_flag && elect_one()) {
          meta[g & (kMetaRing - 1)] = make_int4(ITEM_PAGE, pj, ok ? 1 : 0, (first ? 1 : 0) | (last ? 2 : 0));
          mbar_arrive_expect_tx(bar(BAR_KV_FULL + stage), kStageBytes);
          const uint32_t dst = base + kOffStage + stage * kStageBytes;
#pragma unroll
          for (int c = 0; c < kChunks; ++c)
            tma_load_2d_hint(dst + c * kSubTileBytes, &cache_map, c * 64, idx * kPage, bar(BAR_KV_FULL + stage), stream_policy);
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
      // Q_READY, which also tells when the ring has ended) and runs QK^T for a page as soon as it has landed.
      // Issuing an instruction costs this warp about as many cycles as a small one occupies the pipe, so the 36
      // score instructions and the 16 product instructions of a page are issued by two warps side by side.
      constexpr uint32_t idesc_qk = instr_desc(kPage, false, kRowBlock);
      int g = 0, n = 0, seg = 0;  // ring items, pages, segments handled so far
      while (true) {
        // a segment begins (or the ring ends): the softmax warps say which
        mbar_wait(bar(BAR_Q_READY), seg & 1, abort_flag, dev_status);
        ++seg;
        if (__any_sync(0xffffffffu, *abort_flag != 0) || *ring_done != 0) break;
        ++g;  // the query item
        while (true) {
          const int stage = g % kStages, use = g / kStages;
          mbar_wait(bar(BAR_KV_FULL + stage), use & 1, abort_flag, dev_status);
          const int4 m = meta[g & (kMetaRing - 1)];
          if (n > 0) mbar_wait(bar(BAR_S_FREE), (n - 1) & 1, abort_flag, dev_status);
          tc_fence_after();
          const uint64_t k0 = smem_desc(base + kOffStage + stage * kStageBytes, 16, 1024);
#pragma unroll
          for (int c = 0; c < kChunks; ++c) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              if (elect_one())
                mma_ws_ts(tmem + kColS, tmem + kColQ + c * 32 + kk * 8, desc_advance(k0, c * kSubTileBytes + kk * 32),
                       idesc_qk, (c | kk) ? 1u : 0u);
            }
          }
          if (elect_one()) tc_commit(bar(BAR_S_FULL));
          __syncwarp();
          ++g; ++n;
          if ((m.w & 2) != 0 || m.x != ITEM_PAGE || __any_sync(0xffffffffu, *abort_flag != 0)) break;
        }
      }
    } else if (warp == 6) {
      // ======================================================================== MMA issuer, products
      // Follows the ring in the same way and issues O^T += C^T P^T for a page as soon as its probabilities are
      // there; its commit hands the page's stage back to the TMA warp (the scores of the page are complete by
      // then: the probabilities were made from them).
      constexpr uint32_t idesc_pv = instr_desc(kRowBlock, true);
      int g = 0, n = 0, seg = 0;
      while (true) {
        mbar_wait(bar(BAR_Q_READY), seg & 1, abort_flag, dev_status);
        ++seg;
        if (__any_sync(0xffffffffu, *abort_flag != 0) || *ring_done != 0) break;
        ++g;
        while (true) {
          const int stage = g % kStages, use = g / kStages;
          mbar_wait(bar(BAR_KV_FULL + stage), use & 1, abort_flag, dev_status);
          const int4 m = meta[g & (kMetaRing - 1)];
          // One barrier per P buffer: the softmax warps can deliver P(n) and P(n+1) back to back, and with a single
          // barrier two of its phases could complete before this wait looks at the first.  Per buffer the next
          // phase needs the PV issued below to have completed.
          mbar_wait(bar(BAR_P_READY0 + (n & 1)), (n >> 1) & 1, abort_flag, dev_status);
          tc_fence_after();
          const uint64_t a0 = smem_desc(base + kOffStage + stage * kStageBytes, kSubTileBytes, 1024);
          const uint64_t b0 = smem_desc(base + kOffP + (n & 1) * kPBytes, 16, 1024);
          const uint32_t acc0 = (m.w & 1) != 0 ? 0u : 1u;  // the segment's first page starts the accumulator afresh
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              if (elect_one())
                mma_ss(tmem + kColO + t * 32, desc_advance(a0, (2 * t) * kSubTileBytes + kk * 2048),
                       desc_advance(b0, kk * 32), idesc_pv, kk == 0 ? acc0 : 1u);
            }
          }
          if (elect_one()) {
            tc_commit(bar(BAR_KV_EMPTY + stage));
            tc_commit(bar(BAR_PV_DONE0 + (n & 1)));
          }
          __syncwarp();
          ++g; ++n;
          if ((m.w & 2) != 0 || m.x != ITEM_PAGE || __any_sync(0xffffffffu, *abort_flag != 0)) break;
        }
      }
    } else if (warp < 4) {
      // ======================================================================== softmax + epilogue (warps 0-3)
      const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
      const int my_row = rb * kRowBlock + lane;  // query row of this thread (same in all four replicas)
      int g = 0, n = 0;  // ring items and pages handled so far
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
        const unsigned char* qrow = sm + kOffStage + stage * kStageBytes + lane * 128;
#pragma unroll 1
        for (int c = 0; c < kChunks; ++c) {
          uint32_t v[32];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 x = *reinterpret_cast<const uint4*>(qrow + c * kQTileBytes + ((j ^ (lane & 7)) << 4));
            v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
          }
          tmem_st32(tmem + lane_base + kColQ + c * 32, v);
        }
        tc_wait_st();
        tc_fence_before();
        mbar_arrive(bar(BAR_Q_READY));
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (tid == 0) mbar_arrive(bar(BAR_KV_EMPTY + stage));
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

          mbar_wait(bar(BAR_S_FULL), n & 1, abort_flag, dev_status);
          tc_fence_after();
          uint32_t sq[16];  // this warp's 16 tokens of its row
          tmem_ld16(tmem + lane_base + kColS, sq);
          tc_wait_ld();
          tc_fence_before();
          mbar_arrive(bar(BAR_S_FREE));
          {
            float pmax = -INFINITY;
#pragma unroll
            for (int j = 0; j < 16; ++j)
              pmax = fmaxf(pmax, warp * 16 + j < tok_end ? __uint_as_float(sq[j]) * scale_log2 : -INFINITY);
            pmax_s[(buf * 4 + warp) * 32 + lane] = pmax;
          }
          // one barrier per page: the row maxima meet, and all 128 threads learn together whether the CTA gave up
          int aborted;
          asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, 1, 128, q;\nselp.s32 %0, 1, 0, p;\n}"
                       : "=r"(aborted) : "r"(*abort_flag) : "memory");
          more = (pm.w & 2) == 0 && pm.x == ITEM_PAGE && !aborted;
          // rows [valid, 64) of the page must read as zero; once the CTA has given up, what `pm` says may never have been written
          const int valid = aborted ? kPage : page_ok ? min(kPage, L - pj * kPage) : 0;
          const float rowmax = fmaxf(fmaxf(pmax_s[(buf * 4 + 0) * 32 + lane], pmax_s[(buf * 4 + 1) * 32 + lane]),
                                     fmaxf(pmax_s[(buf * 4 + 2) * 32 + lane], pmax_s[(buf * 4 + 3) * 32 + lane]));
          // Lazy rescale: the reference maximum only moves when some row's new maximum exceeds it by 2^8.  Every
          // warp holds all 32 rows, so the four warps take the same decision without talking to each other.
          float alpha = 1.f;
          bool rescale = false;
          if (first) {
            m_used = rowmax;
          } else {
            // (not after a give-up: what the warps then see may differ, and the rescale has a barrier)
            rescale = __any_sync(0xffffffffu, rowmax > m_used + 8.f) && !aborted;
            if (rescale) {
              const float m_new = fmaxf(m_used, rowmax);
              alpha = (m_new == -INFINITY) ? 1.f : exp2f(m_used - m_new);
              m_used = m_new;
              l_run *= alpha;
            }
          }
          const float m_ref = m_used;

          // ---- probabilities of tokens 16*warp .. 16*warp+15
          uint32_t pk[8];
          float psum = 0.f;
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const int t0 = warp * 16 + j;
            const float p0 = t0 < tok_end ? exp2f(__uint_as_float(sq[j]) * scale_log2 - m_ref) : 0.f;
            const float p1 = t0 + 1 < tok_end ? exp2f(__uint_as_float(sq[j + 1]) * scale_log2 - m_ref) : 0.f;
            psum += p0 + p1;
            pk[j >> 1] = pack_bf16(p0, p1);
          }
          l_run += psum;

          // ---- P buffer `buf` is free once PV of CTA page n-2 is done
          if (n >= 2) mbar_wait(bar(BAR_PV_DONE0 + buf), ((n >> 1) - 1) & 1, abort_flag, dev_status);
          {
            unsigned char* prow = sm + kOffP + buf * kPBytes + lane * 128;
            const int c0w = 2 * warp, sw = lane & 7;
            *reinterpret_cast<uint4*>(prow + ((c0w ^ sw) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *reinterpret_cast<uint4*>(prow + (((c0w + 1) ^ sw) << 4)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          }
          // ---- rows of the page beyond the sequence must contribute exact zeros to O
          if (valid < kPage) {
            unsigned char* pgp = sm + kOffStage + stage * kStageBytes;
            const int rows = kPage - valid;
            for (int i = tid; i < rows * 8 * 8; i += 128) {  // rows x 8 latent sub-tiles x 8 chunks of 16 bytes
              const int rr = valid + i / 64, t = (i >> 3) & 7, ch = i & 7;
              *reinterpret_cast<uint4*>(pgp + t * kSubTileBytes + rr * 128 + ch * 16) = make_uint4(0, 0, 0, 0);
            }
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
        float* dst = o_rows + warp * 32 + lane;
#pragma unroll 1
        for (int t = 0; t < 4; t += 2) {  // two 128-row tiles per round trip to tensor memory
          uint32_t ov[64];
          tmem_ld32(tmem + lane_base + kColO + t * 32, ov);
          tmem_ld32(tmem + lane_base + kColO + (t + 1) * 32, ov + 32);
          tc_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (rb * kRowBlock + j < SH) {
              const float sc = inv_l[j];
              dst[static_cast<size_t>(j) * R + t * 128] = __uint_as_float(ov[j]) * sc;
              dst[static_cast<size_t>(j) * R + (t + 1) * 128] = __uint_as_float(ov[32 + j]) * sc;
            }
          }
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
}  // namespace sm100

bool decode_sm100_supported(const transmla_params_t& p) { return p.kv_lora_rank == sm100::R && p.qk_rope_dim == sm100::DR; }

// Query rows per CTA.  Every row block streams the pages and pays a page's tensor instructions, so with more than 32 rows
// per sequence half as many blocks win (decode_rows64.cu; step, 32 -> 64 rows a CTA: 64 heads S=2 B=64 x 2K-8K 255 -> 193
// us, 32 heads S=2 B=32 x 4K-8K 101 -> 75 us) - unless the batch is so small that a 32-row CTA handles no more than about
// 16 pages (12 with more than two row blocks) anyway: then the shorter start and end of the 32-row kernel count (32 heads
// S=2 B=4 x 4K-8K: 34.1 us against 37.3, B=8 39.8 against 41.3; 64 heads S=2 B=4 x 1K-2K 30.4 against 32.4, x 2K-4K 34.3
// against 34.9, x 4K-8K 42.1 against 40.5).  The rule goes by the page table's capacity: a table with room for much more than a
// small batch holds costs up to 3 us a step (4 x 8192 tokens, 32 heads S=2: 35 against 32).  One kernel with both forms, chosen
// on the device, cost 2 to 4 us in either.
int decode_row_block(const transmla_params_t& p) {
  constexpr int kSms = 148;
  if (!decode_sm100_supported(p) || p.q_len * p.num_heads <= kRowBlock) return kRowBlock;
  const long long blocks = (p.q_len * p.num_heads + kRowBlock - 1) / kRowBlock;
  const long long ctas = (static_cast<long long>(p.batch) * p.max_pages_per_seq + 3) / 4 * blocks;  // of four pages each
  return ctas <= (blocks <= 2 ? 4 : 3) * kSms ? kRowBlock : 64;
}

Partitioning decode_partitioning(const transmla_params_t& p, int G) {
  return {G, p.num_partitions != 0 ? 0 : decode_row_block(p) == 64 ? 8 : 16};
}

// Pages are handed out at run time only when the library chose the partition count itself (a caller who fixes the
// count gets the plan's page ranges, and with them results that do not depend on timing) and only when a sequence
// is shared by 8 or more CTAs: with fewer CTAs per sequence the claims measured no faster than the planned ranges
// (B = 32 and 64 at 8K, ragged B = 32: within 1 %), so those keep the timing-independent plan.
bool dynamic_claims(const transmla_params_t& p, int G) {
  return p.num_partitions == 0 && decode_sm100_supported(p) && G >= 8 * p.batch;
}

cudaError_t launch_decode_sm100(const transmla_params_t& p, int G, const __nv_bfloat16* q_hat,
                                const __nv_bfloat16* cache, const int32_t* page_table, const int32_t* seqlens,
                                const int32_t* cum, const int32_t* plan, float* partial_o, float* partial_lse,
                                int32_t* dev_status, cudaStream_t stream) {
  using namespace sm100;
  // The pool as a 2-D tensor [num_pages * 64 rows, 576 columns]; one box = 64 rows x 64 columns (128 bytes),
  // written to shared memory with the 128-byte swizzle the MMA descriptors expect.  The absorbed queries as a
  // 2-D tensor [B*S*H rows, 576 columns]; one box = 32 rows x 64 columns.
  CUtensorMap map, qmap;
  const int SH = p.q_len * p.num_heads;
  if (!tensor_map_2d(&map, cache, static_cast<uint64_t>(p.num_pages) * kPage, K, kPage) ||
      !tensor_map_2d(&qmap, q_hat, static_cast<uint64_t>(p.batch) * SH, K, kRowBlock))
    return cudaErrorInvalidValue;
  static PerDeviceFlag smem_set;  // zero-initialised; one slot per device
  if (cudaError_t e = ensure_dynamic_smem(decode_sm100_kernel, kSmemBytes, smem_set); e != cudaSuccess) return e;
  dim3 grid(G, (SH + kRowBlock - 1) / kRowBlock);
  int32_t* next = const_cast<int32_t*>(cum) + 3 * p.batch + 1;  // page counters, zeroed by the plan
  return launch_pdl(decode_sm100_kernel, grid, dim3(kThreads), static_cast<size_t>(kSmemBytes), stream, map, qmap,
                    page_table, seqlens, cum, plan, partial_o, partial_lse, dev_status, p.q_len, p.num_heads,
                    p.num_pages, p.max_pages_per_seq, p.softmax_scale * kLog2e, p.batch, dynamic_claims(p, G) ? 1 : 0, next);
}

}  // namespace transmla

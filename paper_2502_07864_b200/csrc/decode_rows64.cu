// Split-KV absorbed-MLA decode (Eq. 9 right, second line) for more than 32 query rows per sequence (S*H > 32),
// r = 512, dR = 64: the kernel of decode_sm100.cu with 64 query rows per CTA.
//
// Why a second kernel: with 32 rows a sequence of 64 (128) query rows has every page streamed by two (four) CTAs, each
// paying the page's 52 tensor instructions (about 1900 cycles whatever the 32 rows hold).  The instructions of the
// weight-stationary form cost the same with 64 rows as with 32 (scores M x 64 tokens: 31 to 35 cycles, products
// M x 256 latents: 78 to 82), so 64 rows halve both the pages through each SM and the tensor time per row.
//   S [64 x 64]  = Q_hat (64 rows: 448 columns of them in tensor memory, 128 in shared memory) x K_hat^T (the page,
//                  K-major), K = 576: 36 instructions
//   O [64 x 512] += P (shared memory, bf16) x C (the same page read MN-major): 4 x 2 instructions of N = 256
// The accumulator of an M = 64 weight-stationary product spreads over all 128 lanes: row i sits in lane i for the first
// half of the columns and in lane 64 + i for the second; an A operand in tensor memory is replicated in both halves.  So
// quadrant q holds the rows 32*(q & 1) + lane, of S the tokens 32*(q >> 1) .. +31, of O the latents of its half.  Eight
// softmax warps share the quadrants, 16 tokens each (with four warps the softmax of a page took 1370 cycles, most of
// them one long dependent stretch per thread, now 1070); a row's factors never leave its four threads.
//
// What bounds it: the tensor instructions of a page (1900 cycles) as long as enough pages are on their way.  A page is
// 2000 to 2400 cycles in coming, stays 3000 in use (scores, softmax, products), and 64 query rows are 72 KB themselves:
// with all of them in shared memory two page stages fit and a page took 3150 cycles.  So tensor memory takes what it
// can of the queries beside O (256 columns) and S (32), and P goes where the page's rope part was once the scores are
// done with it: that makes room for three stages of the pages' latent part and two of the rope part.
// A segment's result leaves through its last page's stage in whole lines: written straight from the lanes, every
// 16-byte store of a warp hit 32 different lines and a segment's end took 12 000 cycles.
//
// Warps 0-3 and 8-11 softmax + epilogue, 4 TMA, 5 scores, 6 products.  Bounded waits and partition walk as in
// decode_sm100.cu.
#include "common.cuh"
#include "partition_walk.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace rows64 {

using namespace sm100;

constexpr int R = 512, DR = 64, K = R + DR;
constexpr int kRows = 64;
constexpr int kSubTileBytes = kPage * 128;            // 8192: 64 rows (tokens or queries) x 64 columns
constexpr int kLatChunks = R / 64;                    // 8 sub-tiles hold a page's latent part; the ninth is the rope part
constexpr int kStageBytes = kLatChunks * kSubTileBytes;  // 65536
constexpr int kStages = 3, kRopeStages = 2;
constexpr int kQTmemChunks = 7;                       // query sub-tiles in tensor memory; sub-tile 7 and the rope part stay in shared
constexpr int kHalves = 2, kHalfChunks = kLatChunks / kHalves;   // a page's latent part is reported in two halves
constexpr int kThreads = 384, kSoftmaxThreads = 256;
constexpr uint32_t kTmemCols = 512;
constexpr int kMetaRing = 8;                          // descriptions of the ring items in flight (a power of two >= 2 * kStages)
enum { ITEM_QUERIES = 1, ITEM_PAGE = 2, ITEM_END = 3 };
constexpr uint32_t kColO = 0, kColS = 256, kColQ = 288;   // O (2 x 128 columns), S (32), Q_hat (7 x 32)

constexpr int kOffLat = 0;
constexpr int kOffRope = kStages * kStageBytes;       // rope part of a page, then its P [64 rows][64 tokens] bf16
constexpr int kOffQ = kOffRope + kRopeStages * kSubTileBytes;
constexpr int kOffBar = kOffQ + 2 * kSubTileBytes;
constexpr int kOffMisc = kOffBar + 256;
// misc: pmax_s[2][8][32] f32, meta[8] int4, tmem base, abort
constexpr int kMiscBytes = 2048 + 16 * kMetaRing + 16;
constexpr int kSmemBytes = kOffMisc + kMiscBytes;
static_assert(kSmemBytes <= 232448 && kOffBar % 256 == 0, "shared memory budget");
static_assert(kRows * 256 * 4 <= kStageBytes, "half of a segment's result passes through a stage");

enum { BAR_LAT_FULL = 0, BAR_LAT_EMPTY = kHalves * kStages, BAR_ROPE_FULL = BAR_LAT_EMPTY + kStages,
       BAR_ROPE_EMPTY = BAR_ROPE_FULL + kRopeStages, BAR_Q_READY = BAR_ROPE_EMPTY + kRopeStages, BAR_Q_EMPTY, BAR_S_FULL,
       BAR_S_FREE, BAR_P_READY, BAR_PV_DONE = BAR_P_READY + 2, BAR_COUNT = BAR_PV_DONE + 2 };
static_assert(BAR_COUNT <= 24, "barrier block");

__global__ void __launch_bounds__(kThreads, 1)
decode_rows64_kernel(const __grid_constant__ CUtensorMap cache_map, const __grid_constant__ CUtensorMap q_map,
                     const int32_t* page_table, const int32_t* seqlens, const int32_t* cum, const int32_t* plan,
                     float* partial_o, float* partial_lse, int32_t* dev_status, int S, int H, int num_pages, int max_pages,
                     float scale_log2, int B, int dynamic, int32_t* next) {
  extern __shared__ __align__(1024) unsigned char smem_aligned[];  // no room to align by hand
  unsigned char* sm = smem_aligned;
  const uint32_t base = smem_u32(sm);
  if ((base & 1023u) != 0) { set_status(dev_status, TRANSMLA_DEV_TIMEOUT); return; }
  float* pmax_s = reinterpret_cast<float*>(sm + kOffMisc);  // [2][8][32]: per page parity, warp, lane
  int4* meta = reinterpret_cast<int4*>(pmax_s + 512);       // [kMetaRing]: what each ring item is
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(meta + kMetaRing);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  auto bar = [&](int i) -> uint32_t { return base + kOffBar + 8 * i; };

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int part = blockIdx.x, rb = blockIdx.y;
  const int SH = S * H;
  pdl_trigger();

  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&cache_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&q_map)) : "memory");
    for (int i = 0; i < kHalves * kStages; ++i) mbar_init(bar(BAR_LAT_FULL + i), 1);
    for (int i = 0; i < kStages; ++i) mbar_init(bar(BAR_LAT_EMPTY + i), 2);   // the scores and the products
    for (int i = 0; i < kRopeStages; ++i) { mbar_init(bar(BAR_ROPE_FULL + i), 1); mbar_init(bar(BAR_ROPE_EMPTY + i), 1); }
    mbar_init(bar(BAR_Q_READY), kSoftmaxThreads);
    mbar_init(bar(BAR_Q_EMPTY), 1);
    mbar_init(bar(BAR_S_FULL), 1);
    mbar_init(bar(BAR_S_FREE), kSoftmaxThreads);
    for (int i = 0; i < 2; ++i) { mbar_init(bar(BAR_P_READY + i), kSoftmaxThreads); mbar_init(bar(BAR_PV_DONE + i), 1); }
    *abort_flag = 0;
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

  if (pl.y > pl.x) {
    if (warp == 4) {
      // ======================================================================== TMA producer
      int g = 0, n = 0, segs = 0;   // ring items, pages and segments issued so far
      const uint64_t stream_policy = l2_evict_first_policy();
      auto acquire = [&]() -> int {
        const int stage = g % kStages, use = g / kStages;
        mbar_wait(bar(BAR_LAT_EMPTY + stage), (use & 1) ^ 1, abort_flag, dev_status);
        return stage;
      };
      auto describe = [&](int4 item) { meta[g & (kMetaRing - 1)] = item; };
      auto issue_queries = [&](int b, int slot, int L) {
        const int stage = acquire();
        mbar_wait(bar(BAR_Q_EMPTY), (segs & 1) ^ 1, abort_flag, dev_status);  // the segment before has its last scores
        if (!*abort_flag && elect_one()) {
          describe(make_int4(ITEM_QUERIES, slot, L, 0));
          const uint32_t full = bar(BAR_LAT_FULL + kHalves * stage);
          mbar_arrive_expect_tx(full, (kLatChunks + 1) * kSubTileBytes);
          const uint32_t dst = base + kOffLat + stage * kStageBytes;
#pragma unroll
          for (int c = 0; c <= kLatChunks; ++c)
            tma_load_2d(c < kQTmemChunks ? dst + c * kSubTileBytes : base + kOffQ + (c - kQTmemChunks) * kSubTileBytes, &q_map,
                        c * 64, b * SH + rb * kRows, full);
          mbar_arrive(full + 8);
        }
        __syncwarp();
        ++segs; ++g;
      };
      auto issue_page = [&](int b, int pj, bool first, bool last) {
        int idx = page_table[static_cast<size_t>(b) * max_pages + pj];
        const bool ok = idx >= 0 && idx < num_pages;
        if (!ok) { if (lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE); idx = 0; }
        const int stage = acquire();
        if (!*abort_flag && elect_one()) {
          describe(make_int4(ITEM_PAGE, pj, ok ? 1 : 0, (first ? 1 : 0) | (last ? 2 : 0)));
          const uint32_t dst = base + kOffLat + stage * kStageBytes;
#pragma unroll
          for (int c = 0; c < kLatChunks; ++c) {
            const uint32_t full = bar(BAR_LAT_FULL + kHalves * stage + c / kHalfChunks);
            if (c % kHalfChunks == 0) mbar_arrive_expect_tx(full, kHalfChunks * kSubTileBytes);
            tma_load_2d_hint(dst + c * kSubTileBytes, &cache_map, c * 64, idx * kPage, full, stream_policy);
          }
        }
        __syncwarp();
        const int slot = n % kRopeStages;
        mbar_wait(bar(BAR_ROPE_EMPTY + slot), ((n / kRopeStages) & 1) ^ 1, abort_flag, dev_status);
        if (!*abort_flag && elect_one()) {
          mbar_arrive_expect_tx(bar(BAR_ROPE_FULL + slot), kSubTileBytes);
          tma_load_2d_hint(base + kOffRope + slot * kSubTileBytes, &cache_map, R, idx * kPage, bar(BAR_ROPE_FULL + slot), stream_policy);
        }
        __syncwarp();
        ++g; ++n;
      };
      const PartitionWalk walk = {page_table, seqlens, cum, next + static_cast<size_t>(rb) * B, partial_lse, part, rb * kRows,
                                  kRows, SH, max_pages, dynamic};
      walk_partition(walk, pl, lane, issue_queries, issue_page);
      {  // closing item
        const int stage = acquire();
        if (elect_one()) {
          describe(make_int4(ITEM_END, 0, 0, 0));
          for (int i = 0; i < kHalves; ++i) mbar_arrive(bar(BAR_LAT_FULL + kHalves * stage + i));
        }
        __syncwarp();
      }
    } else if (warp == 5) {
      // ======================================================================== MMA issuer, scores
      constexpr uint32_t idesc_qk = instr_desc(kPage, false, kRows);
      const uint64_t q7 = smem_desc(base + kOffQ, 16, 1024);
      int n = 0, segs = 0;
      for (int g = 0;; ++g) {
        const int stage = g % kStages, use = g / kStages;
        mbar_wait(bar(BAR_LAT_FULL + kHalves * stage), use & 1, abort_flag, dev_status);
        const int4 m = meta[g & (kMetaRing - 1)];
        if (__any_sync(0xffffffffu, *abort_flag != 0) || m.x == ITEM_END) break;
        if (m.x == ITEM_QUERIES) {
          mbar_wait(bar(BAR_Q_READY), segs & 1, abort_flag, dev_status);  // moved to tensor memory
          ++segs;
          if (elect_one()) mbar_arrive(bar(BAR_LAT_EMPTY + stage));
          __syncwarp();
          continue;
        }
        if (n > 0) mbar_wait(bar(BAR_S_FREE), (n - 1) & 1, abort_flag, dev_status);
        const uint64_t k0 = smem_desc(base + kOffLat + stage * kStageBytes, 16, 1024);
        const int slot = n % kRopeStages;
#pragma unroll
        for (int i = 0; i < kHalves; ++i) {
          if (i > 0) mbar_wait(bar(BAR_LAT_FULL + kHalves * stage + i), use & 1, abort_flag, dev_status);
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int c = i * kHalfChunks; c < (i + 1) * kHalfChunks; ++c) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const uint64_t bd = desc_advance(k0, c * kSubTileBytes + kk * 32);
                if (c < kQTmemChunks)
                  mma_ws_ts(tmem + kColS, tmem + kColQ + c * 32 + kk * 8, bd, idesc_qk, (c | kk) ? 1u : 0u);
                else
                  mma_ws_ss(tmem + kColS, desc_advance(q7, kk * 32), bd, idesc_qk, 1u);
              }
            }
          }
        }
        mbar_wait(bar(BAR_ROPE_FULL + slot), (n / kRopeStages) & 1, abort_flag, dev_status);
        tc_fence_after();
        const uint64_t r0 = smem_desc(base + kOffRope + slot * kSubTileBytes, 16, 1024);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_ws_ss(tmem + kColS, desc_advance(q7, kSubTileBytes + kk * 32), desc_advance(r0, kk * 32), idesc_qk, 1u);
          tc_commit(bar(BAR_S_FULL));
          tc_commit(bar(BAR_LAT_EMPTY + stage));
          if (m.w & 2) tc_commit(bar(BAR_Q_EMPTY));
        }
        __syncwarp();
        ++n;
      }
    } else if (warp == 6) {
      // ======================================================================== MMA issuer, products
      constexpr uint32_t idesc_pv = instr_desc(256, false, kRows) | (1u << 16);  // B (the page) MN-major
      int n = 0, segs = 0;
      for (int g = 0;; ++g) {
        const int stage = g % kStages, use = g / kStages;
        mbar_wait(bar(BAR_LAT_FULL + kHalves * stage), use & 1, abort_flag, dev_status);
        const int4 m = meta[g & (kMetaRing - 1)];
        if (__any_sync(0xffffffffu, *abort_flag != 0) || m.x == ITEM_END) break;
        if (m.x == ITEM_QUERIES) {
          mbar_wait(bar(BAR_Q_READY), segs & 1, abort_flag, dev_status);
          ++segs;
          if (elect_one()) mbar_arrive(bar(BAR_LAT_EMPTY + stage));
          __syncwarp();
          continue;
        }
        const int slot = n % kRopeStages;
        mbar_wait(bar(BAR_P_READY + slot), (n / kRopeStages) & 1, abort_flag, dev_status);
        tc_fence_after();
        const uint64_t p0 = smem_desc(base + kOffRope + slot * kSubTileBytes, 16, 1024);
        const uint64_t v0 = smem_desc(base + kOffLat + stage * kStageBytes, kSubTileBytes, 1024);
        const uint32_t acc0 = (m.w & 1) != 0 ? 0u : 1u;  // the segment's first page starts the accumulator afresh
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
              mma_ws_ss(tmem + kColO + hf * 128, desc_advance(p0, kk * 32),
                        desc_advance(v0, hf * 4 * kSubTileBytes + kk * 2048), idesc_pv, kk == 0 ? acc0 : 1u);
          }
          if ((m.w & 2) == 0) {  // the stage and P of a segment's last page go back after its epilogue
            tc_commit(bar(BAR_LAT_EMPTY + stage));
            tc_commit(bar(BAR_ROPE_EMPTY + slot));
          }
          tc_commit(bar(BAR_PV_DONE + (n & 1)));
        }
        __syncwarp();
        ++n;
      }
    } else if (warp < 4 || warp >= 8) {
      // ======================================================================== softmax + epilogue (warps 0-3, 8-11)
      const int quad = warp & 3, sub = warp >> 3;                  // quadrant; which 16 of its 32 tokens
      const int sw = quad + 4 * sub, stid = sw * 32 + lane;        // softmax warp 0..7, thread 0..255
      const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
      const int row = 32 * (quad & 1) + lane, half = quad >> 1;    // this thread's row of the block; half of the tokens / latents
      const int tok0 = 32 * half + 16 * sub;                       // its first token of every page
      const int my_row = rb * kRows + row;
      const int behind = S - 1 - my_row / H;  // the newest tokens that this row's position does not see
      const bool pos_scale = scale_log2 >= 0.f;
      int g = 0, n = 0;
      // Looks at ring item g, all 256 threads together.  Queries: this thread's row goes to tensor memory, sub-tile by
      // sub-tile (each of a quadrant's two warps takes some), the issuers are told, `seg` gets the segment's slot and length,
      // and true is returned.  They give the stage back.  Otherwise the ring has ended or the CTA gave up.
      auto open_segment = [&](int2& seg) -> bool {
        const int stage = g % kStages;
        mbar_wait(bar(BAR_LAT_FULL + kHalves * stage), (g / kStages) & 1, abort_flag, dev_status);
        const int4 m = meta[g & (kMetaRing - 1)];
        int stop;
        asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, 1, 256, q;\nselp.s32 %0, 1, 0, p;\n}"
                     : "=r"(stop) : "r"(static_cast<int>(*abort_flag != 0 || m.x != ITEM_QUERIES)) : "memory");
        if (stop) return false;
        seg = make_int2(m.y, m.z);
        const unsigned char* qrow = sm + kOffLat + stage * kStageBytes + row * 128;
#pragma unroll 1
        for (int c = sub * 4; c < (sub ? kQTmemChunks : 4); ++c) {
          uint32_t v[32];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 x = *reinterpret_cast<const uint4*>(qrow + c * kSubTileBytes + ((j ^ (row & 7)) << 4));
            v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
          }
          tmem_st32(tmem + lane_base + kColQ + c * 32, v);
        }
        tc_wait_st();
        tc_fence_before();
        mbar_arrive(bar(BAR_Q_READY));
        ++g;
        return true;
      };
      int2 seg, next_seg;   // slot of the segment's partial and length of its sequence
      bool open = open_segment(seg);
      while (open) {
        float m_used = -INFINITY, l_run = 0.f;
        bool more = true;
        while (more) {
          const int stage = g % kStages, slot = n % kRopeStages, buf = n & 1;
          mbar_wait(bar(BAR_LAT_FULL + kHalves * stage), (g / kStages) & 1, abort_flag, dev_status);
          const int4 pm = meta[g & (kMetaRing - 1)];
          const int L = seg.y, pj = pm.y;
          const bool page_ok = pm.x == ITEM_PAGE && pm.z != 0;
          const int n_vis = my_row < SH ? L - behind : 0;
          const int tok_end = page_ok ? n_vis - pj * kPage - tok0 : 0;   // of this thread's 16 tokens, [0, tok_end) are visible
          const bool first = (pm.w & 1) != 0, last = (pm.w & 2) != 0;
          const bool full = __all_sync(0xffffffffu, tok_end >= 16) && pos_scale;   // no masking

          uint32_t sq[16];
          // The products of page n-2 are done before the scores of page n (whose rope part is loaded after them), so this
          // wait costs nothing; it sees to it that every phase of the two barriers is looked at in turn.  With one barrier
          // for all pages the wait for a segment's last products could meet the phase of the page before, whose parity
          // reads as done: the softmax can be a whole page ahead of the products.
          if (n >= 2) mbar_wait(bar(BAR_PV_DONE + buf), ((n >> 1) - 1) & 1, abort_flag, dev_status);
          mbar_wait(bar(BAR_S_FULL), n & 1, abort_flag, dev_status);
          tc_fence_after();
          tmem_ld16(tmem + lane_base + kColS + 16 * sub, sq);
          tc_wait_ld();
          tc_fence_before();
          mbar_arrive(bar(BAR_S_FREE));
          {
            float a = -INFINITY;
            if (full) {
              float c2 = __uint_as_float(sq[1]);
              a = __uint_as_float(sq[0]);
#pragma unroll
              for (int j = 2; j < 16; j += 2) { a = fmaxf(a, __uint_as_float(sq[j])); c2 = fmaxf(c2, __uint_as_float(sq[j + 1])); }
              a = fmaxf(a, c2) * scale_log2;
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j) a = fmaxf(a, j < tok_end ? __uint_as_float(sq[j]) * scale_log2 : -INFINITY);
            }
            pmax_s[(buf * 8 + sw) * 32 + lane] = a;
          }
          // One barrier per page: the four parts of a row's maximum meet, and all 256 threads learn together whether the
          // CTA gave up.
          int aborted;
          asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 q, %1, 0;\nbar.red.or.pred p, 1, 256, q;\nselp.s32 %0, 1, 0, p;\n}"
                       : "=r"(aborted) : "r"(*abort_flag) : "memory");
          more = !last && pm.x == ITEM_PAGE && !aborted;
          // rows [valid, 64) of the page must read as zero; once the CTA has given up, what `pm` says may never have been written
          const int valid = aborted ? kPage : page_ok ? min(kPage, L - pj * kPage) : 0;
          // The row's four threads: both warps of quadrants quad and quad ^ 2.
          float rowmax = -INFINITY;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            rowmax = fmaxf(rowmax, pmax_s[(buf * 8 + (quad & 1) + 2 * i) * 32 + lane]);
          // Lazy rescale: the reference maximum only moves when some row's new maximum exceeds it by 2^8.  The warps that
          // share 32 rows see the same maxima and decide alike.
          bool rescale = false;
          float alpha = 1.f;
          if (first) {
            m_used = rowmax;
          } else {
            rescale = __any_sync(0xffffffffu, rowmax > m_used + 8.f);
            if (rescale) {
              const float m_new = fmaxf(m_used, rowmax);
              alpha = (m_new == -INFINITY) ? 1.f : exp2f(m_used - m_new);
              m_used = m_new;
              l_run *= alpha;
            }
          }
          const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used;
          uint32_t pk[8];
          float ps0 = 0.f, ps1 = 0.f;
          if (full) {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const float p0 = ex2_approx(fmaf(__uint_as_float(sq[j]), scale_log2, neg_m));
              const float p1 = ex2_approx(fmaf(__uint_as_float(sq[j + 1]), scale_log2, neg_m));
              ps0 += p0; ps1 += p1;
              pk[j >> 1] = pack_bf16(p0, p1);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const float p0 = j < tok_end ? ex2_approx(fmaf(__uint_as_float(sq[j]), scale_log2, neg_m)) : 0.f;
              const float p1 = j + 1 < tok_end ? ex2_approx(fmaf(__uint_as_float(sq[j + 1]), scale_log2, neg_m)) : 0.f;
              ps0 += p0; ps1 += p1;
              pk[j >> 1] = pack_bf16(p0, p1);
            }
          }
          l_run += ps0 + ps1;

          // P takes the place of the page's rope part, which the scores have read
          {
            unsigned char* prow = sm + kOffRope + slot * kSubTileBytes + row * 128;
            const int c0 = tok0 >> 3, x = row & 7;
            *reinterpret_cast<uint4*>(prow + ((c0 ^ x) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *reinterpret_cast<uint4*>(prow + (((c0 + 1) ^ x) << 4)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          }
          if (valid < kPage) {  // rows of the page beyond the sequence must contribute exact zeros to O
            unsigned char* pgp = sm + kOffLat + stage * kStageBytes;
            const int rows = kPage - valid;
            for (int i = stid; i < rows * 8 * 8; i += kSoftmaxThreads) {  // rows x 8 latent sub-tiles x 8 chunks of 16 bytes
              const int rr = valid + i / 64, t = (i >> 3) & 7, ch = i & 7;
              *reinterpret_cast<uint4*>(pgp + t * kSubTileBytes + rr * 128 + ch * 16) = make_uint4(0, 0, 0, 0);
            }
          }
          if (rescale) {  // warp-uniform; each of a quadrant's two warps takes half of its 256 columns
            // O is at rest once the products of the page before are done
            if (n >= 1) mbar_wait(bar(BAR_PV_DONE + (buf ^ 1)), ((n - 1) >> 1) & 1, abort_flag, dev_status);
            tc_fence_after();
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
              uint32_t ov[32];
              tmem_ld32(tmem + lane_base + kColO + sub * 128 + t * 32, ov);
              tc_wait_ld();
#pragma unroll
              for (int j = 0; j < 32; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * alpha);
              tmem_st32(tmem + lane_base + kColO + sub * 128 + t * 32, ov);
            }
            tc_wait_st();
          }
          fence_proxy_async();
          tc_fence_before();
          mbar_arrive(bar(BAR_P_READY + slot));
          ++g; ++n;
        }

        // ---- epilogue of the segment.  The queries of the next one go to tensor memory first (every score of this
        // segment has been read), so that its first scores run meanwhile.  Once this segment's last product is there,
        // the place of its last P and the last page's stage are free: the four parts of a row's sum meet in the first;
        // O, normalised, passes through the second, 256 latents of the 64 rows at a time, and leaves in whole lines.
        const int last_stage = (g - 1) % kStages, last_slot = (n - 1) % kRopeStages;
        const int out_slot = seg.x;
        open = open_segment(next_seg);
        seg = next_seg;
        mbar_wait(bar(BAR_PV_DONE + ((n - 1) & 1)), ((n - 1) >> 1) & 1, abort_flag, dev_status);
        tc_fence_after();
        float* l_s = reinterpret_cast<float*>(sm + kOffRope + last_slot * kSubTileBytes);  // [8][32]
        l_s[stid] = l_run;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        float l_tot = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) l_tot += l_s[((quad & 1) + 2 * i) * 32 + lane];
        const float inv = l_tot > 0.f ? 1.f / l_tot : 0.f;
        if (half == 0 && sub == 0 && my_row < SH)
          partial_lse[static_cast<size_t>(out_slot) * SH + my_row] = l_tot > 0.f ? (m_used + log2f(l_tot)) * kLn2 : -INFINITY;
        unsigned char* out_s = sm + kOffLat + last_stage * kStageBytes;
        float* dst = partial_o + (static_cast<size_t>(out_slot) * SH + rb * kRows) * R;
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t ov[64];
          tmem_ld32(tmem + lane_base + kColO + hf * 128 + sub * 64, ov);
          tmem_ld32(tmem + lane_base + kColO + hf * 128 + sub * 64 + 32, ov + 32);
          tc_wait_ld();
          if (hf == 1) asm volatile("bar.sync 1, 256;" ::: "memory");  // the first half has left the staging rows
          unsigned char* srow = out_s + row * 1024;   // 64 chunks of 16 bytes, swizzled by the row
#pragma unroll
          for (int j = 0; j < 64; j += 4)
            *reinterpret_cast<float4*>(srow + (((half * 32 + sub * 16 + j / 4) ^ (row & 7)) << 4)) =
                make_float4(__uint_as_float(ov[j]) * inv, __uint_as_float(ov[j + 1]) * inv, __uint_as_float(ov[j + 2]) * inv,
                            __uint_as_float(ov[j + 3]) * inv);
          asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 16; ++i) {  // a warp takes 8 rows, half a row (512 bytes) at a time
            const int rr = sw * 8 + (i >> 1), ch = (i & 1) * 32 + lane;
            if (rb * kRows + rr < SH)
              *reinterpret_cast<float4*>(dst + static_cast<size_t>(rr) * R + hf * 256 + ch * 4) =
                  *reinterpret_cast<const float4*>(out_s + rr * 1024 + ((ch ^ (rr & 7)) << 4));
          }
        }
        fence_proxy_async();  // stage and slot were used here; their next contents come through the async proxy
        tc_fence_before();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (stid == 0) {
          mbar_arrive(bar(BAR_LAT_EMPTY + last_stage));
          mbar_arrive(bar(BAR_ROPE_EMPTY + last_slot));
        }
      }
    }
  }

  // ---- teardown: everyone arrives, tensor memory is returned
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

}  // namespace rows64

cudaError_t launch_decode_rows64(const transmla_params_t& p, int G, const __nv_bfloat16* q_hat, const __nv_bfloat16* cache,
                                 const int32_t* page_table, const int32_t* seqlens, const int32_t* cum, const int32_t* plan,
                                 float* partial_o, float* partial_lse, int32_t* dev_status, cudaStream_t stream) {
  using namespace rows64;
  CUtensorMap map, qmap;  // boxes of 64 rows x 64 columns of the pool and of the absorbed queries, 128-byte swizzle
  const int SH = p.q_len * p.num_heads;
  if (!tensor_map_2d(&map, cache, static_cast<uint64_t>(p.num_pages) * kPage, K, kPage) ||
      !tensor_map_2d(&qmap, q_hat, static_cast<uint64_t>(p.batch) * SH, K, kRows))
    return cudaErrorInvalidValue;
  static PerDeviceFlag smem_set;
  if (cudaError_t e = ensure_dynamic_smem(decode_rows64_kernel, kSmemBytes, smem_set); e != cudaSuccess) return e;
  dim3 grid(G, (SH + kRows - 1) / kRows);
  int32_t* next = const_cast<int32_t*>(cum) + 3 * p.batch + 1;  // page counters, zeroed by the plan
  return launch_pdl(decode_rows64_kernel, grid, dim3(kThreads), static_cast<size_t>(kSmemBytes), stream, map, qmap,
                    page_table, seqlens, cum, plan, partial_o, partial_lse, dev_status, p.q_len, p.num_heads,
                    p.num_pages, p.max_pages_per_seq, p.softmax_scale * kLog2e, p.batch, dynamic_claims(p, G) ? 1 : 0, next);
}

}  // namespace transmla

// What a decode step needs before its split-KV kernel, on the Blackwell tensor path (r = 512, dR = 64, dn = 128), in one
// launch of any of three kinds of blocks:
//   append   (Eq. 7 left) clusters of eight CTAs: 64 features x up to 64 tokens of y = [W_DKV; W_KR] x, an eighth of D each,
//            through a ring of asynchronous copies (the weights of its first three pieces from before the dependency wait),
//            D [64 features x 64 tokens] += W [64 x 16] X^T as weight-stationary M = 64 products; the CTAs' sums meet
//            through distributed shared memory, CTA i finishes the i-th eighth of the tokens: RoPE, bf16, page slot (or fp32
//            rows for the FP8 append's quantiser).  A value is the same sum in the same order whatever the token count.
//   plan     the split plan (plan_block.cuh)
//   absorb   (Eq. 9 right, first line) a block a head and 256 latents: q_hat [rows x 256] = q_nope [rows x 128] W_UK_h, 128 rows a
//            time as weight-stationary products of 64 rows (82 cycles for 64 x 256 x 16; the plain form takes 286 for 128);
//            the block with a head's first latents copies the rope part
// A barrier wait that gives up (which no launch should see) is reported, and what the block had still to write becomes NaN.
// What bounds it: chains of round trips (look-ups and operands, sums of the other CTAs, stores), 3 to 5 us.  The mma.sync tiles
// of small_kernels.cu, 16 cycles each on a quarter of an SM, made that 6 us at 16 tokens, 15 at 128 and 22 with 64 heads, where
// their registers also allowed two blocks an SM of twice as many.
#include "append_block.cuh"
#include "common.cuh"
#include "plan_block.cuh"
#include "skinny_gemm.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace sm100 {

constexpr int kPrR = 512, kPrDR = 64, kPrDn = 128, kPrRow = kPrR + kPrDR;
constexpr int kPrTok = 64;                                // tokens a cluster
constexpr int kPrSub = 64 * 128;                          // 64 rows x 64 bf16, 128-byte swizzle
// The append's ring has pieces of 128 of the contracted dimension: the weights (2 kPrSub), then the activations of as many
// tokens as there are, in eights.  Four pieces where they fit (32 tokens), which is all of D = 4096, otherwise three.
// (The products read 64 tokens' rows: beyond those of a piece whatever follows, at the end up to kPrSub beyond the ring.)
constexpr int kPrRing = 3 * 4 * kPrSub;
constexpr int kPrQ = 65536;                               // absorb: weights [4][128 x 64] from 0, queries [2][128 x 64] from kPrQ
constexpr int kPrMisc = kPrRing + kPrSub;                 // barriers, tensor-memory base, abort flag
constexpr int kPrSmem = kPrMisc + 256 + 1024;             // and alignment
constexpr int kPrSums = kPrTok + 8;                       // pitch of the sums, floats, [token][feature]
static_assert(kPrQ + 2 * 128 * 128 <= kPrMisc && kPrTok * kPrSums * 4 <= kPrMisc && kPrMisc % 256 == 0, "shared memory map");
static_assert(kPlanSmemSeqs * 4 <= kPrMisc, "the plan's prefix sums");

struct PrologueArgs {
  const __nv_bfloat16* x;
  const __nv_bfloat16* w_dkv_kr;
  const int32_t* pos_base;     // token (b, s) sits at pos_base[b] + pos_shift + s
  const int32_t* page_table;
  __nv_bfloat16* cache;
  float* rows_f32;             // not null: the rows go here, in token order, instead of the cache
  const __nv_bfloat16* q_nope;
  const __nv_bfloat16* q_pe;
  const __nv_bfloat16* w_uk;
  __nv_bfloat16* q_hat;
  const int32_t* seqlens;
  int32_t* cum;
  int32_t* plan;
  int32_t* dev_status;
  int pos_shift, B, S, H, D, num_pages, max_pages;
  int n_append, others;        // clusters; blocks behind them: the plan's (if any) and the absorb's
  float theta;
  Partitioning parts;
};

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}
// 16-byte chunk c of row rr of a 128-byte-swizzled tile whose rows are 64 bf16
__device__ __forceinline__ uint32_t swizzled(int rr, int c) { return rr * 128 + ((c ^ (rr & 7)) << 4); }

constexpr int kPrWhere = TRANSMLA_DEV_IN_PROLOGUE;
constexpr uint32_t kPrNan = 0x7fffffffu;

template <long long kLimit>
__device__ __forceinline__ void append_role(const PrologueArgs& a, unsigned char* sm, uint32_t base, uint32_t* tmem_base_s,
                                            volatile int* abort_flag) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x % kSliceCtas, cluster = blockIdx.x / kSliceCtas;
  constexpr int kFTiles = kPrRow / 64;
  const int f0 = cluster % kFTiles * 64, t0 = cluster / kFTiles * kPrTok, T = a.B * a.S, K = a.D;
  const int rows = min(kPrTok, T - t0), x_sub = ((rows + 7) & ~7) * 128, piece_bytes = 2 * kPrSub + 2 * x_sub;
  const int ring = 4 * piece_bytes <= kPrRing ? 4 : 3;
  const int k_lo = rank * (K / kSliceCtas), k_hi = k_lo + K / kSliceCtas, pieces = (K / kSliceCtas + 127) / 128;
  auto bar = [&](int i) -> uint32_t { return base + kPrMisc + 8 * i; };
  auto copy = [&](int piece, const __nv_bfloat16* src, int count, int at, int sub) {  // 16 bytes a thread and turn
    unsigned char* dst = sm + piece % ring * piece_bytes + at;
    for (int i = tid; i < count * 16; i += 256) {
      const int rr = i >> 4, c = i & 15, k = k_lo + piece * 128 + c * 8;
      const bool in = k < k_hi;  // the rest of a short piece is filled with zeros
      cp_async16(dst + (c >> 3) * sub + swizzled(rr, c & 7), src + (in ? static_cast<size_t>(rr) * K + k : 0), in ? 16 : 0);
    }
  };
  const __nv_bfloat16* w = a.w_dkv_kr + static_cast<size_t>(f0) * K;
  const __nv_bfloat16* x = a.x + static_cast<size_t>(t0) * K;
  for (int p = 0; p < ring && p < pieces; ++p) copy(p, w, 64, 0, kPrSub);
  cp_async_commit();
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(bar(i), 1);  // 4: the last product
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(tmem_base_s, 32);
  // This thread's token and pair of features, of those that its CTA finishes
  const int t = t0 + rank * (kPrTok / kSliceCtas) + warp, f = f0 + 2 * lane;
  const bool rotated = f >= kPrR;
  const double freq = rotated ? rope_freq((f - kPrR) >> 1, kPrDR, a.theta) : 0.0;
  tc_fence_before();
  pdl_wait();  // activations and everything that is written may belong to kernels still in flight; weights may not
  for (int p = 0; p < ring; ++p) {
    if (p < pieces) copy(p, x, rows, 2 * kPrSub, x_sub);  // (tokens beyond the last: whatever is there; columns of a product do not mix)
    cp_async_commit();
  }
  bool mine = t < T;
  float cs = 1.f, sn = 0.f;
  __nv_bfloat16* dst = nullptr;
  if (mine) {
    const int b = t / a.S, pos = a.pos_base[b] + a.pos_shift + t % a.S;
    if (a.rows_f32 == nullptr) {
      const int pj = pos / kPage;
      int page = -1;
      if (pos >= 0 && pj < a.max_pages) page = a.page_table[static_cast<size_t>(b) * a.max_pages + pj];
      if (page < 0 || page >= a.num_pages) {
        set_status(a.dev_status, TRANSMLA_DEV_BAD_PAGE);
        mine = false;
      } else {
        dst = a.cache + (static_cast<size_t>(page) * kPage + pos % kPage) * kPrRow;
      }
    }
    if (rotated) rope_angle(pos, freq, cs, sn);
  }
  for (int p = 0; p < pieces; ++p) {
    // (the weights' group, one of activations a piece of the first ring, then one an iteration)
    if (p == 0) { if (ring == 4) cp_async_wait<3>(); else cp_async_wait<2>(); }
    else if (ring == 4) cp_async_wait<2>();
    else cp_async_wait<1>();
    fence_proxy_async();
    __syncthreads();
    if (warp == 0) {
      tc_fence_after();
      const uint32_t tmem = *tmem_base_s;
      const uint32_t at = base + p % ring * piece_bytes;
      const uint64_t w0 = smem_desc(at, 16, 1024), x0 = smem_desc(at + 2 * kPrSub, 16, 1024);
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          mma_ws_ss(tmem, desc_advance(w0, (kk >> 2) * kPrSub + (kk & 3) * 32), desc_advance(x0, (kk >> 2) * x_sub + (kk & 3) * 32), instr_desc(kPrTok, false, 64), (p | kk) != 0);
        }
        tc_commit(bar(p + 1 < pieces ? p % ring : 4));
      }
      __syncwarp();
    }
    if (p > 0) {
      const int q = p + ring - 1;
      if (q < pieces) {
        if (mbar_wait<kLimit, kPrWhere>(bar((p - 1) % ring), ((p - 1) / ring) & 1, abort_flag, a.dev_status)) {
          copy(q, w, 64, 0, kPrSub);
          copy(q, x, rows, 2 * kPrSub, x_sub);
        }
      }
      cp_async_commit();
    }
  }
  const bool done = mbar_wait<kLimit, kPrWhere>(bar(4), 0, abort_flag, a.dev_status);
  const bool bad = __any_sync(0xffffffffu, !done || *abort_flag != 0);
  if (bad) mbar_retire(bar(4), 0);
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  float* sums = reinterpret_cast<float*>(sm);  // [token][kPrSums]: every product has completed
  {
    // feature i of tokens 0-31 in lane i, of tokens 32-63 in lane 64 + i
    const int quad = warp & 3, hf = warp >> 2, feature = (quad & 1) * 32 + lane, tok = (quad >> 1) * 32 + hf * 16;
    uint32_t v[16];
    tmem_ld16(tmem + (static_cast<uint32_t>(quad * 32) << 16) + hf * 16, v);
    tc_wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) sums[(tok + j) * kPrSums + feature] = __uint_as_float(bad ? kPrNan : v[j]);
  }
  tc_fence_before();
  slice_cluster_sync();
  if (mine) {
    const uint32_t local = smem_u32(sums + (t - t0) * kPrSums + 2 * lane);
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
    const float nre = re * cs - im * sn, nim = im * cs + re * sn;
    if (rotated) { re = nre; im = nim; }
    if (a.rows_f32 != nullptr) *reinterpret_cast<float2*>(a.rows_f32 + static_cast<size_t>(t) * kPrRow + f) = make_float2(re, im);
    else *reinterpret_cast<uint32_t*>(dst + f) = pack_bf16(re, im);
  }
  slice_cluster_sync();  // nobody leaves while its memory may still be read
  tc_fence_after();
  if (warp == 0) tmem_free(tmem, 32);
}

template <long long kLimit>
__device__ __forceinline__ void absorb_role(const PrologueArgs& a, int h, int half, unsigned char* sm, uint32_t base,
                                            uint32_t* tmem_base_s, volatile int* abort_flag) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, BS = a.B * a.S, H = a.H;
  const uint32_t bar = base + kPrMisc;
  const __nv_bfloat16* w = a.w_uk + static_cast<size_t>(h) * kPrDn * kPrR + half * 256;
#pragma unroll
  for (int i = tid; i < kPrDn * 32; i += 256) {  // [4 x 64 latents][128 k][64]: N-major
    const int k = i >> 5, c = i & 31;
    cp_async16(sm + (c >> 3) * (2 * kPrSub) + swizzled(k, c & 7), w + static_cast<size_t>(k) * kPrR + c * 8, 16);
  }
  cp_async_commit();
  if (tid == 0) {
    mbar_init(bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(tmem_base_s, 256);
  tc_fence_before();
  pdl_wait();  // the queries may come from the kernel before this one; the weights above may not
  int tile = 0;
  uint32_t tmem = 0;
  for (int p0 = 0; p0 < BS; p0 += 128, ++tile) {
    const int rows = min(128, BS - p0);
    if (tile > 0) __syncthreads();  // the tile before has left the queries' place
    for (int i = tid; i < rows * 16; i += 256) {  // (rows beyond the last: whatever is there; rows of a product do not mix)
      const int rr = i >> 4, c = i & 15;
      cp_async16(sm + kPrQ + (c >> 3) * (2 * kPrSub) + swizzled(rr, c & 7), a.q_nope + (static_cast<size_t>(p0 + rr) * H + h) * kPrDn + c * 8, 16);
    }
    cp_async_commit();
    if (half == 0) {  // the rope part is a plain copy, made while the operands are on their way
      for (int i0 = tid; i0 < rows * 8; i0 += 256 * 4) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * 256;
          v[u] = make_uint4(0, 0, 0, 0);
          if (i < rows * 8) v[u] = ld_u128(a.q_pe + (static_cast<size_t>(p0 + (i >> 3)) * H + h) * kPrDR + (i & 7) * 8);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * 256;
          if (i < rows * 8) *reinterpret_cast<uint4*>(a.q_hat + (static_cast<size_t>(p0 + (i >> 3)) * H + h) * kPrRow + kPrR + (i & 7) * 8) = v[u];
        }
      }
    }
    cp_async_wait<0>();
    fence_proxy_async();
    __syncthreads();
    tc_fence_after();
    tmem = *tmem_base_s;
    if (warp == 0) {
      const uint64_t q0 = smem_desc(base + kPrQ, 16, 1024), w0 = smem_desc(base, 2 * kPrSub, 1024);
      if (elect_one()) {
        for (int m = 0; m * 64 < rows; ++m) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_ws_ss(tmem + m * 128, desc_advance(q0, m * kPrSub + (kk >> 2) * 2 * kPrSub + (kk & 3) * 32), desc_advance(w0, kk * 2048),
                      instr_desc(256, false, 64) | (1u << 16), kk != 0);
        }
        tc_commit(bar);
      }
      __syncwarp();
    }
    const bool done = mbar_wait<kLimit, kPrWhere>(bar, tile & 1, abort_flag, a.dev_status);
    const bool bad = __any_sync(0xffffffffu, !done || *abort_flag != 0);
    if (bad) mbar_retire(bar, tile & 1);
    tc_fence_after();
    // Write-out: 32 rows x 64 latents a warp (rows i of latents 0-127 in lane i, of 128-255 in lane 64 + i), through the warp's own
    // 4 KB of the queries' place, whole lines.
    const int quad = warp & 3, n0 = (quad >> 1) * 128 + (warp >> 2) * 64;
    unsigned char* mine = sm + kPrQ + warp * 4096;
    for (int m = 0; m * 64 < rows; ++m) {
      const int r0 = m * 64 + (quad & 1) * 32;
      if (r0 >= rows) continue;
      uint32_t v[64];
      const uint32_t addr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + m * 128 + (warp >> 2) * 64;
      tmem_ld32(addr, v);
      tmem_ld32(addr + 32, v + 32);
      tc_wait_ld();
      if (bad) {
#pragma unroll
        for (int e = 0; e < 64; ++e) v[e] = kPrNan;
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint32_t* e = v + 8 * c;
        auto two = [&](int i) { return pack_bf16(__uint_as_float(e[i]), __uint_as_float(e[i + 1])); };
        *reinterpret_cast<uint4*>(mine + swizzled(lane, c)) = make_uint4(two(0), two(2), two(4), two(6));
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int rr = i * 4 + (lane >> 3), c = lane & 7;
        const uint4 o = *reinterpret_cast<const uint4*>(mine + swizzled(rr, c));
        if (r0 + rr < rows)
          *reinterpret_cast<uint4*>(a.q_hat + (static_cast<size_t>(p0 + r0 + rr) * H + h) * kPrRow + half * 256 + n0 + c * 8) = o;
      }
      __syncwarp();
    }
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_free(*tmem_base_s, 256);
}

template <long long kLimit>
__global__ void __launch_bounds__(256, 2) prologue_sm100_kernel(const __grid_constant__ PrologueArgs a) {
  extern __shared__ unsigned char smem_unaligned[];
  const uint32_t raw = smem_u32(smem_unaligned), base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_unaligned + (base - raw);
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(sm + kPrMisc + 128);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  pdl_trigger();
  const int bid = static_cast<int>(blockIdx.x) - a.n_append * kSliceCtas;
  if (bid < 0) append_role<kLimit>(a, sm, base, tmem_base_s, abort_flag);
  else if (bid >= a.others) return;  // the grid is whole clusters
  else if (bid == 0) plan_block(a.seqlens, a.B, a.parts, (a.S * a.H + kRowBlock - 1) / kRowBlock, a.max_pages, a.cum, a.plan, a.dev_status, sm);
  else absorb_role<kLimit>(a, (bid - 1) >> 1, (bid - 1) & 1, sm, base, tmem_base_s, abort_flag);
}

}  // namespace sm100

bool prologue_sm100_supported(const transmla_params_t& p) {
  return p.kv_lora_rank == sm100::kPrR && p.qk_rope_dim == sm100::kPrDR && p.qk_nope_dim == sm100::kPrDn;
}

template <long long kLimit = kWaitCycles>
static cudaError_t launch_prologue_sm100(const transmla_params_t& p, sm100::PrologueArgs& a, bool append, bool absorb, cudaStream_t stream) {
  auto kernel = sm100::prologue_sm100_kernel<kLimit>;
  a.B = p.batch; a.S = p.q_len; a.H = p.num_heads; a.D = p.hidden_dim;
  a.num_pages = p.num_pages; a.max_pages = p.max_pages_per_seq; a.theta = p.rope_theta;
  a.n_append = append ? sm100::kPrRow / 64 * ((p.batch * p.q_len + sm100::kPrTok - 1) / sm100::kPrTok) : 0;
  a.others = absorb ? 1 + 2 * p.num_heads : 0;
  static PerDeviceFlag smem_set;
  if (cudaError_t e = ensure_dynamic_smem(kernel, sm100::kPrSmem, smem_set); e != cudaSuccess) return e;
  if (!append)  // small blocks that need not find room in eights beside the kernel before them
    return launch_pdl(kernel, dim3(a.others), dim3(256), static_cast<size_t>(sm100::kPrSmem), stream, a);
  return launch_slices(kernel, (a.n_append + (a.others + kSliceCtas - 1) / kSliceCtas) * kSliceCtas,
                       static_cast<size_t>(sm100::kPrSmem), stream, a);
}

cudaError_t launch_append_sm100(const transmla_params_t& p, const __nv_bfloat16* x, const __nv_bfloat16* w, const int32_t* positions,
                                const int32_t* page_table, __nv_bfloat16* cache, float* rows_f32, int32_t* dev_status, cudaStream_t stream) {
  sm100::PrologueArgs a = {};
  a.x = x; a.w_dkv_kr = w; a.pos_base = positions; a.page_table = page_table; a.cache = cache; a.rows_f32 = rows_f32;
  a.dev_status = dev_status;
  return launch_prologue_sm100(p, a, true, false, stream);
}

cudaError_t launch_absorb_sm100(const transmla_params_t& p, const Partitioning& parts, const __nv_bfloat16* x, const __nv_bfloat16* w_dkv_kr,
                                const int32_t* page_table, __nv_bfloat16* cache, const __nv_bfloat16* q_nope, const __nv_bfloat16* q_pe,
                                const __nv_bfloat16* w_uk, __nv_bfloat16* q_hat, const int32_t* seqlens, int32_t* cum, int32_t* plan,
                                int32_t* dev_status, cudaStream_t stream, bool give_up) {
  sm100::PrologueArgs a = {};
  a.x = x; a.w_dkv_kr = w_dkv_kr; a.pos_base = seqlens; a.pos_shift = -p.q_len; a.page_table = page_table; a.cache = cache;
  a.q_nope = q_nope; a.q_pe = q_pe; a.w_uk = w_uk; a.q_hat = q_hat; a.seqlens = seqlens; a.cum = cum; a.plan = plan;
  a.parts = parts; a.dev_status = dev_status;
  return give_up ? launch_prologue_sm100<0>(p, a, x != nullptr, true, stream) : launch_prologue_sm100(p, a, x != nullptr, true, stream);
}

}  // namespace transmla

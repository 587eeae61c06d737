// Combine + up-projection (Eq. 9 right, last line before W_O) for many query rows on the Blackwell tensor path (r = 512, dv = 128).
// Block = one head x kRows query rows: sixteen warps merge the split partials into shared memory as a bf16 high/low pair, then
// out [rows x 128] = (o_hi + o_lo) W_UV_h^T as weight-stationary products of 32 or 64 rows; W_UV_h comes by asynchronous copies
// from before the dependency wait.
// A barrier wait that gives up (which no launch should see) is reported, and the block's part of out becomes NaN.
// What bounds it: the partials (30 bytes a cycle and SM from L2) and the look-ups before them.  The mma.sync form (small_kernels.cu)
// spends 16 cycles of an SM's quarter on each 16 x 8 x 16 product: 9 us of the launch with 64 heads x 128 rows, 5 with 32 x 128,
// 3 with 32 x 64.  Fewer rows than that (one wave of blocks of 8) stay there: its products take 1 to 2 us, and its
// weights wait in registers.
#include "combine.cuh"
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace sm100 {

constexpr int kCbR = 512, kCbDv = 128, kCbThreads = 512, kCbWSub = kCbDv * 128;  // 128 columns of out x 64 latents

template <int kRows>
struct CombineMap {
  static constexpr int kM = kRows <= 32 ? 32 : 64;            // rows of a product
  static constexpr int kSub = kM * 128;                       // rows x 64 latents
  static constexpr int kSlots = kRows <= 32 ? 8 : 6;          // of W_UV_h's eight pieces of 64 latents, as many as fit
  static constexpr int kLo = 8 * kSub, kW = 16 * kSub, kMisc = kW + kSlots * kCbWSub, kBytes = kMisc + 256 + 1024;
  static_assert(kBytes <= 232448 && kMisc % 256 == 0, "shared memory budget");
};

template <int kRows, long long kLimit>
__global__ void __launch_bounds__(kCbThreads, 1)
combine_sm100_kernel(const int32_t* cum, const int32_t* plan, const float* partial_o, const float* partial_lse,
                     const __nv_bfloat16* __restrict__ w_uv, __nv_bfloat16* out, float* lse_out, int32_t* dev_status, int B, int S, int H, int G) {
  using Map = CombineMap<kRows>;
  constexpr int kAtOnce = kRows > 16 ? 2 : 1, kSegs = 4 / kAtOnce;
  extern __shared__ unsigned char smem_unaligned[];
  const uint32_t raw = smem_u32(smem_unaligned), base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_unaligned + (base - raw);
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(sm + Map::kMisc + 128);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  constexpr int kWhere = TRANSMLA_DEV_IN_COMBINE;
  auto bar = [&](int i) -> uint32_t { return base + Map::kMisc + 8 * i; };  // 0: all products; 1, 2: those with pieces 0 and 1
  pdl_trigger();
  const int h = blockIdx.x, bs0 = blockIdx.y * kRows, BS = B * S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto copy_weights = [&](int piece) {
    unsigned char* dst = sm + Map::kW + piece % Map::kSlots * kCbWSub;
    const __nv_bfloat16* src = w_uv + static_cast<size_t>(h) * kCbDv * kCbR + piece * 64;
#pragma unroll
    for (int i = tid; i < kCbDv * 8; i += kCbThreads) {
      const int n = i >> 3, c = i & 7;
      cp_async16(dst + n * 128 + ((c ^ (n & 7)) << 4), src + static_cast<size_t>(n) * kCbR + c * 8, 16);
    }
  };
  for (int piece = 0; piece < Map::kSlots; ++piece) copy_weights(piece);
  cp_async_commit();
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) mbar_init(bar(i), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  constexpr uint32_t kCols = Map::kM == 32 ? 32 : 64;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(kCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();  // the partials and the prefix sums come from the kernels before this one
  const MergeArgs merge = {cum, plan, partial_o, partial_lse, B, S, H, kCbR, G};
#pragma unroll 1
  for (int r0 = warp; r0 < kRows; r0 += 16 * kAtOnce) {
    float o[kAtOnce][4][4], lse[kAtOnce];
    merge_rows<kAtOnce, 4, kSegs>(merge, h, bs0 + r0, 16, lane * 4, o, lse);
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      const int rr = r0 + 16 * u;
      if (lse_out != nullptr && lane == 0 && bs0 + rr < BS) lse_out[static_cast<size_t>(bs0 + rr) * H + h] = lse[u];
#pragma unroll
      for (int c = 0; c < 4; ++c) {  // latents c * 128 + 4 lane ..: 8 bytes of a 128-byte-swizzled row
        const float (&v)[4] = o[u][c];
        float lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) lo[e] = v[e] - __bfloat162float(__float2bfloat16_rn(v[e]));
        const int off = (2 * c + (lane >> 4)) * Map::kSub + rr * 128 + ((((lane & 15) >> 1) ^ (rr & 7)) << 4) + (lane & 1) * 8;
        *reinterpret_cast<uint2*>(sm + off) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
        *reinterpret_cast<uint2*>(sm + Map::kLo + off) = make_uint2(pack_bf16(lo[0], lo[1]), pack_bf16(lo[2], lo[3]));
      }
    }
  }
  cp_async_wait<0>();
  fence_proxy_async();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  // (Rows of a product that have not been written are whatever is there: rows do not mix, and nothing of them is stored.)
  auto products = [&](int piece) {
    const uint64_t hi = smem_desc(base + piece * Map::kSub, 16, 1024), lo = smem_desc(base + Map::kLo + piece * Map::kSub, 16, 1024);
    const uint64_t w = smem_desc(base + Map::kW + piece % Map::kSlots * kCbWSub, 16, 1024);
    constexpr uint32_t idesc = instr_desc(kCbDv, false, Map::kM);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      mma_ws_ss(tmem, desc_advance(lo, kk * 32), desc_advance(w, kk * 32), idesc, (piece | kk) != 0);
      mma_ws_ss(tmem, desc_advance(hi, kk * 32), desc_advance(w, kk * 32), idesc, 1u);
    }
  };
  if (warp == 0) {
    if (elect_one()) {
      for (int piece = 0; piece < Map::kSlots; ++piece) {
        products(piece);
        if (Map::kSlots + piece < 8) tc_commit(bar(1 + piece));
      }
      if (Map::kSlots == 8) tc_commit(bar(0));
    }
    __syncwarp();
  }
  if (Map::kSlots < 8) {  // the last pieces take the places of the first
    for (int piece = Map::kSlots; piece < 8; ++piece) {
      if (mbar_wait<kLimit, kWhere>(bar(1 + piece - Map::kSlots), 0, abort_flag, dev_status)) copy_weights(piece);
    }
    cp_async_commit();
    cp_async_wait<0>();
    fence_proxy_async();
    __syncthreads();
    if (warp == 0) {
      if (elect_one()) {
        for (int piece = Map::kSlots; piece < 8; ++piece) products(piece);
        tc_commit(bar(0));
      }
      __syncwarp();
    }
  }
  const bool done = mbar_wait<kLimit, kWhere>(bar(0), 0, abort_flag, dev_status);
  const bool bad = __any_sync(0xffffffffu, !done || *abort_flag != 0);
  if (bad) mbar_retire(bar(0), 0);
  tc_fence_after();
  // 32 rows: quadrant q has columns 32 q ..; 64 rows: row i of columns 0-63 in lane i, of 64-127 in lane 64 + i.  16 columns a warp.
  const int quad = warp & 3, part = warp >> 2;
  if (Map::kM == 64 || part < 2) {
    const int rr = Map::kM == 32 ? lane : (quad & 1) * 32 + lane, n0 = Map::kM == 32 ? quad * 32 + part * 16 : (quad >> 1) * 64 + part * 16;
    uint32_t v[16];
    tmem_ld16(tmem + (static_cast<uint32_t>(quad * 32) << 16) + part * 16, v);
    tc_wait_ld();
    if (rr < kRows && bs0 + rr < BS) {
      auto two = [&](int i) { return bad ? 0x7fff7fffu : pack_bf16(__uint_as_float(v[i]), __uint_as_float(v[i + 1])); };
      uint4* dst = reinterpret_cast<uint4*>(out + (static_cast<size_t>(bs0 + rr) * H + h) * kCbDv + n0);
      dst[0] = make_uint4(two(0), two(2), two(4), two(6));
      dst[1] = make_uint4(two(8), two(10), two(12), two(14));
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

}  // namespace sm100

bool combine_sm100_supported(const transmla_params_t& p) { return p.kv_lora_rank == sm100::kCbR && p.v_dim == sm100::kCbDv; }

template <long long kLimit>
static cudaError_t launch_rows(const transmla_params_t& p, int G, const int32_t* cum, const int32_t* plan, const float* partial_o,
                               const float* partial_lse, const __nv_bfloat16* w_uv, __nv_bfloat16* out, float* lse_out,
                               int32_t* dev_status, cudaStream_t stream) {
  using namespace sm100;
  const int BS = p.batch * p.q_len, H = p.num_heads;
  static PerDeviceFlag smem_set[3];
  auto launch = [&](auto kernel, int rows, int bytes, PerDeviceFlag& set) -> cudaError_t {
    if (cudaError_t e = ensure_dynamic_smem(kernel, bytes, set); e != cudaSuccess) return e;
    return launch_pdl(kernel, dim3(H, (BS + rows - 1) / rows), dim3(kCbThreads), static_cast<size_t>(bytes), stream, cum, plan, partial_o,
                      partial_lse, w_uv, out, lse_out, dev_status, p.batch, p.q_len, H, G);
  };
  // One wave of blocks, one an SM, with as few rows a block as that allows; beyond a wave as many rows a block as there are, up
  // to 64: W_UV_h is then read less often.  16 / 32 / 64 rows a block, alone: 160 heads x 16 rows 10.8 / 11.9 / 15.1 us, x 32 16.4 / 13.1 / 16.2;
  // 512 x 32 47.0 / 34.6 / 41.7; 1.7 waves of 64 (64 x 256) 39.5 / 26.6 / 20.2 (mma.sync, 16 rows 37.2), 2.2 (32 x 300) 26.7 / 18.9 / 18.5 (26.7),
  // just over one (64 x 129) 22.0 / 17.8 / 16.9 (21.0).
  constexpr int kSms = 148;
  auto blocks = [&](int rows) { return static_cast<long long>(H) * ((BS + rows - 1) / rows); };
  if (blocks(16) <= kSms || BS <= 16) return launch(combine_sm100_kernel<16, kLimit>, 16, CombineMap<16>::kBytes, smem_set[0]);
  if (blocks(32) <= kSms || BS <= 32) return launch(combine_sm100_kernel<32, kLimit>, 32, CombineMap<32>::kBytes, smem_set[1]);
  return launch(combine_sm100_kernel<64, kLimit>, 64, CombineMap<64>::kBytes, smem_set[2]);
}

cudaError_t launch_combine_sm100(const transmla_params_t& p, int G, const int32_t* cum, const int32_t* plan, const float* partial_o,
                                 const float* partial_lse, const __nv_bfloat16* w_uv, __nv_bfloat16* out, float* lse_out,
                                 int32_t* dev_status, cudaStream_t stream, bool give_up) {
  return (give_up ? launch_rows<0> : launch_rows<kWaitCycles>)(p, G, cum, plan, partial_o, partial_lse, w_uv, out, lse_out, dev_status, stream);
}

}  // namespace transmla

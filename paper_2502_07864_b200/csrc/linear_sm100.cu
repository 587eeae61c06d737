// Weight-streaming linear maps on the Blackwell tensor path: y[M, N] = x[M, K] w[N, K]^T for the few tokens of a
// decode step (Eq. 8 right column: c^Q, q^C, q^R; Eq. 9 last line: W_O).
//
// The weights are the large operand (tens of MB, read once), the activations the small one.  A CTA owns 128
// output features and one slice of K:
//   D^T[128 features x T tokens] += W_tile[128 x 64] (A, shared memory, K-major) x X_tile[T x 64]^T (B, K-major)
// with the accumulator in tensor memory, so that the 128 lanes of the MMA are always full whatever the number of
// tokens (16 <= T <= 256, tokens padded to a multiple of 16; rows beyond M read as zero through the tensor map).
// Per CTA the shared-memory traffic is (128 + T) x K_slice x 2 bytes, i.e. the activations are re-read once per
// 128 features, not once per 8 or 32 as in the mma.sync tiles of skinny_gemm.cuh.
// K is cut into `splits` slices so that every SM streams weights (N / 128 tiles alone would occupy 32-48 SMs).
// The slices of a tile are the CTAs of one thread-block cluster: each leaves its fp32 partial in its own shared
// memory (the ring is free by then), and after a cluster barrier every CTA adds the slices of its share of the
// tokens in slice order, reading the others' shared memory directly, applies RoPE where asked and writes bf16 (no
// float atomics: reruns give the same bits).
// What bounds it: the weight stream, 585 cycles a stage at 16 tokens, which is 31 bytes a cycle and SM and over the SMs in use
// also about the HBM rate, and what stands at either end of the stream.  The ring takes the whole shared memory and is filled with weights before the CTA waits for the kernel
// before it (half the ring beside that kernel's CTAs, with the rest requested for L2, was 6 to 30 us slower a layer: the
// requests go through the same path as the loads).  The code behind the stream is small: unrolled over the tokens, with its
// sine at 16 places, its fetch from memory took 9 to 12 thousand cycles of a launch's 28 to 35 thousand, now 4.
// The layer step of LLaMA-2-7B, 16 x 8192 tokens: 86 -> 71 us with the append among the tiles (75 without), 128 short
// sequences 120 -> 98; Qwen2.5-72B, 40 short sequences: 222 -> 127 (all against the mma.sync tiles below 48 tokens and the
// unrolled epilogue).
//
// Warps: 0 TMA producer, 1 MMA issuer, 2-5 epilogue (each owns the 32 tensor-memory lanes of its quadrant).
#include "common.cuh"
#include "linear_args.cuh"
#include "skinny_gemm.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace sm100 {

constexpr int kLinBM = 128;                      // output features per CTA
constexpr int kLinBK = 64;                       // contracted elements per ring stage (128 bytes per row)
constexpr int kLinMaxT = 256;                    // tokens per CTA at most (MMA N)
constexpr int kLinMaxStages = 12;
constexpr int kLinWBytes = kLinBM * 128;         // 16384
constexpr int kLinRingBytes = 221184;            // stages of (weight tile + activation tile); as many as fit, at most 12
constexpr int kLinThreads = 192;
constexpr int kLinSmemBytes = kLinRingBytes + 256 + 1024;
enum { LB_FULL = 0, LB_EMPTY = kLinMaxStages, LB_DONE = 2 * kLinMaxStages };

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// four floats at the same shared-memory offset in the CTA of rank `rank` of this cluster
__device__ __forceinline__ float4 ld_cluster_f32x4(const float* local, uint32_t rank) {
  uint32_t remote;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(remote) : "memory");
  return v;
}
struct LinSm100Params {
  __nv_bfloat16* out[3];   // [M, N_j]; job 2 is the append (Eq. 7 left): the cache
  int N[3];                // output features of job j (multiples of 128, but for the append's r + dR)
  int rope_d[2];           // > 0: consecutive blocks of rope_d features are rotated (Eq. 1, d := rope_d)
  int tiles01[2];          // tiles of jobs 0 and 1; those behind belong to the append
  int M, S, K, splits;
  const int32_t* page_table;
  int r, dR, num_pages, max_pages;
  int stages;              // ring depth: as many (weight tile + activation box) stages as fit
  int x_box_rows;          // rows of the activation box (tokens of a full block, padded to 16)
  const int32_t* pos_base; // position of token (b, s) = pos_base[b] + pos_shift + s (rotated jobs only)
  int pos_shift;
  float theta;
};

__global__ void __launch_bounds__(kLinThreads, 1)
linear_sm100_kernel(const __grid_constant__ CUtensorMap w_map0, const __grid_constant__ CUtensorMap w_map1,
                    const __grid_constant__ CUtensorMap w_map2, const __grid_constant__ CUtensorMap x_map, const LinSm100Params p, int32_t* dev_status) {
  extern __shared__ unsigned char smem_unaligned[];
  const uint32_t raw = smem_u32(smem_unaligned);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_unaligned + (base - raw);
  const uint32_t bar_base = base + kLinRingBytes;
  auto bar = [&](int i) -> uint32_t { return bar_base + 8 * i; };
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(sm + kLinRingBytes + 8 * (2 * kLinMaxStages + 1));
  const int kLinStages = p.stages;
  const uint32_t kLinStageBytes = kLinWBytes + static_cast<uint32_t>(p.x_box_rows) * 128u;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = blockIdx.x / p.splits, split = blockIdx.x % p.splits;
  const int tiles0 = p.tiles01[0], tiles1 = p.tiles01[1];
  const int job = tile < tiles0 ? 0 : tile < tiles0 + tiles1 ? 1 : 2;
  const int f0 = (tile - (job == 0 ? 0 : job == 1 ? tiles0 : tiles0 + tiles1)) * kLinBM;  // first output feature within the job
  const int t0 = blockIdx.y * kLinMaxT;                        // first token of the block
  const int T = min(kLinMaxT, p.M - t0);                       // tokens of this block
  const int TP = (T + 15) & ~15;                               // MMA N
  const int ktiles = p.K / kLinBK;
  const int kt0 = static_cast<int>(static_cast<long long>(split) * ktiles / p.splits);
  const int kt1 = static_cast<int>(static_cast<long long>(split + 1) * ktiles / p.splits);
  const CUtensorMap* w_map = job == 0 ? &w_map0 : job == 1 ? &w_map1 : &w_map2;
  uint32_t tmem_cols = 32;
  while (tmem_cols < static_cast<uint32_t>(TP)) tmem_cols <<= 1;
  pdl_trigger();

  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(w_map)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&x_map)) : "memory");
    for (int i = 0; i < kLinMaxStages; ++i) { mbar_init(bar(LB_FULL + i), 1); mbar_init(bar(LB_EMPTY + i), 1); }
    mbar_init(bar(LB_DONE), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  const uint32_t stage_tx = kLinStageBytes;  // rows of the activation box beyond M arrive as zeros

  if (warp == 0) {
    // ======================================================================== TMA producer
    // Weights do not depend on earlier kernels of the stream: the first stages' weight tiles are requested before
    // the dependency wait, their activation tiles after it.
    const int n_it = kt1 - kt0, early = min(n_it, kLinStages);
    for (int i = 0; i < early; ++i) {
      if (elect_one()) {
        mbar_arrive_expect_tx(bar(LB_FULL + i), stage_tx);
        tma_load_2d(base + i * kLinStageBytes, w_map, (kt0 + i) * kLinBK, f0, bar(LB_FULL + i));
      }
      __syncwarp();
    }
    pdl_wait();
    for (int i = 0; i < early; ++i) {
      if (elect_one()) tma_load_2d(base + i * kLinStageBytes + kLinWBytes, &x_map, (kt0 + i) * kLinBK, t0, bar(LB_FULL + i));
      __syncwarp();
    }
    for (int i = early; i < n_it; ++i) {
      const int stage = i % kLinStages, use = i / kLinStages;
      mbar_wait(bar(LB_EMPTY + stage), (use & 1) ^ 1, abort_flag, dev_status);
      if (!*abort_flag && elect_one()) {
        mbar_arrive_expect_tx(bar(LB_FULL + stage), stage_tx);
        tma_load_2d(base + stage * kLinStageBytes, w_map, (kt0 + i) * kLinBK, f0, bar(LB_FULL + stage));
        tma_load_2d(base + stage * kLinStageBytes + kLinWBytes, &x_map, (kt0 + i) * kLinBK, t0, bar(LB_FULL + stage));
      }
      __syncwarp();
    }
  } else if (warp == 1) {
    // ======================================================================== MMA issuer
    const uint32_t idesc = instr_desc(TP, false);
    const int n_it = kt1 - kt0;
    pdl_wait();  // no activations arrive before: the bounded waits below must not count the kernel before this one
    for (int i = 0; i < n_it; ++i) {
      const int stage = i % kLinStages, use = i / kLinStages;
      mbar_wait(bar(LB_FULL + stage), use & 1, abort_flag, dev_status);
      tc_fence_after();
      const uint64_t a0 = smem_desc(base + stage * kLinStageBytes, 16, 1024);
      const uint64_t b0 = smem_desc(base + stage * kLinStageBytes + kLinWBytes, 16, 1024);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        if (elect_one()) mma_ss(tmem, desc_advance(a0, kk * 32), desc_advance(b0, kk * 32), idesc, (i | kk) ? 1u : 0u);
      }
      if (elect_one()) tc_commit(bar(LB_EMPTY + stage));
      __syncwarp();
    }
    if (elect_one()) tc_commit(bar(LB_DONE));
    __syncwarp();
  } else {
    // ======================================================================== epilogue (warps 2-5)
    const int quad = warp & 3;                                 // tensor-memory lanes 32*quad .. 32*quad+31
    const int fl = quad * 32 + lane;                           // feature of this thread within the tile
    const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
    const int N = p.N[job], rope_d = job < 2 ? p.rope_d[job] : 0;
    float* part_s = reinterpret_cast<float*>(sm);              // [T][128]: the ring is free when every MMA has retired
    const int f = f0 + 4 * lane;                               // the lane's four features in the second half
    const int rot_d = job < 2 ? rope_d : p.dR, rot_from = job < 2 ? 0 : p.r;
    const bool rotated = rot_d > 0 && f >= rot_from && f < N;
    double freq[2] = {};                                       // angles in fp64, as in the mma.sync tiles
    if (rotated)
      for (int i = 0; i < 2; ++i) freq[i] = rope_freq(((f - rot_from + 2 * i) % rot_d) >> 1, rot_d, p.theta);
    pdl_wait();  // the output may still be in use by earlier kernels
    mbar_wait(bar(LB_DONE), 0, abort_flag, dev_status);
    tc_fence_after();
#pragma unroll 1
    for (int c = 0; c < TP; c += 16) {
      uint32_t v[16];
      tmem_ld16(tmem + lane_base + c, v);
      tc_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j) part_s[(c + j) * kLinBM + fl] = __uint_as_float(v[j]);
    }
    tc_fence_before();
    // The slices of the tile meet: CTA `split` adds the slices of its share of the tokens, a warp a token.
    cluster_sync_all();
    const int share = (T + p.splits - 1) / p.splits, te = min(T, (split + 1) * share);
#pragma unroll 1
    for (int t = split * share + quad; t < te; t += 4) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int s = 0; s < p.splits; ++s) {
        const float4 v = ld_cluster_f32x4(part_s + t * kLinBM + 4 * lane, s);
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
      }
      const int tok = t0 + t, pos = rot_d > 0 || job == 2 ? p.pos_base[tok / p.S] + p.pos_shift + tok % p.S : 0;
      if (rotated) {
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {  // one copy of the sine's code
          rope_pair_at(acc.x, acc.y, pos, freq[0]);
          acc = make_float4(acc.z, acc.w, acc.x, acc.y);
          const double g = freq[0];
          freq[0] = freq[1];
          freq[1] = g;
        }
      }
      size_t row = tok;
      if (job == 2) {  // the token's slot of the cache
        const int b = tok / p.S, pj = pos / kPage;
        int page = -1;
        if (pos >= 0 && pj < p.max_pages) page = p.page_table[static_cast<size_t>(b) * p.max_pages + pj];
        if (page < 0 || page >= p.num_pages) {
          if (lane == 0) set_status(dev_status, TRANSMLA_DEV_BAD_PAGE);
          continue;
        }
        if (f >= N) continue;
        row = static_cast<size_t>(page) * kPage + pos % kPage;
      }
      *reinterpret_cast<uint2*>(p.out[job] + row * N + f) = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
    }
  }
  if (warp < 2) cluster_sync_all();
  cluster_sync_all();  // nobody leaves while its memory may still be read

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
}

static bool encode_2d(CUtensorMap* map, const void* ptr, int rows, int cols, int box_rows) {
  return tensor_map_2d(map, ptr, static_cast<uint64_t>(rows), static_cast<uint32_t>(cols), static_cast<uint32_t>(box_rows), kLinBK);
}

}  // namespace sm100

// Slices of K per 128-feature tile wanted: as many as keep tiles x slices within the SM count of a B200, each at least four
// stages long, at most the portable size of a cluster.
static int linear_sm100_splits(int n_tiles, int K) {
  const int ktiles = K / sm100::kLinBK;
  int s = 148 / n_tiles;
  if (s > 8) s = 8;
  if (s > ktiles / 4) s = ktiles / 4;
  return s < 1 ? 1 : s;
}

// Where this kernel can be used: whole tiles of 128 features, whole ring stages, enough of both to be worth a launch of
// this kind (smaller maps are not measured).
bool linear_sm100_supported(const LinearArgs& a) {
  if (a.n_jobs < 1 || a.n_jobs > 2 || a.job[0].K < 512) return false;
  int tiles = 0;
  for (int j = 0; j < a.n_jobs; ++j) tiles += a.job[j].N / sm100::kLinBM;
  if (tiles < 4) return false;
  for (int j = 0; j < a.n_jobs; ++j) {
    if (a.job[j].N % sm100::kLinBM || a.job[j].K % sm100::kLinBK || a.job[j].K != a.job[0].K || a.job[j].x != a.job[0].x) return false;
    if (a.job[j].rope_d % 2) return false;
  }
  return true;
}

// The append can ride along: a lane's four features are all latent or all rope key.
bool linear_sm100_takes_append(const AppendJob& ap, const LinearArgs& a) {
  return ap.x == a.job[0].x && ap.D == a.job[0].K && ap.r % 4 == 0 && ap.dR % 4 == 0;
}

cudaError_t launch_linear_sm100(const LinearArgs& a, int32_t* dev_status, cudaStream_t stream) {
  using namespace sm100;
  LinSm100Params p = {};
  CUtensorMap wmap[3], xmap;
  int tiles = 0;
  for (int j = 0; j < a.n_jobs; ++j) {
    p.out[j] = a.job[j].out; p.N[j] = a.job[j].N; p.rope_d[j] = a.job[j].rope_d;
    if (!encode_2d(&wmap[j], a.job[j].w, a.job[j].N, a.job[j].K, kLinBM)) return cudaErrorInvalidValue;
    p.tiles01[j] = a.job[j].N / kLinBM;
    tiles += p.tiles01[j];
  }
  if (a.n_jobs == 1) wmap[1] = wmap[0];
  wmap[2] = wmap[0];
  if (a.append.blocks > 0) {
    const AppendJob& ap = a.append;
    p.out[2] = ap.cache; p.N[2] = ap.r + ap.dR; p.page_table = ap.page_table;
    p.r = ap.r; p.dR = ap.dR; p.num_pages = ap.num_pages; p.max_pages = ap.max_pages;
    if (!encode_2d(&wmap[2], ap.w, p.N[2], ap.D, kLinBM)) return cudaErrorInvalidValue;
    tiles += (p.N[2] + kLinBM - 1) / kLinBM;
  }
  const int T = a.M < kLinMaxT ? a.M : kLinMaxT;
  p.x_box_rows = (T + 15) & ~15;
  p.stages = kLinRingBytes / (kLinWBytes + p.x_box_rows * 128);
  if (p.stages > kLinMaxStages) p.stages = kLinMaxStages;
  if (!encode_2d(&xmap, a.job[0].x, a.M, a.job[0].K, p.x_box_rows)) return cudaErrorInvalidValue;
  p.M = a.M; p.S = a.S; p.K = a.job[0].K;
  p.splits = linear_sm100_splits(tiles, p.K);
  p.pos_base = a.pos_base; p.pos_shift = a.pos_shift; p.theta = a.theta;
  static PerDeviceFlag smem_set;  // zero-initialised; one slot per device
  if (cudaError_t e = ensure_dynamic_smem(linear_sm100_kernel, kLinSmemBytes, smem_set); e != cudaSuccess) return e;
  const int token_blocks = (a.M + kLinMaxT - 1) / kLinMaxT;
  // The K slices of a tile are launched as one thread-block cluster (they are neighbours in blockIdx.x).  All clusters
  // have to fit on the device at once, one CTA per SM (a cluster lives inside one GPC, so fewer fit than SMs / size
  // suggests): the slice count is lowered until they do.
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kLinThreads);
  cfg.dynamicSmemBytes = kLinSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  static PerDeviceFlag max_clusters[9];  // co-resident clusters of each size on each device, asked once (0 = not yet)
  const int slot = current_device_slot();
  for (; p.splits > 1; --p.splits) {
    attr[1].val.clusterDim.x = p.splits;
    cfg.gridDim = dim3(tiles * p.splits, token_blocks);
    int fit = slot >= 0 ? max_clusters[p.splits].value[slot].load(std::memory_order_acquire) : 0;
    if (fit == 0) {
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, linear_sm100_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = -1; }
      fit = n > 0 ? n : -1;
      if (slot >= 0) max_clusters[p.splits].value[slot].store(fit, std::memory_order_release);
    }
    if (fit >= tiles * token_blocks) break;
  }
  attr[1].val.clusterDim.x = p.splits;
  cfg.gridDim = dim3(tiles * p.splits, token_blocks);
  return cudaLaunchKernelEx(&cfg, linear_sm100_kernel, wmap[0], wmap[1], wmap[2], xmap, p, dev_status);
}

}  // namespace transmla

// fp32 matrix products of the conversion on the Blackwell tensor path: C[M,N] = alpha * op(A) op(B).
//
// Every fp32 operand value is split exactly into three bf16 terms, x = hi + mid + lo (8 + 8 + 8 significand bits, each
// rounded to nearest, so a term is at most 2^-8 of the one before), and a product is the six term products down to 2^-16 of
// the largest; the three left out are below 2^-23 and of either sign, as the rounding of an fp32 product is.  The tensor
// core adds into its fp32 accumulator by truncation, which over thousands of steps would be a bias: an accumulator takes
// one chunk of K (32) only, then the worker threads add it to fp32 sums in their registers, rounding to nearest.  Relative
// error of a sum of 8192 products 2.6e-7 (a chain of fp32 multiply-adds: 1.4e-6; four chunks an accumulator: 8.8e-7).
// The terms are exact for 2^-110 <= |x| < 3.39e38 (the largest bf16 value): beyond, see the write-out.
// A barrier wait that gives up (which no launch should see) raises TRANSMLA_DEV_TIMEOUT where the caller has a status word,
// and what the CTA has not finished becomes NaN: the issuer stops then, so that everybody whose sums are not complete gives
// up as well.
//
// A CTA pair (cta_group::2) works on a 256 x 256 tile of C, or a single CTA on a 128 x 128 one; either way a CTA converts
// 128 rows of op(A) and 128 columns of op(B) a chunk.  Converting warps read fp32 (whole 128-byte lines whatever the storage
// order) ahead, split, and write the terms to a four-stage ring in shared memory - K-major where K is contiguous in memory
// (64-byte swizzle), MN-major where it is not (128-byte swizzle, 64-wide pieces).  Adding warps drain the accumulators (two, in
// tensor memory).  One warp of the pair's first CTA issues the products.
// A pair has eight warps of either kind, 128 sums a thread, a chunk ahead: an accumulator has to be drained while the product
// behind it runs (1540 cycles), and with all sixteen warps doing both it waited for the conversion its warp was in, 2730 cycles
// a chunk; now about 1800, of which the converters wait 1100 for a free stage.  What bounds it is the tensor pipe under the
// power limit: 6 x 240 TFLOP/s of bf16 products, which is the rate cuBLAS sustains for seconds, at 1.45 GHz.
// A single CTA's product is a quarter of that, and converting bounds its chunks.  Where A's K is not contiguous all sixteen
// warps do both, two groups of eight taking the chunks in turn, 32 sums a thread; otherwise eight and eight, 64 sums a thread, two
// chunks ahead.  One kind / two kinds, a single CTA a tile: covariance of 16 x 128 x 128 x 16384 (ta) 564 / 613 us, 512 x 4096 x 8064 (ta) 241 /
// 250, 128 x 128 x 4096 (ta) 114.7 / 114.7, (tb) 112.6 / 106.5; 1024 x 1024 x 4096 (tb) 114.7 / 109.3; 4096 x 512 x 4096 (tb) 114.7 / 116.7.
// Rates (fp32 products), before -> now: 8192 x 4096 x 4096 218 -> 241 TFLOP/s, X^T X of 8192 x 8064 370 -> 436 (half of it
// mirrored), 8064 x 512 x 8064 196 -> 228; the fp32 multiply-add kernel before those reached 48, 50 and 42.
// (Arrivals that release to the other CTA wait for the thread's loads in flight: none in the converters.  fp32 pieces fetched
// through shared memory: more of its traffic, no gain.  Two fp16 terms and three products a value: 311, 512 and 240 TFLOP/s,
// but errors 5 to 25 % larger, and no range.)
#include "conversion.cuh"
#include "sm100_ptx.cuh"

namespace transmla {
namespace conv {

using namespace sm100;

namespace {

constexpr int kRows = 128, kKc = 32;           // rows of op(A) and columns of op(B) a CTA converts; K per chunk
constexpr int kStages = 4;
constexpr int kConverters = 256, kAdders = 256, kThreads = kConverters + kAdders + 128;  // the last warpgroup has one warp at work: issuer or messenger
constexpr int kPlane = kRows * kKc * 2;        // 8192 bytes: one term of one operand's chunk
constexpr int kStageBytes = 6 * kPlane;
constexpr int kOffBar = kStages * kStageBytes;
constexpr int kSmemBytes = kOffBar + 256 + 1024;
constexpr int kLaunchRegs = 96, kIssuerRegs = 32, kBothRegs = 112;
// A single CTA's converters have a second chunk on its way (a pair's wait for stages instead).
template <int kCtas>
struct RegisterSplit {
  static constexpr int kConverter = kCtas == 2 ? 72 : 104, kAdder = kCtas == 2 ? 152 : 120;
  static_assert(kConverters * kConverter + kAdders * kAdder + 128 * kIssuerRegs <= kThreads * kLaunchRegs, "register split");
};
static_assert((kConverters + kAdders) * kBothRegs + 128 * kIssuerRegs <= kThreads * kLaunchRegs, "register split, one kind of warp");
static_assert(kSmemBytes <= 232448, "shared memory budget");
static_assert(kThreads * kLaunchRegs <= 65536, "registers at launch");
enum { BAR_FULL = 0, BAR_EMPTY = kStages, BAR_D_FULL = 2 * kStages, BAR_D_FREE = BAR_D_FULL + 2,
       BAR_FULL2 = BAR_D_FREE + 2, BAR_D_FREE2 = BAR_FULL2 + kStages, BAR_LAST = BAR_D_FREE2 + 2, BAR_COUNT };  // ..2: the second CTA's word
static_assert(BAR_COUNT <= 24, "barrier block");

// The pair's instructions.  The first CTA issues for both: A and B descriptors address the same offsets in both CTAs (128
// rows of A and half of B's columns each), and each CTA's tensor memory gets its 128 rows of D.
__device__ __forceinline__ void mma2_ss(uint32_t d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(d), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit2(uint32_t bar) {  // arrives on the barrier at this offset in both CTAs
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(static_cast<uint16_t>(3)) : "memory");
}
// Arrives on the first CTA's barrier at this offset.
__device__ __forceinline__ void mbar_arrive_first(uint32_t bar) {
  asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %0, 0;\nmbarrier.arrive.release.cluster.shared::cluster.b64 _, [a];\n}"
               ::"r"(bar) : "memory");
}

// The same without a release: for an arrival that hands over tensor memory and nothing in memory (tcgen05.wait::ld has completed
// the reads before it is issued).
__device__ __forceinline__ void mbar_arrive_first_relaxed(uint32_t bar) {
  asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %0, 0;\nmbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [a];\n}"
               ::"r"(bar) : "memory");
}

// Bounded wait as mbar_wait; kCluster: the other CTA's threads arrive on the barrier too.
template <bool kCluster>
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
  if (!kCluster) return mbar_try_wait(bar, parity);
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
template <bool kCluster, long long kLimit>  // a limit of 0: whatever is not there at the first look
__device__ __forceinline__ void wait_for(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (!kCluster && mbar_test(bar, parity)) return;
  if (*abort_flag) return;
  if (kLimit == 0) { *abort_flag = 1; return; }
  if (try_wait<kCluster>(bar, parity)) return;
  const long long t0 = clock64();
  while (!try_wait<kCluster>(bar, parity)) {
    if (*abort_flag || clock64() - t0 > kLimit) { *abort_flag = 1; return; }
  }
}

__device__ __forceinline__ float2 add2(float2 s, uint32_t x, uint32_t y) {
  asm("{\n.reg .b64 a, b;\nmov.b64 a, {%0, %1};\nmov.b64 b, {%2, %3};\nadd.rn.f32x2 a, a, b;\nmov.b64 {%0, %1}, a;\n}"
      : "+f"(s.x), "+f"(s.y) : "r"(x), "r"(y));
  return s;
}

struct GemmArgs {
  const float* A;
  const float* B;
  float* C;
  long long stride_a, stride_b, stride_c;
  int M, N, K, lda, ldb, ldc, tiles_n, symmetric;
  float alpha;
  int32_t* dev_status;    // may be null
};

// Eight consecutive values along the operand's contiguous dimension, zeros beyond its edges.  Group g of a chunk: with K
// contiguous four groups make a row's 32 k, otherwise eight groups make 64 rows of one k.
template <bool kContig>
__device__ __forceinline__ void load_group(float (&x)[8], const float* P, bool vec, int ld, int r0, int R, int k0, int K, int g) {
  int major, minor, major_end, minor_end;
  if (kContig) { major = r0 + (g >> 2); minor = k0 + (g & 3) * 8; major_end = R; minor_end = K; }
  else { major = k0 + ((g >> 3) & 31); minor = r0 + (g >> 8) * 64 + (g & 7) * 8; major_end = K; minor_end = R; }
  const float* src = P + static_cast<size_t>(major) * ld + minor;
  if (vec && major < major_end && minor + 7 < minor_end) {
    const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = major < major_end && minor + i < minor_end ? src[i] : 0.f;
  }
}
// Splits a group and writes its terms to the three planes at `dst`, `plane` bytes apart.
template <bool kContig>
__device__ __forceinline__ void store_group(const float (&x)[8], unsigned char* dst, int plane, int g) {
  uint32_t t[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a = x[2 * i], b = x[2 * i + 1];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const uint32_t v = pack_bf16(a, b);
      t[p][i] = v;
      a -= bf16_lo(v);  // exact
      b -= bf16_hi(v);
    }
  }
  int off;
  if (kContig) { const int r = g >> 2; off = r * 64 + (((g & 3) ^ ((r >> 1) & 3)) << 4); }
  else { const int k = (g >> 3) & 31; off = (g >> 8) * 4096 + k * 128 + (((g & 7) ^ (k & 7)) << 4); }
#pragma unroll
  for (int p = 0; p < 3; ++p)
    *reinterpret_cast<uint4*>(dst + p * plane + off) = make_uint4(t[p][0], t[p][1], t[p][2], t[p][3]);
}
template <bool kContig>
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr) {
  if (!kContig) return smem_desc(addr, 4096, 1024);
  return (smem_desc(addr, 16, 512) & ~(7ull << 61)) | (4ull << 61);  // 64-byte swizzle
}

// One element of op(A) op(B) as a chain of fp32 multiply-adds.
template <bool kAContig, bool kBContig>
__device__ __forceinline__ float plain_sum(const GemmArgs& args, int m, int n) {
  const float* a = args.A + args.stride_a * blockIdx.y + (kAContig ? static_cast<size_t>(m) * args.lda : m);
  const float* b = args.B + args.stride_b * blockIdx.y + (kBContig ? static_cast<size_t>(n) * args.ldb : n);
  float s = 0.f;
#pragma unroll 1
  for (int k = 0; k < args.K; ++k)
    s = fmaf(a[kAContig ? k : static_cast<size_t>(k) * args.lda], b[kBContig ? k : static_cast<size_t>(k) * args.ldb], s);
  return s;
}

template <int kCtas, bool kAContig, bool kBContig, long long kLimit>
__global__ void __launch_bounds__(kThreads, 1) gemm_split_kernel(const __grid_constant__ GemmArgs args) {
  extern __shared__ unsigned char smem_unaligned[];
  constexpr int kTile = kRows * kCtas;   // tile of C, both ways
  constexpr bool kOneKind = kCtas == 1 && !kAContig;  // of warps: all sixteen convert and add
  const uint32_t raw = smem_u32(smem_unaligned);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_unaligned + (base - raw);
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(sm + kOffBar + 192);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_base_s + 1);
  auto bar = [&](int i) -> uint32_t { return base + kOffBar + 8 * i; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x % kCtas, tile = blockIdx.x / kCtas;
  int tm, tn;
  if (args.symmetric) {  // tiles on and below the diagonal, row by row
    tm = 0; tn = tile;
    while (tn > tm) tn -= ++tm;
  } else {
    tm = tile / args.tiles_n; tn = tile % args.tiles_n;
  }
  const int m0 = tm * kTile + rank * kRows;           // this CTA's rows of op(A) and of C
  const int n0 = tn * kTile;                          // the tile's columns of C
  const float* A = args.A + args.stride_a * blockIdx.y;
  const float* B = args.B + args.stride_b * blockIdx.y;
  const int M = args.M, N = args.N, K = args.K;
  const int chunks = (K + kKc - 1) / kKc;
  auto sync_ctas = [] {
    if (kCtas == 2) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
  };

  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(bar(BAR_FULL + i), 8); mbar_init(bar(BAR_EMPTY + i), 1); mbar_init(bar(BAR_FULL2 + i), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar(BAR_D_FULL + i), 1); mbar_init(bar(BAR_D_FREE + i), kOneKind ? 16 : 8); mbar_init(bar(BAR_D_FREE2 + i), 8); }
    mbar_init(bar(BAR_LAST), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    if (kCtas == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(2u * kTile) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)), "r"(2u * kTile) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  sync_ctas();
  tc_fence_after();
  const uint32_t tmem = *tmem_base_s;
  auto wait = [&](uint32_t b, uint32_t parity) { wait_for<false, kLimit>(b, parity, abort_flag); };
  auto wait_cluster = [&](uint32_t b, uint32_t parity) { wait_for<true, kLimit>(b, parity, abort_flag); };

  if (warp >= (kConverters + kAdders) / 32) {
    // ========================================================================== MMA issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssuerRegs));
    if (warp == (kConverters + kAdders) / 32 && rank == 0) {
      constexpr uint32_t idesc = instr_desc(kTile, !kAContig, kTile) | (kBContig ? 0u : 1u << 16);
      for (int c = 0; c < chunks; ++c) {
        const int stage = c % kStages, buf = c & 1;
        if (c >= 2) {
          wait(bar(BAR_D_FREE + buf), ((c >> 1) - 1) & 1);
          if (kCtas == 2) wait_cluster(bar(BAR_D_FREE2 + buf), ((c >> 1) - 1) & 1);
        }
        wait(bar(BAR_FULL + stage), (c / kStages) & 1);
        if (kCtas == 2) wait_cluster(bar(BAR_FULL2 + stage), (c / kStages) & 1);
        if (__any_sync(0xffffffffu, *abort_flag != 0)) break;  // no further products: those who wait for them give up too
        tc_fence_after();
        const uint64_t a0 = operand_desc<kAContig>(base + stage * kStageBytes);
        const uint64_t b0 = operand_desc<kBContig>(base + stage * kStageBytes + 3 * kPlane);
        if (elect_one()) {
          constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};  // small terms first
#pragma unroll
          for (int p = 0; p < 6; ++p) {
#pragma unroll
            for (int ks = 0; ks < kKc / 16; ++ks) {
              const uint64_t ad = desc_advance(a0, pa[p] * kPlane + ks * (kAContig ? 32 : 2048));
              const uint64_t bd = desc_advance(b0, pb[p] * kPlane + ks * (kBContig ? 32 : 2048));
              if (kCtas == 2) mma2_ss(tmem + buf * kTile, ad, bd, idesc, (p | ks) != 0);
              else mma_ss(tmem + buf * kTile, ad, bd, idesc, (p | ks) != 0);
            }
          }
          if (kCtas == 2) { tc_commit2(bar(BAR_EMPTY + stage)); tc_commit2(bar(BAR_D_FULL + buf)); }
          else { tc_commit(bar(BAR_EMPTY + stage)); tc_commit(bar(BAR_D_FULL + buf)); }
        }
        __syncwarp();
      }
      // Every product has retired before the CTA goes on to its end, also where a wait gave up.
      if (elect_one()) { if (kCtas == 2) tc_commit2(bar(BAR_LAST)); else tc_commit(bar(BAR_LAST)); }
      __syncwarp();
      for (const long long t0 = clock64(); !mbar_try_wait(bar(BAR_LAST), 0) && clock64() - t0 < kWaitCycles;) {}
    } else if (warp == (kConverters + kAdders) / 32) {
      // The second CTA's messenger tells the issuer of written stages: an arrival that releases to the other CTA waits for
      // everything its thread has in flight, which the workers must not.
      for (int c = 0; c < chunks; ++c) {
        wait(bar(BAR_FULL + c % kStages), (c / kStages) & 1);
        if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
        if (elect_one()) mbar_arrive_first(bar(BAR_FULL2 + c % kStages));
        __syncwarp();
      }
    }
  } else {
    // ========================================================================== converting and adding
    const bool vec_a = (args.lda & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
    const bool vec_b = (args.ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
    const int nb0 = n0 + rank * kRows;                  // this CTA's columns of op(B)
    const int ctid = tid & 255;                         // thread of its group of converting warps: two pieces of A and two of B a chunk
    constexpr int kAhead = kCtas == 2 || kOneKind ? 1 : 2;  // chunks on their way, of a group
    float xa[kAhead][2][8], xb[kAhead][2][8];
    // Away from the edges a thread's pieces sit at fixed distances from one address per operand.
    const bool inside = vec_a && vec_b && m0 + kRows <= M && nb0 + kRows <= N;
    const float* next_a = A + (kAContig ? static_cast<size_t>(m0 + (ctid >> 2)) * args.lda + (ctid & 3) * 8
                                        : static_cast<size_t>(ctid >> 3) * args.lda + m0 + (ctid & 7) * 8);
    const float* next_b = B + (kBContig ? static_cast<size_t>(nb0 + (ctid >> 2)) * args.ldb + (ctid & 3) * 8
                                        : static_cast<size_t>(ctid >> 3) * args.ldb + nb0 + (ctid & 7) * 8);
    auto load8 = [](float (&x)[8], const float* src) {
      const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
      x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    };
    auto load = [&](int c, int s = 0) {
      if (inside && (c + 1) * kKc <= K) {
        const float* a = next_a + (kAContig ? static_cast<size_t>(c) * kKc : static_cast<size_t>(c) * kKc * args.lda);
        const float* b = next_b + (kBContig ? static_cast<size_t>(c) * kKc : static_cast<size_t>(c) * kKc * args.ldb);
        load8(xa[s][0], a);
        load8(xa[s][1], a + (kAContig ? static_cast<size_t>(64) * args.lda : 64));
        load8(xb[s][0], b);
        load8(xb[s][1], b + (kBContig ? static_cast<size_t>(64) * args.ldb : 64));
        return;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        load_group<kAContig>(xa[s][u], A, vec_a, args.lda, m0, M, c * kKc, K, ctid + u * 256);
        load_group<kBContig>(xb[s][u], B, vec_b, args.ldb, nb0, N, c * kKc, K, ctid + u * 256);
      }
    };
    auto convert = [&](int c, int s = 0) {
      const int stage = c % kStages;
      if (c >= kStages) wait(bar(BAR_EMPTY + stage), (c / kStages - 1) & 1);
      unsigned char* st = sm + stage * kStageBytes;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        store_group<kAContig>(xa[s][u], st, kPlane, ctid + u * 256);
        store_group<kBContig>(xb[s][u], st + 3 * kPlane, kPlane, ctid + u * 256);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_FULL + stage));
    };
    // Columns of the tile a thread sums: those of its warp's half (of eight warps) or quarter (of sixteen).
    constexpr int kCols = kTile / (kOneKind ? 4 : 2);
    const int index = kOneKind ? warp : warp - kConverters / 32, quad = warp & 3, part = index >> 2;
    const uint32_t d_addr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + part * kCols;
    auto drain = [&](int d, float (&acc)[kCols]) {
      const int buf = d & 1;
      wait(bar(BAR_D_FULL + buf), (d >> 1) & 1);
      tc_fence_after();
#pragma unroll
      for (int j0 = 0; j0 < kCols; j0 += 16) {
        uint32_t v[16];
        tmem_ld16(d_addr + buf * kTile + j0, v);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          if constexpr (kOneKind) {  // (two at a time there: 2 to 6 % slower)
            acc[j0 + j] += __uint_as_float(v[j]);
            acc[j0 + j + 1] += __uint_as_float(v[j + 1]);
          } else {
            const float2 sum = add2(make_float2(acc[j0 + j], acc[j0 + j + 1]), v[j], v[j + 1]);
            acc[j0 + j] = sum.x;
            acc[j0 + j + 1] = sum.y;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) { if (rank == 0) mbar_arrive(bar(BAR_D_FREE + buf)); else mbar_arrive_first_relaxed(bar(BAR_D_FREE2 + buf)); }
    };
    auto write_out = [&](float (&acc)[kCols]) {
      // (After a give-up other warps may still be writing terms over these sums' staging place: NaN goes straight to C.)
      const bool bad = __any_sync(0xffffffffu, *abort_flag != 0);
      // ---- write-out through shared memory (every product has completed), in whole lines
      constexpr int kPitch = kCols + 4;
      float* mine = reinterpret_cast<float*>(sm) + index * 32 * kPitch;
#pragma unroll
      for (int j = 0; j < kCols; j += 4)
        *reinterpret_cast<float4*>(mine + lane * kPitch + j) =
            make_float4(acc[j] * args.alpha, acc[j + 1] * args.alpha, acc[j + 2] * args.alpha, acc[j + 3] * args.alpha);
      // Where the split does not hold the sum is taken once more, by fp32 multiply-adds: an infinite or too large operand value
      // has no exact terms and made its sums NaN, and operands so small that all sums of a region (32 rows x a quarter of the
      // tile's columns) stay below 2^-63 may have lost their last terms.
      constexpr int kRegion = kTile / 4;
      constexpr int kRegions = kCols / kRegion;
      float size[kRegions][4 / kRegions] = {}, all = 0.f;
#pragma unroll
      for (int j = 0; j < kCols; ++j) size[j / kRegion][j % (4 / kRegions)] += fabsf(acc[j]);
      uint32_t small = 0;                               // bits of the warp's regions
#pragma unroll
      for (int g = 0; g < kRegions; ++g) {
        float region = 0.f;
#pragma unroll
        for (int i = 0; i < 4 / kRegions; ++i) region += size[g][i];
        if (__all_sync(0xffffffffu, region < 0x1p-63f) && __any_sync(0xffffffffu, region > 0.f)) small |= 1u << g;
        all += region;
      }
      if (small != 0 || __any_sync(0xffffffffu, !(all < INFINITY))) {
#pragma unroll 1
        for (int j = 0; j < kCols; ++j) {
          const int m = m0 + quad * 32 + lane, n = n0 + part * kCols + j;
          if (m < M && n < N && ((small >> (j / kRegion) & 1u) || !isfinite(mine[lane * kPitch + j])))
            mine[lane * kPitch + j] = args.alpha * plain_sum<kAContig, kBContig>(args, m, n);
        }
      }
      __syncwarp();
      float* C = args.C + args.stride_c * blockIdx.y;
      const int mw = m0 + quad * 32, nw = n0 + part * kCols;
      const bool whole = !bad && !args.symmetric && n0 + kTile <= N && (args.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
      if (whole) {  // 16 bytes a lane
        constexpr int kLanes = kCols / 4, kAtOnce = 32 / kLanes;   // of a row; rows
        const int j = lane % kLanes * 4;
#pragma unroll 4
        for (int r = lane / kLanes; r < 32; r += kAtOnce)
          if (mw + r < M) *reinterpret_cast<float4*>(C + static_cast<size_t>(mw + r) * args.ldc + nw + j) = *reinterpret_cast<const float4*>(mine + r * kPitch + j);
      }
      for (int r = 0; r < 32 && !whole; ++r) {
        const int m = mw + r;
        if (m >= M) break;
#pragma unroll
        for (int j = lane; j < kCols; j += 32) {
          const int n = nw + j;
          if (n < N && (!args.symmetric || n <= m)) C[static_cast<size_t>(m) * args.ldc + n] = bad ? __int_as_float(0x7fffffff) : mine[r * kPitch + j];
        }
      }
      if (args.symmetric) {
        const int m = mw + lane;
        for (int j = 0; j < kCols; ++j) {
          const int n = nw + j;
          if (n < m && m < M) C[static_cast<size_t>(n) * args.ldc + m] = bad ? __int_as_float(0x7fffffff) : mine[lane * kPitch + j];
        }
      }
    };
    if constexpr (kOneKind) {
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kBothRegs));
      float acc[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[j] = 0.f;
      const int group = warp >> 3;  // two groups of eight warps take the chunks in turn
      int drained = 0;
      if (group < chunks) load(group);
      for (int c = group; c < chunks; c += 2) {
        convert(c);
        if (c + 2 < chunks) load(c + 2);
        while (drained + 2 <= c) drain(drained++, acc);
      }
      while (drained < chunks) drain(drained++, acc);
      write_out(acc);
    } else if (warp < kConverters / 32) {
      constexpr int kRegs = RegisterSplit<kCtas>::kConverter;
      if constexpr (kRegs < kLaunchRegs) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs));
      else asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs));
#pragma unroll
      for (int s = 0; s < kAhead; ++s)
        if (s < chunks) load(s, s);
      for (int c0 = 0; c0 < chunks; c0 += kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
          const int c = c0 + s;
          if (c >= chunks) break;
          convert(c, s);
          if (c + kAhead < chunks) load(c + kAhead, s);
        }
      }
    } else {
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(RegisterSplit<kCtas>::kAdder));
      float acc[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[j] = 0.f;
      for (int d = 0; d < chunks; ++d) drain(d, acc);
      write_out(acc);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag) set_status(args.dev_status, TRANSMLA_DEV_TIMEOUT);
  sync_ctas();  // neither CTA leaves while the other may still reach its barriers
  tc_fence_after();
  if (warp == 0) {
    if (kCtas == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * kTile) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * kTile) : "memory");
  }
}

template <int kCtas, bool kAContig, bool kBContig, long long kLimit = kWaitCycles>
cudaError_t launch(GemmArgs args, int batch, cudaStream_t stream) {
  static PerDeviceFlag smem_set;
  auto kernel = gemm_split_kernel<kCtas, kAContig, kBContig, kLimit>;
  if (cudaError_t e = ensure_dynamic_smem(kernel, kSmemBytes, smem_set); e != cudaSuccess) return e;
  constexpr int kTile = kRows * kCtas;
  const long long tiles_m = (args.M + kTile - 1) / kTile;
  args.tiles_n = (args.N + kTile - 1) / kTile;
  const long long tiles = args.symmetric ? tiles_m * (tiles_m + 1) / 2 : tiles_m * args.tiles_n;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles * kCtas), batch);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCtas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = kCtas == 2 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args);
}
// Short sums, K <= 16: plain fp32 multiply-adds, 128 x 128 of C a block, 8 x 8 a thread.  Half a chunk would be empty in the
// kernel above, whose truncation shows where few products leave nothing to average: error of a product 2.5e-8 here, 4.5e-8
// there (K = 16: 7.4e-8 and 4.8e-8).  Bound by the stores of C.  4096 x 4096 x 16: 23.8 against 38.4 us; 8192 x 8192 x 16: 88.6 against
// 131; at K = 24 the split kernel is the faster one (40 against 45 us at 4096 x 4096).
constexpr int kShortK = 16, kShortTile = 128, kShortPitch = kShortTile + 4;
template <bool kAContig, bool kBContig>
__global__ void __launch_bounds__(256) gemm_short_kernel(const __grid_constant__ GemmArgs args) {
  __shared__ __align__(16) float a_s[kShortK][kShortPitch], b_s[kShortK][kShortPitch];
  const int m0 = blockIdx.x / args.tiles_n * kShortTile, n0 = blockIdx.x % args.tiles_n * kShortTile;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, K = args.K;
  const float* A = args.A + args.stride_a * blockIdx.y;
  const float* B = args.B + args.stride_b * blockIdx.y;
  float* C = args.C + args.stride_c * blockIdx.y;
#pragma unroll
  for (int e = tid; e < kShortK * kShortTile; e += 256) {  // consecutive threads read consecutive addresses
    const int ka = kAContig ? e % kShortK : e / kShortTile, ra = kAContig ? e / kShortK : e % kShortTile;
    const int kb = kBContig ? e % kShortK : e / kShortTile, rb = kBContig ? e / kShortK : e % kShortTile;
    const bool in_a = ka < K && m0 + ra < args.M, in_b = kb < K && n0 + rb < args.N;
    a_s[ka][ra] = in_a ? A[kAContig ? static_cast<size_t>(m0 + ra) * args.lda + ka : static_cast<size_t>(ka) * args.lda + m0 + ra] : 0.f;
    b_s[kb][rb] = in_b ? B[kBContig ? static_cast<size_t>(n0 + rb) * args.ldb + kb : static_cast<size_t>(kb) * args.ldb + n0 + rb] : 0.f;
  }
  __syncthreads();
  float acc[8][8] = {};
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(&a_s[k][ty * 4]), a1 = *reinterpret_cast<const float4*>(&a_s[k][64 + ty * 4]);
    const float4 b0 = *reinterpret_cast<const float4*>(&b_s[k][tx * 4]), b1 = *reinterpret_cast<const float4*>(&b_s[k][64 + tx * 4]);
    const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
  }
  const bool vec = (args.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + ty * 4 + (i & 3) + (i >> 2) * 64;
    if (m >= args.M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n = n0 + tx * 4 + h * 64;
      float* dst = C + static_cast<size_t>(m) * args.ldc + n;
      const float4 v = make_float4(acc[i][4 * h] * args.alpha, acc[i][4 * h + 1] * args.alpha, acc[i][4 * h + 2] * args.alpha, acc[i][4 * h + 3] * args.alpha);
      if (vec && n + 3 < args.N) { *reinterpret_cast<float4*>(dst) = v; continue; }
      if (n < args.N) dst[0] = v.x;
      if (n + 1 < args.N) dst[1] = v.y;
      if (n + 2 < args.N) dst[2] = v.z;
      if (n + 3 < args.N) dst[3] = v.w;
    }
  }
}

template <bool kAContig, bool kBContig>
cudaError_t launch_size(GemmArgs args, int batch, cudaStream_t stream) {
  if (args.K <= kShortK) {
    args.tiles_n = (args.N + kShortTile - 1) / kShortTile;
    const long long tiles = static_cast<long long>((args.M + kShortTile - 1) / kShortTile) * args.tiles_n;
    gemm_short_kernel<kAContig, kBContig><<<dim3(static_cast<unsigned>(tiles), batch), 256, 0, stream>>>(args);
    return cudaGetLastError();
  }
  // A pair does four times the work of a single CTA with two CTAs; the single one pays where it fills the device better.  Single
  // CTAs / pairs, K = 2048, orders tb, ta, none: 2 waves of either (2700 x 1600) 132 / 148, 139 / 153, 138 / 152 us; 5 waves against 4 (30000
  // x 301) 328 / 348, 369 / 358, 393 / 361; 4 against 3 (13000 x 520) 253 / 248, 261 / 243, 266 / 236; 3 against 2 (3100 x 1600) 181 / 152, 195 / 154,
  // 185 / 154; 2 against 1 (2048 x 2048, K = 4096) 235 / 158.  So the line lies between 1 and 1.25.
  constexpr long long kSms = 148;
  auto waves = [&](int tile, long long at_once) {
    const long long tm = (args.M + tile - 1) / tile, tn = (args.N + tile - 1) / tile;
    return ((args.symmetric ? tm * (tm + 1) / 2 : tm * tn) * batch + at_once - 1) / at_once;
  };
  if (waves(kRows, kSms) * 7 < waves(2 * kRows, kSms / 2) * 8) return launch<1, kAContig, kBContig>(args, batch, stream);
  return launch<2, kAContig, kBContig>(args, batch, stream);
}

}  // namespace

cudaError_t gemm_f32(int ta, int tb, int M, int N, int K, float alpha, const float* A, int lda, long long strideA,
                     const float* B, int ldb, long long strideB, float* C, int ldc, long long strideC, int batch,
                     int32_t* dev_status, cudaStream_t stream) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  // X^T X (or X X^T) is symmetric: the tiles above the diagonal are mirrored instead of computed
  const int symmetric = A == B && ta != tb && M == N && lda == ldb && strideA == strideB;
  const GemmArgs args = {A, B, C, strideA, strideB, strideC, M, N, K, lda, ldb, ldc, 0, symmetric, alpha, dev_status};
  if (!ta) return tb ? launch_size<true, true>(args, batch, stream) : launch_size<true, false>(args, batch, stream);
  return tb ? launch_size<false, true>(args, batch, stream) : launch_size<false, false>(args, batch, stream);
}

cudaError_t gemm_f32_gives_up(int pairs, int M, int N, int K, const float* A, const float* B, float* C, int32_t* dev_status,
                              cudaStream_t stream) {
  const GemmArgs args = {A, B, C, 0, 0, 0, M, N, K, K, N, N, 0, 0, 1.f, dev_status};
  return pairs ? launch<2, true, false, 0>(args, 1, stream) : launch<1, true, false, 0>(args, 1, stream);
}

}  // namespace conv
}  // namespace transmla

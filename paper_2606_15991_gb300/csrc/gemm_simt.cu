// FP32 GEMM on the CUDA cores (FFMA, FP32 accumulation, no TF32): one 64x64
// C tile per tile program with a K loop (§3.6, Listing 6). Plain partitions
// launch one program per tile; mapped partitions launch persistent programs
// that walk their tiles (strided slots or a device queue), slots being turned
// into tiles by the band raster shared with the tensor-core GEMM.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "sm100_ptx.cuh"
#include "tp_internal.h"

namespace tp {
namespace {

constexpr int BM = 64, BN = 64;

constexpr int TM = 8, TN = 4;                   // elements per thread
constexpr int TX = BN / TN, TY = BM / TM;       // threads along the columns and the rows
constexpr int TH = TX * TY;                     // 128
constexpr int KC = 32;                          // K elements per ring stage
constexpr int kStages = 3;
constexpr int kPitchA = KC + 4, kPitchB = BN + 4;  // floats per row of a stage's A (64 x KC) and B (KC x 64)
constexpr int kStageA = BM * kPitchA;           // floats
constexpr int kStage = kStageA + KC * kPitchB;
constexpr size_t kSmem = (size_t)kStages * kStage * sizeof(float);
constexpr int kCtas = 4;                        // CTAs that share an SM (128 registers a thread, 53 KB each)
static_assert(kSmem >= BM * BN * sizeof(float), "a split program's partial block overlays the ring");

struct SimtArgs {
  const float* a;
  const float* b;
  float* c;
  int64_t M, N, K;
  int64_t sam, sak, sbk, sbn;  // element strides of A (m, k) and B (k, n)
  int64_t gm, gn;              // tile grid
  int32_t kind, group_m;
  int32_t split;               // K slices per tile (cluster size); 1 = none
  int32_t bk;                  // K granularity of the slices (cfg.bk)
  unsigned* queue;
  uint32_t* counts;
  int32_t* owner;
};

// Schedule slot -> (tm, tn): bands of group_m tile rows, column by column
// inside a band (group_m = 1 is row-major).
__device__ __forceinline__ void raster(int64_t s, int64_t gm, int64_t gn, int64_t g, int64_t* tm,
                                       int64_t* tn) {
  const int64_t per = g * gn;
  const int64_t first = (s / per) * g;
  const int64_t rows = min(g, gm - first);
  const int64_t r = s % per;
  *tm = first + r % rows;
  *tn = r / rows;
}

// Asynchronous copy of `bytes` (0..kBytes) from global to shared memory, the
// rest of the kBytes zero-filled.
template <int kBytes>
__device__ __forceinline__ void copy_async(uint32_t dst, const float* src, int bytes) {
  if constexpr (kBytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Two FP32 fused multiply-adds, each rounded as fmaf rounds.
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}

// How a block of an operand reaches shared memory.
enum Fetch : int {
  kRows16,  // 16-byte copies: contiguous block rows on 16-byte boundaries
  kRows4,   // 4-byte copies, a warp along a block row
  kCols4,   // 4-byte copies, a warp on 8 block rows x 4 columns: contiguous block columns
};

// Copies the valid part (nrows x ncols) of a kR x kC block at `src` (element
// strides srow, scol) to `dst` (kPitch floats per row) and zero-fills the
// rest. A warp's copies write distinct banks in every form (kPitch mod 32 = 4).
template <int kFetch, int kR, int kC, int kPitch>
__device__ __forceinline__ void fetch_block(uint32_t dst, const float* src, int64_t srow, int64_t scol, int nrows, int ncols) {
  static_assert(kPitch % 32 == 4, "kCols4 writes 8 rows x 4 columns at once");
  const int tid = threadIdx.x;
  // opaque to the compiler, which would otherwise keep every copy's offset in
  // registers across the K loop and spill the accumulators
  asm volatile("" : "+l"(srow), "+l"(scol), "+r"(nrows));
  if constexpr (kFetch == kRows16) {
    constexpr int kQ = kC / 4;  // 16-byte pieces per row
    const int c = tid % kQ * 4, r0 = tid / kQ;
    const int valid = max(0, min(4, ncols - c)) * 4;
    const float* at = src + r0 * srow + c;
#pragma unroll
    for (int e = 0; e < kR * kQ / TH; ++e) {
      const int row = r0 + e * (TH / kQ);
      const int bytes = row < nrows ? valid : 0;
      copy_async<16>(dst + (uint32_t)(row * kPitch + c) * 4, bytes ? at : src, bytes);
      at += (TH / kQ) * srow;
    }
  } else if constexpr (kFetch == kRows4) {
    const int c = tid % kC, r0 = tid / kC;
    const float* at = src + r0 * srow + c * scol;
#pragma unroll
    for (int e = 0; e < kR * kC / TH; ++e) {
      const int row = r0 + e * (TH / kC);
      const int bytes = row < nrows && c < ncols ? 4 : 0;
      copy_async<4>(dst + (uint32_t)(row * kPitch + c) * 4, bytes ? at : src, bytes);
      at += (TH / kC) * srow;
    }
  } else {
    // warp w takes the 8 x 4 blocks w, w + 4, ... of the block, down the rows first
    constexpr int kRB = kR / 8;
#pragma unroll
    for (int e = 0; e < kR * kC / TH; ++e) {
      const int blk = e * (TH / 32) + tid / 32;
      const int row = blk % kRB * 8 + (tid & 7), c = blk / kRB * 4 + (tid >> 3 & 3);
      const int bytes = row < nrows && c < ncols ? 4 : 0;
      copy_async<4>(dst + (uint32_t)(row * kPitch + c) * 4, bytes ? src + row * srow + c * scol : src, bytes);
    }
  }
}

// FP32 GEMM fed by asynchronous copies. Each of the 128 threads owns an 8 x 4
// block of the tile and multiplies with the two-wide FMA, whose pairs are
// neighbouring columns (one B load) times a duplicated A element: a single
// FFMA stream peaks at 57-69 TFLOP/s on this chip for its register reads, the
// two-wide form at 70-76. K arrives in chunks of 32 through a ring of three
// stages, one block barrier per chunk; four CTAs share an SM, so their
// barriers, shared-memory loads and tails overlap. A's rows stay as stored
// (padded to 36 floats: the four rows a warp reads at once lie in different
// banks), so a thread's four k of a row are one 16-byte load.
// Bound by the FMA pipe (69 % busy at 2048^3, ncu) and the issue of what feeds
// it: 49 TFLOP/s at 2048^3 aligned, 47 unaligned (the register-staged kernel
// that this replaces, 256 threads of 4 x 4 at one CTA per SM: 41 fed by TMA,
// 27 unaligned); 1000 x 3001 x 777, nothing aligned, 184 -> 113 us. Blocks of
// 8 x 8 (64 threads) and 4 x 4 (256) ran 2048^3 at 45 and 43 TFLOP/s; pairs
// along K, which need no duplication, leave no registers to load ahead: 35.
// With split = S > 1 a tile program is a cluster of S CTAs: CTA r runs the K
// steps [r*n/S, (r+1)*n/S) of cfg.bk and keeps its partial 64 x 64 block in
// shared memory; after a cluster barrier CTA r adds, for rows
// [r*64/S, (r+1)*64/S), the S partials in slice order 0..S-1 (reading the
// others through distributed shared memory) and stores them, so every element
// still has one writer and C is bit-reproducible.
template <int kFetchA, int kFetchB, bool COUNT>
__global__ void __launch_bounds__(TH, kCtas) gemm_f32_kernel(const __grid_constant__ SimtArgs p) {
  extern __shared__ __align__(16) float smem[];
  __shared__ int64_t slot;
  const uint32_t base = sm100::smem_u32(smem);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  // a warp is 8 threads along the columns x 4 along the rows; a thread's rows
  // are ty + TY i and its columns 4 tx .. 4 tx + 3
  const int tx = warp % (TX / 8) * 8 + (lane & 7), ty = warp / (TX / 8) * 4 + (lane >> 3);
  const int64_t T = p.gm * p.gn;
  const int S = p.split;
  const uint32_t r = S > 1 ? sm100::cluster_ctarank() : 0u;
  // the operands may be the previous kernel's output, and C its input
  sm100::grid_dependency_wait();
  sm100::allow_dependents();
  int64_t s = S > 1 ? (int64_t)(blockIdx.x / S) : (int64_t)blockIdx.x;
  if (p.kind == TP_MAP_QUEUE) {
    if (tid == 0) slot = atomicAdd(p.queue, 1u);
    __syncthreads();
    s = slot;
  }
  // this CTA's K slice, in whole steps of bk
  const int64_t steps = (p.K + p.bk - 1) / p.bk;
  const int64_t kbeg = S > 1 ? (int64_t)r * steps / S * p.bk : 0;
  const int64_t kend = S > 1 ? min(p.K, (int64_t)(r + 1) * steps / S * p.bk) : p.K;
  const int nch = kend > kbeg ? (int)((kend - kbeg + KC - 1) / KC) : 0;
  while (s < T) {
    int64_t tm, tn;
    raster(s, p.gm, p.gn, p.group_m, &tm, &tn);
    const int64_t m0 = tm * BM, n0 = tn * BN;
    const int mrows = (int)min((int64_t)BM, p.M - m0), ncols = (int)min((int64_t)BN, p.N - n0);
    // chunk ch of the slice into its ring stage
    auto load = [&](int ch) {
      const int64_t k0 = kbeg + (int64_t)ch * KC;
      const int klen = (int)min((int64_t)KC, kend - k0);
      const uint32_t sa = base + (uint32_t)((ch % kStages) * kStage * 4);
      fetch_block<kFetchA, BM, KC, kPitchA>(sa, p.a + m0 * p.sam + k0 * p.sak, p.sam, p.sak, mrows, klen);
      fetch_block<kFetchB, KC, BN, kPitchB>(sa + kStageA * 4, p.b + k0 * p.sbk + n0 * p.sbn, p.sbk, p.sbn, klen, ncols);
    };
    uint64_t acc[TM][TN / 2];  // pairs of neighbouring columns
#pragma unroll
    for (int i = 0; i < TM; ++i) acc[i][0] = acc[i][1] = 0;
#pragma unroll
    for (int ch = 0; ch < kStages - 1; ++ch) {
      if (ch < nch) load(ch);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int ch = 0; ch < nch; ++ch) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
      __syncthreads();  // chunk ch has landed for every thread, and chunk ch - 1's stage is free
      if (ch + kStages - 1 < nch) load(ch + kStages - 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
      const float* As = smem + (ch % kStages) * kStage + ty * kPitchA;
      const float* Bs = smem + (ch % kStages) * kStage + kStageA + 4 * tx;
#pragma unroll
      for (int g = 0; g < KC / 4; ++g) {
        float4 av[TM], bv[4];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(As + TY * i * kPitchA + 4 * g);
#pragma unroll
        for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(Bs + (4 * g + j) * kPitchB);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t b01 = pack2(bv[j].x, bv[j].y), b23 = pack2(bv[j].z, bv[j].w);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float a = j == 0 ? av[i].x : j == 1 ? av[i].y : j == 2 ? av[i].z : av[i].w;
            const uint64_t aa = pack2(a, a);
            fma2(acc[i][0], aa, b01);
            fma2(acc[i][1], aa, b23);
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    float4 out[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const float2 lo = unpack2(acc[i][0]), hi = unpack2(acc[i][1]);
      out[i] = make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    __syncthreads();  // the ring is free (the next tile's loads, the partial block below)
    // this thread's row i is stored by this CTA
    auto mine = [&](int i) { return S == 1 || (ty + TY * i) / (BM / S) == (int)r; };
    if (S > 1) {
      // the partial blocks meet through distributed shared memory: CTA r adds
      // rows [r*64/S, +64/S) of the S partials in slice order
      float(*Ps)[BN] = reinterpret_cast<float(*)[BN]>(smem);
#pragma unroll
      for (int i = 0; i < TM; ++i) *reinterpret_cast<float4*>(&Ps[ty + TY * i][4 * tx]) = out[i];
      sm100::cluster_sync();  // every CTA's partial is in its shared memory
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        if (!mine(i)) continue;
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int src = 0; src < S; ++src) {
          float4 v = out[i];
          if (src != (int)r) {
            const uint32_t at = sm100::mapa(sm100::smem_u32(&Ps[ty + TY * i][4 * tx]), (uint32_t)src);
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                         : "r"(at)
                         : "memory");
          }
          sum = src == 0 ? v : make_float4(sum.x + v.x, sum.y + v.y, sum.z + v.z, sum.w + v.w);
        }
        out[i] = sum;
      }
      sm100::cluster_sync();  // the peers' reads of this CTA's partial are done
    }
    const bool vec = (p.N % 4 == 0) && ((reinterpret_cast<uintptr_t>(p.c) & 15) == 0);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if (!mine(i) || ty + TY * i >= mrows) continue;
      const int64_t e = (m0 + ty + TY * i) * p.N + n0 + 4 * tx;
      const float f[4] = {out[i].x, out[i].y, out[i].z, out[i].w};
      if (vec && 4 * tx + 4 <= ncols) {
        *reinterpret_cast<float4*>(p.c + e) = out[i];
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (4 * tx + j < ncols) p.c[e + j] = f[j];
      }
      if constexpr (COUNT) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (4 * tx + j < ncols) {
            atomicAdd(p.counts + e + j, 1u);
            p.owner[e + j] = (int32_t)(blockIdx.x / S);
          }
      }
    }
    if (p.kind == TP_MAP_IDENTITY) break;
    if (p.kind == TP_MAP_STRIDED) {
      s += gridDim.x / S;
    } else {
      __syncthreads();
      if (tid == 0) slot = atomicAdd(p.queue, 1u);
      __syncthreads();
      s = slot;
    }
  }
}

template <int kFetchA, int kFetchB, bool COUNT>
cudaError_t launch_inst(const SimtArgs& p, int64_t programs, cudaStream_t st) {
  auto k = gemm_f32_kernel<kFetchA, kFetchB, COUNT>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(programs * p.split));
  cfg.blockDim = dim3(TH);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k, p);
}

// The fetch of an operand whose block rows have element stride `row` and
// whose block columns have stride `col`.
int fetch_of(const float* ptr, int64_t row, int64_t col) {
  if (col == 1 && row % 4 == 0 && (reinterpret_cast<uintptr_t>(ptr) & 15) == 0) return kRows16;
  return row == 1 && col != 1 ? kCols4 : kRows4;
}

template <int kFetchA>
cudaError_t launch_b(const SimtArgs& p, int fetch_b, int64_t programs, cudaStream_t st) {
  switch (fetch_b) {
    case kRows16: return launch_inst<kFetchA, kRows16, false>(p, programs, st);
    case kRows4: return launch_inst<kFetchA, kRows4, false>(p, programs, st);
    default: return launch_inst<kFetchA, kCols4, false>(p, programs, st);
  }
}

cudaError_t launch_async(const SimtArgs& p, int64_t programs, cudaStream_t st) {
  // instrumented launches: one form for every layout
  if (p.counts) return launch_inst<kRows4, kRows4, true>(p, programs, st);
  const int fb = fetch_of(p.b, p.sbk, p.sbn);
  switch (fetch_of(p.a, p.sam, p.sak)) {
    case kRows16: return launch_b<kRows16>(p, fb, programs, st);
    case kRows4: return launch_b<kRows4>(p, fb, programs, st);
    default: return launch_b<kCols4>(p, fb, programs, st);
  }
}

// ------------------------------------------------ TMA-fed FP32 GEMM
// The same tiles, K order and split-K reduction as gemm_f32_kernel (so the
// same C bit for bit) for launches that leave an SM one CTA at most: a
// producer thread copies each 32-wide K chunk of the tile's A rows (64 x 32
// floats, 128-byte rows, 128-byte swizzle) and B columns (32 x 64 floats,
// 256-byte rows) into a ring of 16 KB stages while eight compute warps (4 x 4
// elements per thread) multiply the chunks already landed, with no block
// barrier per K step. Alone on its SM the eight warps hide each other's
// latencies better than gemm_f32_kernel's four: 512^3 split in two (128 CTAs)
// 11.9 us against 15.2, one tile of K = 512 17.5 against 18.4; with two CTAs
// per SM and more the order turns (1024^3, 256 CTAs: 63.3 against 56.9).
// Five stages and 96 registers, so that the next launch's CTAs could move in
// early, were no faster (12.0 us).
constexpr int kFChunk = 32;
constexpr int kFStages = 8;
constexpr uint32_t kFChunkA = BM * kFChunk * 4;  // 8 KB
constexpr uint32_t kFChunkB = kFChunk * BN * 4;  // 8 KB
constexpr uint32_t kFStageBytes = kFChunkA + kFChunkB;
constexpr int kFWarps = 8;                       // compute warps (4 x 4 elements per thread)
constexpr int kFThreads = 32 * kFWarps + 32;     // + the producer warp
constexpr size_t kFSmem = 1024 + (size_t)kFStages * kFStageBytes + BM * BN * 4 + 8 * (2 * kFStages) + 16;

struct F32TmaArgs {
  float* c;
  int64_t M, N, K;
  int64_t gm, gn;
  int32_t kind, group_m, split;
  int32_t nchunks;  // K chunks of 32
  uint32_t* counts;
  int32_t* owner;
  int* err;
  uint64_t wait_ns;
};

template <bool COUNT>
__global__ void __launch_bounds__(kFThreads, 1)
    gemm_f32_tma_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                        const __grid_constant__ F32TmaArgs p) {
  using namespace sm100;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // 128-byte swizzle: 1024-byte aligned stages
  uint8_t* gbase = smem_raw + (base - raw);
  auto Ps = reinterpret_cast<float(*)[BN]>(gbase + (size_t)kFStages * kFStageBytes);
  const uint32_t bars = base + kFStages * kFStageBytes + BM * BN * 4;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (kFStages + s); };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + (bars - base) + 8 * 2 * kFStages);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int S = p.split;
  const uint32_t r = S > 1 ? cluster_ctarank() : 0u;
  if (tid == 0) {
    for (int s = 0; s < kFStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), kFWarps);
    }
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&map_a);
    tma_prefetch_desc(&map_b);
  }
  __syncthreads();
  // A and B may be the previous kernel's output, and C its input
  grid_dependency_wait();
  allow_dependents();
  const int64_t T = p.gm * p.gn;
  const int64_t s0 = (int64_t)(blockIdx.x / S);
  const int64_t step = p.kind == TP_MAP_IDENTITY ? T : (int64_t)(gridDim.x / S);
  const int32_t c0 = (int32_t)(((int64_t)r * p.nchunks) / S), c1 = (int32_t)(((int64_t)(r + 1) * p.nchunks) / S);
  if (warp == kFWarps) {
    // ---------------- producer
    if (lane == 0) {
      uint32_t fills[kFStages] = {};
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int64_t s = s0; s < T && ok; s += step) {
        int64_t tm, tn;
        raster(s, p.gm, p.gn, p.group_m, &tm, &tn);
        for (int32_t ch = c0; ch < c1; ++ch) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.err, p.wait_ns)) { ok = false; break; }
          const uint32_t dst = base + kFStageBytes * (uint32_t)stage;
          mbar_arrive_expect_tx(full_bar(stage), kFStageBytes);
          tma_load_2d(dst, &map_a, ch * kFChunk, (int32_t)(tm * BM), full_bar(stage), policy_evict_last());
          tma_load_2d(dst + kFChunkA, &map_b, (int32_t)(tn * BN), ch * kFChunk, full_bar(stage), policy_evict_last());
          fills[stage]++;
          if (++stage == kFStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok)  // every copy this thread issued lands before the CTA retires
        for (int s2 = 0; s2 < kFStages; ++s2)
          if (fills[s2]) mbar_wait(full_bar(s2), (fills[s2] - 1u) & 1u, nullptr, nullptr, 200000000ull);
    }
    __syncwarp();
    // split programs hold one tile: the producer warp joins the two
    // cluster barriers of the epilogue below
    if (S > 1) {
      cluster_sync();
      cluster_sync();
    }
    return;
  }
  // ---------------- compute warps: thread (tx, ty) owns rows 4ty..4ty+3 and
  // columns 4tx..4tx+3 of the tile
  const int tx = tid % 16, ty = tid / 16;
  int stage = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int64_t s = s0; s < T || (S > 1 && s == s0); s += step) {
    const bool have = s < T;  // a split cluster without a tile still joins the cluster barriers
    int64_t tm = 0, tn = 0;
    if (have) raster(s, p.gm, p.gn, p.group_m, &tm, &tn);
    float acc[4][4] = {};
    for (int32_t ch = c0; have && ok && ch < c1; ++ch) {
      const bool got = mbar_wait(full_bar(stage), phase, abort_flag, p.err, p.wait_ns);
      if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
      const uint32_t sa = base + kFStageBytes * (uint32_t)stage;
      const uint32_t sb = sa + kFChunkA;
#pragma unroll
      for (int g = 0; g < kFChunk / 4; ++g) {
        // A rows 4ty+i, k = 4g..4g+3 (16-byte piece g of a 128-byte row,
        // stored at piece g ^ (row & 7)); B rows k = 4g+j, columns 4tx..
        float av[4][4], bv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t row = (uint32_t)(4 * ty + i);
          uint32_t w[4];
          ld_shared_v4(sa + row * 128u + ((((uint32_t)g) ^ (row & 7u)) << 4), w);
#pragma unroll
          for (int q = 0; q < 4; ++q) av[i][q] = __uint_as_float(w[q]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t w[4];
          ld_shared_v4(sb + (uint32_t)(4 * g + j) * 256u + (uint32_t)tx * 16u, w);
#pragma unroll
          for (int q = 0; q < 4; ++q) bv[j][q] = __uint_as_float(w[q]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][q] = fmaf(av[i][j], bv[j][q], acc[i][q]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty_bar(stage));
      if (++stage == kFStages) { stage = 0; phase ^= 1u; }
    }
    const int64_t m0 = tm * BM, n0 = tn * BN;
    bool mine = have;  // this thread's rows are stored by this CTA
    if (S > 1) {
      // partial blocks in shared memory, summed in slice order by the CTA
      // that owns the rows (peers read through distributed shared memory)
      if (have) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          *reinterpret_cast<float4*>(&Ps[4 * ty + i][4 * tx]) =
              make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      }
      cluster_sync();
      mine = have && (4 * ty) / (BM / S) == (int)r;
      if (mine) {
        float sum[4][4];
        for (int src = 0; src < S; ++src) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float4 v;
            if (src == (int)r) {
              v = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            } else {
              const uint32_t at = mapa(smem_u32(&Ps[4 * ty + i][4 * tx]), (uint32_t)src);
              asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                           : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                           : "r"(at)
                           : "memory");
            }
            const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) sum[i][q] = src == 0 ? vv[q] : sum[i][q] + vv[q];
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[i][q] = sum[i][q];
      }
      cluster_sync();  // the peers' reads of this CTA's partial are done
    }
    if (!ok) mine = false;
    const bool vec = (p.N % 4 == 0) && ((reinterpret_cast<uintptr_t>(p.c) & 15) == 0);
#pragma unroll
    for (int i = 0; i < 4 && mine; ++i) {
      const int64_t row = m0 + 4 * ty + i;
      if (row >= p.M) continue;
      const int64_t col = n0 + 4 * tx;
      if (vec && col + 4 <= p.N) {
        *reinterpret_cast<float4*>(p.c + row * p.N + col) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (col + q < p.N) p.c[row * p.N + col + q] = acc[i][q];
      }
      if constexpr (COUNT) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (col + q < p.N) {
            atomicAdd(p.counts + row * p.N + col + q, 1u);
            p.owner[row * p.N + col + q] = (int32_t)(blockIdx.x / S);
          }
      }
    }
    if (S > 1 || !ok) break;
  }
}

template <bool COUNT>
cudaError_t launch_f32_tma(const CUtensorMap& ma, const CUtensorMap& mb, const F32TmaArgs& p, int64_t programs,
                           cudaStream_t st) {
  auto k = gemm_f32_tma_kernel<COUNT>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFSmem);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(programs * p.split));
  cfg.blockDim = dim3(kFThreads);
  cfg.dynamicSmemBytes = kFSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k, ma, mb, p);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  });
  return fn;
}

// fp32 [rows, cols] row-major (row pitch ld floats) in boxes of box_cols x
// box_rows, zero fill past the edges
bool f32_map(CUtensorMap* map, const float* ptr, int64_t rows, int64_t cols, int64_t ld, int box_cols, int box_rows,
             bool swizzle) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * 4)};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

tp_status launch_gemm_simt(tp_ctx* ctx, tp_partition* c, const tp_tensor* a, const tp_tensor* b,
                           const tp_gemm_config* cfg, const tp_exec* ex, cudaStream_t stream,
                           unsigned* queue, int* err) {
  if (c->tile[0] != BM || c->tile[1] != BN)
    return fail(TP_ERR_UNSUPPORTED, "the FP32 GEMM uses 64 x 64 output tiles");
  if ((ex->write_counts == nullptr) != (ex->write_owner == nullptr))
    return fail(TP_ERR_INVALID, "write_counts and write_owner must be given together");
  SimtArgs p{};
  p.a = static_cast<const float*>(a->ptr);
  p.b = static_cast<const float*>(b->ptr);
  p.c = static_cast<float*>(c->t.ptr);
  p.M = a->shape[0];
  p.K = a->shape[1];
  p.N = b->shape[1];
  p.sam = a->strides[0];
  p.sak = a->strides[1];
  p.sbk = b->strides[0];
  p.sbn = b->strides[1];
  p.gm = c->grid[0];
  p.gn = c->grid[1];
  p.kind = c->kind;
  // a plain partition is program p -> tile p in row-major order (§3.4)
  p.group_m = (c->kind != TP_MAP_IDENTITY && cfg && cfg->group_m > 0) ? cfg->group_m : 1;
  p.queue = queue;
  p.counts = ex->write_counts;
  p.owner = ex->write_owner;
  if (p.M == 0 || p.N == 0) return TP_OK;
  const int64_t grid = c->kind == TP_MAP_IDENTITY ? c->num_tiles : c->num_programs;
  const int bk = (cfg && cfg->bk > 0) ? cfg->bk : 32;
  p.split = (cfg && cfg->split_k > 1) ? cfg->split_k : 1;
  if (cfg && (cfg->split_k < 0 || cfg->split_k > 4 || (p.split & (p.split - 1))))
    return fail(TP_ERR_INVALID, "FP32 GEMM split_k must be 0, 1, 2 or 4");
  if (p.split > 1 && c->kind == TP_MAP_QUEUE)
    return fail(TP_ERR_UNSUPPORTED, "FP32 GEMM split_k with a queue map (each CTA would dequeue its own tile)");
  if (bk != 8 && bk != 16 && bk != 32) return fail(TP_ERR_UNSUPPORTED, "FP32 GEMM bk must be 8, 16 or 32");
  p.bk = bk;
  const bool count = p.counts != nullptr;
  cudaError_t e;
  // TMA-fed kernel: at most one CTA per SM (measured where the kernel is
  // defined), unit-stride rows 16-byte aligned, K chunks of 32 (the bk = 32
  // schedule), identity or strided maps, split programs one tile each
  const int64_t T = p.gm * p.gn;
  const bool tma_ok = bk == 32 && p.sak == 1 && p.sbn == 1 && p.sam % 4 == 0 && p.sbk % 4 == 0 &&
                      ((reinterpret_cast<uintptr_t>(p.a) | reinterpret_cast<uintptr_t>(p.b)) & 15) == 0 &&
                      p.K > 0 && p.K < ((int64_t)1 << 30) && p.M < ((int64_t)1 << 31) && p.N < ((int64_t)1 << 31) &&
                      c->kind != TP_MAP_QUEUE && (p.split == 1 || grid >= T) && grid * p.split <= ctx->sm_count;
  if (tma_ok) {
    CUtensorMap ma, mb;
    if (f32_map(&ma, p.a, p.M, p.K, p.sam, kFChunk, BM, true) && f32_map(&mb, p.b, p.K, p.N, p.sbk, BN, kFChunk, false)) {
      F32TmaArgs t{};
      t.c = p.c;
      t.M = p.M;
      t.N = p.N;
      t.K = p.K;
      t.gm = p.gm;
      t.gn = p.gn;
      t.kind = p.kind;
      t.group_m = p.group_m;
      t.split = p.split;
      t.nchunks = (int32_t)((p.K + kFChunk - 1) / kFChunk);
      t.counts = p.counts;
      t.owner = p.owner;
      t.err = err;
      t.wait_ns = 2000000000ull;
      e = count ? launch_f32_tma<true>(ma, mb, t, grid, stream) : launch_f32_tma<false>(ma, mb, t, grid, stream);
      if (e != cudaSuccess) return cuda_fail(e, "FP32 GEMM launch");
      return TP_OK;
    }
  }
  e = launch_async(p, grid, stream);
  if (e != cudaSuccess) return cuda_fail(e, "FP32 GEMM launch");
  return TP_OK;
}

}  // namespace tp

// The FP32 GEMM's kernel and its launches (see gemm_simt.cu), in a header
// because the instrumented instances are compiled beside the others: an
// instrumented launch runs the form that its operands take without.
#pragma once

#include <algorithm>
#include <type_traits>

#include "sm100_ptx.cuh"
#include "tp_internal.h"

namespace tp {

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

// Launches with write counts (gemm_simt_counted.cu).
cudaError_t launch_f32_counted(const SimtArgs& p, int64_t programs, int sms, cudaStream_t st);

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
constexpr size_t kSmemSm = 227 * 1024;           // shared memory of an SM
constexpr int kCtas = 4;                        // CTAs that share an SM (128 registers a thread, 53 KB each)
static_assert(kSmem >= BM * BN * sizeof(float), "a split program's partial block overlays the ring");

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

// The same shared-memory address in CTA `rank` of the cluster, as a pointer
// that plain loads take.
__device__ __forceinline__ const float* peer_shared(const float* q, uint32_t rank) {
  uint64_t r;
  asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<uint64_t>(q)), "r"(rank));
  return reinterpret_cast<const float*>(r);
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
// stages, one block barrier per chunk; the operands of the next two k are
// loaded from shared memory while the current two are multiplied; up to four
// CTAs share an SM, so their barriers and tails overlap. A's rows stay as
// stored (padded to 36 floats: the four rows a warp reads at once lie in
// different banks).
// Bound by the FMA pipe (busy 69 % of the cycles at 2048^3, ncu) and the issue
// of what feeds it. One product over and over in a replayed graph, its operands
// in L2, against the kernels this replaces (register-staged, 256 threads of
// 4 x 4 at one CTA per SM; TMA-fed with a producer warp for aligned operands):
//   2048^3 aligned 419 -> 343 us, unaligned 628 -> 352
//   1000 x 3001 x 777, nothing aligned, 184 -> 109 us
//   512^3 in two K slices (128 CTAs) 11.9 -> 10.6 us, in four 15.8 -> 10.7
// Blocks of 8 x 8 (64 threads) and 4 x 4 (256) ran 2048^3 at 45 and 43 TFLOP/s
// against 50; pairs along K, which need no duplication, leave no registers to
// load ahead: 35; two or four thread groups sharing a tile's K, for launches of
// one CTA per SM, were no faster there (one tile's k takes 57 cycles in every
// form).
// With split = S > 1 a tile program is a cluster of S CTAs: CTA r runs the K
// steps [r*n/S, (r+1)*n/S) of cfg.bk and keeps its partial 64 x 64 block in
// shared memory; after a cluster barrier CTA r adds, for rows
// [r*64/S, (r+1)*64/S), the S partials in slice order 0..S-1 (reading the
// others through distributed shared memory, all loads before the first sum: one
// after another they cost 3 us) and stores them, so every element still has one
// writer and C is bit-reproducible.
template <int kFetchA, int kFetchB, bool kSplit, bool COUNT>
__global__ void __launch_bounds__(TH, kCtas) gemm_f32_kernel(const __grid_constant__ SimtArgs p) {
  extern __shared__ __align__(16) float smem[];
  __shared__ int64_t slot;
  const uint32_t base = sm100::smem_u32(smem);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  // a warp is 8 threads along the columns x 4 along the rows; a thread's rows
  // are ty + TY i and its columns 4 tx .. 4 tx + 3
  const int tx = warp % (TX / 8) * 8 + (lane & 7), ty = warp / (TX / 8) * 4 + (lane >> 3);
  const int64_t T = p.gm * p.gn;
  const int S = kSplit ? p.split : 1;
  const uint32_t r = kSplit ? sm100::cluster_ctarank() : 0u;
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
    // A fragment is two k of this thread's rows and columns. The next one is
    // loaded while the current one is multiplied, across chunk boundaries too,
    // so shared memory's latency never stands before the FMAs.
    struct Frag {
      float2 a[TM];
      float4 b[2];
    } fr[2];
    auto fetch_frag = [&](Frag& f, int ch, int g) {
      const float* As = smem + (ch % kStages) * kStage + ty * kPitchA + 2 * g;
      const float* Bs = smem + (ch % kStages) * kStage + kStageA + 4 * tx + 2 * g * kPitchB;
#pragma unroll
      for (int i = 0; i < TM; ++i) f.a[i] = *reinterpret_cast<const float2*>(As + TY * i * kPitchA);
#pragma unroll
      for (int j = 0; j < 2; ++j) f.b[j] = *reinterpret_cast<const float4*>(Bs + j * kPitchB);
    };
#pragma unroll
    for (int ch = 0; ch < kStages; ++ch) {
      if (ch < nch) load(ch);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (nch > 0) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
      __syncthreads();
      fetch_frag(fr[0], 0, 0);
    }
    for (int ch = 0; ch < nch; ++ch) {
#pragma unroll
      for (int g = 0; g < KC / 2; ++g) {
        if (g + 1 < KC / 2) {
          fetch_frag(fr[(g + 1) & 1], ch, g + 1);
        } else if (ch + 1 < nch) {
          asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
          // chunk ch + 1 has landed for every thread, and every thread holds
          // its last fragment of chunk ch: that stage is free
          __syncthreads();
          if (ch + kStages < nch) load(ch + kStages);
          asm volatile("cp.async.commit_group;" ::: "memory");
          fetch_frag(fr[0], ch + 1, 0);
        }
        const Frag& f = fr[g & 1];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint64_t b01 = pack2(f.b[j].x, f.b[j].y), b23 = pack2(f.b[j].z, f.b[j].w);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float a = j == 0 ? f.a[i].x : f.a[i].y;
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
    const bool vec = (p.N % 4 == 0) && ((reinterpret_cast<uintptr_t>(p.c) & 15) == 0);
    // four columns of one tile row
    auto store = [&](int row, int cl, float4 o) {
      if (row >= mrows) return;
      const int64_t e = (m0 + row) * p.N + n0 + cl;
      const float f[4] = {o.x, o.y, o.z, o.w};
      if (vec && cl + 4 <= ncols) {
        *reinterpret_cast<float4*>(p.c + e) = o;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (cl + j < ncols) p.c[e + j] = f[j];
      }
      if constexpr (COUNT) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (cl + j < ncols) {
            atomicAdd(p.counts + e + j, 1u);
            p.owner[e + j] = (int32_t)(blockIdx.x / S);
          }
      }
    };
    if constexpr (!kSplit) {
#pragma unroll
      for (int i = 0; i < TM; ++i) store(ty + TY * i, 4 * tx, out[i]);
    } else {
      // the partial blocks meet through distributed shared memory
      float(*Ps)[BN] = reinterpret_cast<float(*)[BN]>(smem);
#pragma unroll
      for (int i = 0; i < TM; ++i) *reinterpret_cast<float4*>(&Ps[ty + TY * i][4 * tx]) = out[i];
      sm100::cluster_sync();  // every CTA's partial is in its shared memory
      auto finish = [&](auto slices) {
        constexpr int kS = decltype(slices)::value, kN = BM * BN / 4 / kS / TH;
        const int row0 = (int)r * (BM / kS) + tid / 16, cl = tid % 16 * 4;
        float4 v[kN][kS];  // all loads before the first sum: one round trip
#pragma unroll
        for (int i = 0; i < kN; ++i)
#pragma unroll
          for (int src = 0; src < kS; ++src)
            v[i][src] = *reinterpret_cast<const float4*>(peer_shared(&Ps[row0 + TH / 16 * i][cl], (uint32_t)src));
        sm100::cluster_sync();  // the peers' reads of this CTA's partial are done
#pragma unroll
        for (int i = 0; i < kN; ++i) {
          float4 sum = v[i][0];
#pragma unroll
          for (int src = 1; src < kS; ++src)
            sum = make_float4(sum.x + v[i][src].x, sum.y + v[i][src].y, sum.z + v[i][src].z, sum.w + v[i][src].w);
          store(row0 + TH / 16 * i, cl, sum);
        }
      };
      if (S == 2) finish(std::integral_constant<int, 2>{});
      else finish(std::integral_constant<int, 4>{});
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

template <int kFetchA, int kFetchB, bool kSplit, bool COUNT>
cudaError_t launch_inst(const SimtArgs& p, int64_t programs, int sms, cudaStream_t st) {
  constexpr auto k = gemm_f32_kernel<kFetchA, kFetchB, kSplit, COUNT>;
  // Clusters are packed onto as few SMs as hold them: a split launch asks for
  // enough shared memory that no SM takes more CTAs than an even spread needs.
  const int64_t per_sm = (programs * p.split + sms - 1) / sms;
  auto spread = [](int64_t ctas) { return std::max(kSmem, kSmemSm / (size_t)(ctas + 1) + 1024); };
  const size_t smem = p.split == 1 || per_sm >= kCtas ? kSmem : spread(per_sm);
  cudaError_t e = allow_smem<k>((int)(kSplit ? spread(1) : kSmem));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(programs * p.split));
  cfg.blockDim = dim3(TH);
  cfg.dynamicSmemBytes = smem;
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

template <int kFetchA, bool kSplit, bool COUNT>
cudaError_t launch_b(const SimtArgs& p, int fetch_b, int64_t programs, int sms, cudaStream_t st) {
  switch (fetch_b) {
    case kRows16: return launch_inst<kFetchA, kRows16, kSplit, COUNT>(p, programs, sms, st);
    case kRows4: return launch_inst<kFetchA, kRows4, kSplit, COUNT>(p, programs, sms, st);
    default: return launch_inst<kFetchA, kCols4, kSplit, COUNT>(p, programs, sms, st);
  }
}

template <bool kSplit, bool COUNT>
cudaError_t launch_a(const SimtArgs& p, int64_t programs, int sms, cudaStream_t st) {
  const int fb = fetch_of(p.b, p.sbk, p.sbn);
  switch (fetch_of(p.a, p.sam, p.sak)) {
    case kRows16: return launch_b<kRows16, kSplit, COUNT>(p, fb, programs, sms, st);
    case kRows4: return launch_b<kRows4, kSplit, COUNT>(p, fb, programs, sms, st);
    default: return launch_b<kCols4, kSplit, COUNT>(p, fb, programs, sms, st);
  }
}

template <bool COUNT>
cudaError_t launch(const SimtArgs& p, int64_t programs, int sms, cudaStream_t st) {
  return p.split > 1 ? launch_a<true, COUNT>(p, programs, sms, st) : launch_a<false, COUNT>(p, programs, sms, st);
}

}  // namespace
}  // namespace tp

// Per-tensor-scaled FP8-E4M3 path: amax reduction, quantisation to E4M3 and
// the scaled tensor-core GEMM entry point.
//
//   amax = max |x| over the whole tensor
//   s    = 448 / amax in fp32 (s = 1 for an all-zero tensor)
//   q    = E4M3(satfinite(RN(x * s)))  (the product in fp32)
//   C    = (qA . qB) * 1 / (s_A * s_B), FP32 accumulation, bf16 output
#include <cuda_bf16.h>

#include <algorithm>

#include "sm100_ptx.cuh"
#include "tp_internal.h"

namespace tp {
namespace {

constexpr int kThreads = 256;

// Sixteen elements as they lie in memory (16-byte pieces), and as floats.
template <typename T> struct Raw {
  static constexpr int N = (int)sizeof(T);  // 16 * sizeof(T) / 16
  uint4 v[N];
};
template <typename T>
__device__ __forceinline__ void load16(Raw<T>& r, const T* p) {
#pragma unroll
  for (int i = 0; i < Raw<T>::N; ++i) r.v[i] = __ldcs(reinterpret_cast<const uint4*>(p) + i);
}
__device__ __forceinline__ void unpack16(const Raw<float>& r, float* f) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[4 * i] = __uint_as_float(r.v[i].x);
    f[4 * i + 1] = __uint_as_float(r.v[i].y);
    f[4 * i + 2] = __uint_as_float(r.v[i].z);
    f[4 * i + 3] = __uint_as_float(r.v[i].w);
  }
}
__device__ __forceinline__ void unpack16(const Raw<__nv_bfloat16>& r, float* f) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r.v[i]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 q = __bfloat1622float2(h[j]);
      f[8 * i + 2 * j] = q.x;
      f[8 * i + 2 * j + 1] = q.y;
    }
  }
}
// Vectors of 16 elements that a thread keeps in flight: 128 bytes.
template <typename T> constexpr int kFlight = 8 / (int)sizeof(T);

__device__ __forceinline__ float ld_f(const float* p) { return *p; }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// *amax = 0, ahead of the reduction's atomics. A kernel rather than a memset,
// so that it and the reduction start as dependents of the work before them.
__global__ void clear_amax_kernel(unsigned* out_bits) {
  sm100::allow_dependents();
  sm100::grid_dependency_wait();
  *out_bits = 0u;
}

// Non-negative floats order like their bit patterns, so max |x| can be taken
// with an unsigned atomicMax on the bits. HBM-bound for large tensors, bound
// by the loads' round trips below: kFlight vectors in flight per thread and a
// grid of one such round per thread where that fills the chip. 2000 x 5120
// bf16 (20 MB), cold: 7.9 us, 8.5 with one vector in flight and four rounds.
template <typename T>
__global__ void __launch_bounds__(kThreads) amax_kernel(const T* __restrict__ x, int64_t n, bool vec,
                                                        unsigned* out_bits) {
  constexpr int U = kFlight<T>;
  sm100::allow_dependents();
  sm100::grid_dependency_wait();
  float m = 0.f;
  const int64_t tid = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t nthreads = (int64_t)gridDim.x * kThreads;
  int64_t done = 0;
  if (vec) {
    const int64_t nv = n / 16;
    for (int64_t v = tid; v < nv; v += U * nthreads) {
      Raw<T> r[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (v + u * nthreads < nv) load16(r[u], x + (v + u * nthreads) * 16);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (v + u * nthreads >= nv) break;
        float f[16];
        unpack16(r[u], f);
#pragma unroll
        for (int i = 0; i < 16; ++i) m = fmaxf(m, fabsf(f[i]));
      }
    }
    done = nv * 16;
  }
  for (int64_t i = done + tid; i < n; i += nthreads) m = fmaxf(m, fabsf(ld_f(x + i)));
  unsigned b = __float_as_uint(m);
  b = __reduce_max_sync(0xffffffffu, b);
  if ((threadIdx.x & 31) == 0 && b != 0) atomicMax(out_bits, b);
}

// Two E4M3 codes from two fp32 values, round to nearest even with
// saturation to +-448; `lo` lands in the low byte.
__device__ __forceinline__ uint16_t cvt_e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}

__device__ __forceinline__ float scale_from_amax(const float* amax) {
  const float a = *amax;
  return a > 0.f ? 448.f / a : 1.f;
}

struct QuantArgs {
  const void* x;
  uint8_t* q;
  int64_t n;
  int64_t tile;      // elements per tile (contiguous)
  int64_t ntiles;
  int32_t kind;      // identity or strided
  int32_t parts;     // CTAs of one program, each on every parts-th round of its tile
  const float* amax;
  float* scale;
  uint32_t* counts;
  int32_t* owner;
};

// A tile program is `parts` CTAs (a tile of few large rows would otherwise keep
// an SM busy for many round trips while others have no tile); each thread has
// kFlight vectors in flight. Bound as amax_kernel is: 2000 x 5120 bf16 in
// 16-row tiles, cold, 14.1 us with one CTA per tile (125 of them, 20 round
// trips each), 8.4 with four. Amax, scale and codes of that tensor and the
// FP8 product with a 10240 x 5120 weight: 105 -> 95.5 us per replay.
template <typename T, bool kCount>
__global__ void __launch_bounds__(kThreads) quantize_kernel(const __grid_constant__ QuantArgs a) {
  constexpr int U = kFlight<T>;
  sm100::allow_dependents();
  sm100::grid_dependency_wait();
  const float s = scale_from_amax(a.amax);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.scale = s;
  const T* x = static_cast<const T*>(a.x);
  const bool vec = (a.tile % 16) == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(a.q)) & 15) == 0;
  const int32_t prog = (int32_t)blockIdx.x / a.parts, part = (int32_t)blockIdx.x % a.parts;
  const int64_t step = a.kind == TP_MAP_IDENTITY ? a.ntiles : (int64_t)gridDim.x / a.parts;
  auto count = [&](int64_t g) {
    if constexpr (kCount) {
      atomicAdd(a.counts + g, 1u);
      a.owner[g] = prog;
    }
  };
  for (int64_t t = prog; t < a.ntiles; t += step) {
    const int64_t start = t * a.tile;
    const int64_t len = min(a.tile, a.n - start);
    int64_t done = 0;
    if (vec) {
      const int64_t nv = len / 16;
      for (int64_t v = (int64_t)part * U * kThreads + threadIdx.x; v < nv; v += (int64_t)a.parts * U * kThreads) {
        Raw<T> r[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (v + u * kThreads < nv) load16(r[u], x + start + (v + u * kThreads) * 16);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (v + u * kThreads >= nv) break;
          float f[16];
          unpack16(r[u], f);
          uint4 out;
          uint16_t* h = reinterpret_cast<uint16_t*>(&out);
#pragma unroll
          for (int i = 0; i < 8; ++i) h[i] = cvt_e4m3x2(f[2 * i] * s, f[2 * i + 1] * s);
          const int64_t g = start + (v + u * kThreads) * 16;
          *reinterpret_cast<uint4*>(a.q + g) = out;
          if constexpr (kCount)
            for (int i = 0; i < 16; ++i) count(g + i);
        }
      }
      done = nv * 16;
    }
    for (int64_t i = done + (int64_t)part * kThreads + threadIdx.x; i < len; i += (int64_t)a.parts * kThreads) {
      const int64_t g = start + i;
      a.q[g] = (uint8_t)(cvt_e4m3x2(ld_f(x + g) * s, 0.f) & 0xFF);
      count(g);
    }
  }
}

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), int64_t grid, int threads, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T>
cudaError_t launch_amax(const T* x, int64_t n, int sms, unsigned* bits, cudaStream_t st) {
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const int64_t per = (int64_t)kThreads * (vec ? 16 * kFlight<T> : 16);  // elements of a CTA's round
  const int64_t grid = std::min<int64_t>((n + per - 1) / per, 8 * (int64_t)sms);
  return launch_pdl(amax_kernel<T>, grid, kThreads, st, x, n, vec, bits);
}

template <typename T>
cudaError_t launch_quantize(QuantArgs a, int64_t programs, int sms, cudaStream_t st) {
  // as many CTAs per program as keep every SM's four busy, each with a round
  const int64_t rounds = (std::min(a.tile, a.n) + (int64_t)kThreads * 16 * kFlight<T> - 1) / ((int64_t)kThreads * 16 * kFlight<T>);
  a.parts = (int32_t)std::max<int64_t>(1, std::min<int64_t>(rounds, 4 * (int64_t)sms / programs));
  return a.counts ? launch_pdl(quantize_kernel<T, true>, programs * a.parts, kThreads, st, a)
                  : launch_pdl(quantize_kernel<T, false>, programs * a.parts, kThreads, st, a);
}

}  // namespace
}  // namespace tp

using namespace tp;

extern "C" {

tp_status tp_amax(tp_ctx* ctx, const tp_tensor* x, float* amax, const tp_exec* ex) {
  if (!ctx || !x || !amax || !ex) return fail(TP_ERR_INVALID, "null argument");
  if (x->dtype != TP_F32 && x->dtype != TP_BF16) return fail(TP_ERR_UNSUPPORTED, "amax supports F32 and BF16");
  if (!is_contiguous(*x)) return fail(TP_ERR_UNSUPPORTED, "amax input must be contiguous");
  Op o(__func__);
  tp_status s = o.begin(ctx, ex, {}, {x});
  if (s != TP_OK) return s;
  const int64_t n = numel(*x);
  unsigned* bits = reinterpret_cast<unsigned*>(amax);
  cudaError_t e = launch_pdl(clear_amax_kernel, 1, 1, o.stream, bits);
  if (e == cudaSuccess && n > 0)
    e = x->dtype == TP_F32 ? launch_amax(static_cast<const float*>(x->ptr), n, ctx->sm_count, bits, o.stream)
                           : launch_amax(static_cast<const __nv_bfloat16*>(x->ptr), n, ctx->sm_count, bits, o.stream);
  return o.end(e);
}

tp_status tp_quantize_fp8(tp_ctx* ctx, tp_partition* q, const tp_tensor* x, const float* amax, float* scale,
                          const tp_exec* ex) {
  if (!ctx || !q || !x || !amax || !scale || !ex) return fail(TP_ERR_INVALID, "null argument");
  if (x->dtype != TP_F32 && x->dtype != TP_BF16) return fail(TP_ERR_UNSUPPORTED, "quantize input must be F32 or BF16");
  if (q->t.dtype != TP_F8E4M3 && q->t.dtype != TP_U8) return fail(TP_ERR_SHAPE, "quantize output must be F8E4M3");
  if (x->rank != q->rank) return fail(TP_ERR_SHAPE, "input rank differs from output rank");
  for (int i = 0; i < q->rank; ++i)
    if (x->shape[i] != q->shape[i]) return fail(TP_ERR_SHAPE, "input shape differs from output shape");
  if (!is_contiguous(*x)) return fail(TP_ERR_UNSUPPORTED, "quantize input must be contiguous");
  // each tile must be one contiguous run of elements: full rows beyond axis 0
  int64_t tile = q->tile[0];
  for (int i = 1; i < q->rank; ++i) {
    if (q->tile[i] != q->shape[i]) return fail(TP_ERR_UNSUPPORTED, "quantize tiles must span whole rows");
    tile *= q->shape[i];
  }
  if (q->kind == TP_MAP_QUEUE) return fail(TP_ERR_UNSUPPORTED, "quantize maps tiles by slot (identity/strided)");
  if ((ex->write_counts == nullptr) != (ex->write_owner == nullptr))
    return fail(TP_ERR_INVALID, "write_counts and write_owner must be given together");
  Op o(__func__);
  tp_status s = o.begin(ctx, ex, {q}, {x});
  if (s != TP_OK) return s;
  QuantArgs a{};
  a.x = x->ptr;
  a.q = static_cast<uint8_t*>(q->t.ptr);
  a.n = numel(*x);
  a.tile = tile;
  a.ntiles = q->num_tiles;
  a.kind = q->kind;
  a.amax = amax;
  a.scale = scale;
  a.counts = ex->write_counts;
  a.owner = ex->write_owner;
  const int64_t grid = q->kind == TP_MAP_IDENTITY ? q->num_tiles : q->num_programs;
  if (grid > 0x7fffffff) {
    o.abort();
    return fail(TP_ERR_UNSUPPORTED, "too many tile programs");
  }
  cudaError_t e = cudaSuccess;
  if (a.n > 0)
    e = x->dtype == TP_F32 ? launch_quantize<float>(a, grid, ctx->sm_count, o.stream)
                           : launch_quantize<__nv_bfloat16>(a, grid, ctx->sm_count, o.stream);
  return o.end(e);
}

tp_status tp_gemm_fp8(tp_ctx* ctx, tp_partition* c, const tp_tensor* qa, const tp_tensor* qb,
                      const float* scale_a, const float* scale_b, const tp_gemm_config* cfg, const tp_exec* ex) {
  if (!ctx || !c || !qa || !qb || !scale_a || !scale_b || !ex) return fail(TP_ERR_INVALID, "null argument");
  if (qa->rank != 2 || qb->rank != 2 || c->rank != 2) return fail(TP_ERR_RANK, "GEMM operands are rank 2");
  const int64_t M = qa->shape[0], K = qa->shape[1], N = qb->shape[1];
  if (qb->shape[0] != K || c->shape[0] != M || c->shape[1] != N)
    return fail(TP_ERR_SHAPE, "need A: M x K, B: K x N, C: M x N");
  auto f8 = [](int32_t d) { return d == TP_F8E4M3 || d == TP_U8; };
  if (!f8(qa->dtype) || !f8(qb->dtype) || c->t.dtype != TP_BF16)
    return fail(TP_ERR_UNSUPPORTED, "tp_gemm_fp8 takes E4M3 A and B and a BF16 C");
  Op o(__func__);
  o.allow_checked = true;
  tp_status s = o.begin(ctx, ex, {c}, {qa, qb});
  if (s != TP_OK) return s;
  o.check_err = true;
  s = launch_gemm_tc_impl(ctx, c, qa, qb, cfg, ex, o.stream, 1, scale_a, scale_b, o.err);
  if (s != TP_OK) {
    o.abort();
    return s;
  }
  return o.end(cudaGetLastError());
}

}  // extern "C"

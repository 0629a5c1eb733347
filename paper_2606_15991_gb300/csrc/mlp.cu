// Learned tile proposer: a 3-layer ReLU MLP that scores every configuration
// of the GEMM autotuner's single-pass class for a shape (features: log2 M,
// log2 N, log2 K and a one-hot dtype), trained on the GPU by this file's
// kernels on the autotuner's own measurements (target: TFLOP/s of the config
// over the best TFLOP/s of the shape). The proposal is the arg-max config;
// the exhaustive autotuner over the same class stays the fallback for low
// scores and shapes outside the trained range. Every config of that class
// computes each C element as one K-ordered accumulation by one program, so
// whichever config the proposal or its fallback picks, C is bit-identical:
// the proposal never changes numerics. Split-K configs, which round
// differently, are outside the class and never proposed.
//
//   h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), y = W3 h2 + b3
//   L  = sum V (y - T)^2 / max(1, sum V)      (V masks invalid configs)
//   Adam with bias correction.
// Parameters are one contiguous fp32 buffer [W1, b1, W2, b2, W3, b3] (row-
// major [out, in] matrices). Every reduction runs in a fixed order, so
// training is deterministic.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "sm100_ptx.cuh"
#include "tp_internal.h"

struct tp_mlp {
  tp_ctx* ctx = nullptr;
  int32_t in = 0, hidden = 0, out = 0, max_batch = 0;
  int64_t nparams = 0;
  int64_t step = 0;
  float* params = nullptr;  // device
  float* m = nullptr;
  float* v = nullptr;
  float* h1 = nullptr;      // [B, H] activations
  float* h2 = nullptr;
  float* y = nullptr;       // [B, C] scores (propose, and outputs that overlap X)
  float* grads = nullptr;   // gradients whose output overlaps X
  float* dy = nullptr;      // [B, C] unscaled loss gradient
  float* dz1 = nullptr;     // [B, H]
  float* dz2 = nullptr;
  float* part = nullptr;    // partial loss sums, two per CTA of the rows kernel
  float* xbuf = nullptr;    // [B, in] features (propose)
};

namespace tp {
namespace {

struct Off {
  int64_t w1, b1, w2, b2, w3, b3, n;
};

__host__ __device__ inline Off offsets(int F, int H, int C) {
  Off o;
  o.w1 = 0;
  o.b1 = o.w1 + (int64_t)H * F;
  o.w2 = o.b1 + H;
  o.b2 = o.w2 + (int64_t)H * H;
  o.w3 = o.b2 + H;
  o.b3 = o.w3 + (int64_t)C * H;
  o.n = o.b3 + C;
  return o;
}

__device__ __forceinline__ void copy4_async(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sm100::smem_u32(dst)), "l"(src), "r"(valid ? 4 : 0)
               : "memory");
}

// ------------------------------------------------------------ rows kernel
// Forward and, with kGrad, backward through the activations of two batch rows
// per CTA, 128 threads a row: thread j computes units j, j + 128, ... of each
// layer, summing over the layer's inputs in order. All weights are first
// copied to shared memory (rows padded to an odd stride, so that both a
// product with W and one with W^T read distinct banks); a network too large
// for that reads them from global memory. Bound by latency: one copy of the
// weights and five short dependent sums. One row per CTA with uncoalesced
// weight reads, a one-block loss and a second row kernel took 12.4, 13.4 and
// 17.9 us of a 256-row batch of the 5-64-64-72 network (ncu); with
// grads_kernel's 77 us, and two launches instead of four and a copy, the
// synchronous loss-and-gradients call went from 106 to 28 us, most of them
// the call itself.
// The gradient of the loss is left unscaled here (2 V (y - T)): the divisor
// max(1, sum V) spans the batch, so grads_kernel applies it to the sums.
constexpr int kRowThreads = 128;
constexpr int kRowsPerCta = 2;

struct RowsArgs {
  const float* P;
  const float* X;
  const float* T;   // kGrad: targets, mask
  const float* V;
  int32_t B, F, H, C;
  int32_t ld1, ld2;  // row strides of W1 and of W2, W3 as read
  int32_t staged;    // weights and biases in shared memory
  float* Y;          // [B, C] or null
  float* h1;         // kGrad, [B, H]: activations and the gradients at z1, z2
  float* h2;
  float* dz1;
  float* dz2;
  float* dy;         // kGrad, [B, C]
  float* part;       // kGrad: {sum V, sum V d^2} of each CTA
};

// Shared memory of the rows kernel, in floats: activations of the CTA's rows,
// then the staged parameters.
__host__ __device__ inline int64_t rows_acts(int H, int C) { return (int64_t)kRowsPerCta * (3 * H + C); }
__host__ __device__ inline int64_t rows_params(int F, int H, int C) {
  return (int64_t)H * (F | 1) + (int64_t)(H + C) * (H | 1) + 2 * H + C;
}

template <bool kGrad>
__global__ void __launch_bounds__(kRowThreads* kRowsPerCta) rows_kernel(const __grid_constant__ RowsArgs a) {
  extern __shared__ float sh[];
  __shared__ float red[2][kRowThreads * kRowsPerCta / 32];
  const int F = a.F, H = a.H, C = a.C;
  const Off o = offsets(F, H, C);
  const int tid = threadIdx.x, g = tid / kRowThreads, j0 = tid % kRowThreads;
  const int b = blockIdx.x * kRowsPerCta + g;
  const bool row = b < a.B;
  float* h1s = sh + g * (3 * H + C);
  float* h2s = h1s + H;
  float* dz2s = h2s + H;
  float* dys = dz2s + H;
  const float *w1 = a.P + o.w1, *w2 = a.P + o.w2, *w3 = a.P + o.w3, *b1 = a.P + o.b1, *b2 = a.P + o.b2, *b3 = a.P + o.b3;
  sm100::grid_dependency_wait();
  sm100::allow_dependents();
  if (a.staged) {
    float* q = sh + rows_acts(H, C);
    auto stage = [&](const float*& w, int rows, int cols, int ld) {
      const int lane = tid & 31;
      for (int r = tid / 32; r < rows; r += kRowThreads * kRowsPerCta / 32)
        for (int c = lane; c < cols; c += 32) copy4_async(q + (int64_t)r * ld + c, w + (int64_t)r * cols + c, true);
      w = q;
      q += (int64_t)rows * ld;
    };
    stage(w1, H, F, a.ld1);
    stage(b1, 1, H, H);
    stage(w2, H, H, a.ld2);
    stage(b2, 1, H, H);
    stage(w3, C, H, a.ld2);
    stage(b3, 1, C, C);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const float* x = a.X + (int64_t)b * F;
  // the loss's inputs of this thread's first output, fetched ahead of their use
  float t0 = 0.f, v0 = 0.f;
  if (kGrad && row && j0 < C) {
    t0 = a.T[(int64_t)b * C + j0];
    v0 = a.V[(int64_t)b * C + j0];
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  for (int j = j0; j < H; j += kRowThreads) {
    float s = b1[j];
    for (int f = 0; f < F; ++f) s = fmaf(w1[(int64_t)j * a.ld1 + f], row ? x[f] : 0.f, s);
    s = fmaxf(s, 0.f);
    h1s[j] = s;
    if (kGrad && row) a.h1[(int64_t)b * H + j] = s;
  }
  __syncthreads();
  for (int j = j0; j < H; j += kRowThreads) {
    float s = b2[j];
    const float* w = w2 + (int64_t)j * a.ld2;
#pragma unroll 8
    for (int i = 0; i < H; ++i) s = fmaf(w[i], h1s[i], s);
    s = fmaxf(s, 0.f);
    h2s[j] = s;
    if (kGrad && row) a.h2[(int64_t)b * H + j] = s;
  }
  __syncthreads();
  float sv = 0.f, se = 0.f;
  for (int c = j0; c < C; c += kRowThreads) {
    float s = b3[c];
    const float* w = w3 + (int64_t)c * a.ld2;
#pragma unroll 8
    for (int i = 0; i < H; ++i) s = fmaf(w[i], h2s[i], s);
    if (row && a.Y) a.Y[(int64_t)b * C + c] = s;
    if constexpr (kGrad) {
      float t = t0, v = v0;
      if (c != j0 && row) {
        t = a.T[(int64_t)b * C + c];
        v = a.V[(int64_t)b * C + c];
      }
      const float d = row ? s - t : 0.f;
      v = row ? v : 0.f;
      sv += v;
      se = fmaf(v * d, d, se);
      const float dy = 2.f * v * d;
      dys[c] = dy;
      if (row) a.dy[(int64_t)b * C + c] = dy;
    }
  }
  if constexpr (kGrad) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      sv += __shfl_xor_sync(0xffffffffu, sv, off);
      se += __shfl_xor_sync(0xffffffffu, se, off);
    }
    if ((tid & 31) == 0) {
      red[0][tid / 32] = sv;
      red[1][tid / 32] = se;
    }
    __syncthreads();
    if (tid < 2) {
      float s = 0.f;
      for (int w = 0; w < kRowThreads * kRowsPerCta / 32; ++w) s += red[tid][w];  // fixed order
      a.part[2 * (int64_t)blockIdx.x + tid] = s;
    }
    // dz2 = (dy W3) * (h2 > 0), dz1 = (dz2 W2) * (h1 > 0)
    for (int j = j0; j < H; j += kRowThreads) {
      float s = 0.f;
#pragma unroll 8
      for (int c = 0; c < C; ++c) s = fmaf(dys[c], w3[(int64_t)c * a.ld2 + j], s);
      s = h2s[j] > 0.f ? s : 0.f;
      dz2s[j] = s;
      if (row) a.dz2[(int64_t)b * H + j] = s;
    }
    __syncthreads();
    for (int j = j0; j < H; j += kRowThreads) {
      float s = 0.f;
#pragma unroll 8
      for (int i = 0; i < H; ++i) s = fmaf(dz2s[i], w2[(int64_t)i * a.ld2 + j], s);
      if (row) a.dz1[(int64_t)b * H + j] = h1s[j] > 0.f ? s : 0.f;
    }
  }
}

// ----------------------------------------------------------- grads kernel
// Every parameter's gradient: products left^T right over the batch rows, in
// row order, one 8 x 32 block of a weight matrix per CTA (one element per
// thread), both factors brought in chunks of 128 rows by asynchronous copies;
// the CTAs of a matrix's first columns also sum its bias. Then the batch's
// divisor is applied and, with lr > 0, one Adam step is taken on the element,
// so that a training step is two launches. One thread per parameter walking
// the batch took 77 us of a 256-row batch; both kernels together now take less
// than the launch overhead of the synchronous call (28 us, see rows_kernel).
constexpr int kGradRows = 8, kGradCols = 32, kGradChunk = 128;
constexpr int kGradThreads = kGradRows * kGradCols;

struct GradsArgs {
  int32_t B, F, H, C, parts;
  const float* X;
  const float* h1;
  const float* h2;
  const float* dz1;
  const float* dz2;
  const float* dy;
  const float* part;  // rows_kernel's partial sums
  float* G;           // gradients out, or null
  float* loss;        // or null
  float* P;           // Adam: parameters and moments, or null: no step
  float* m;
  float* v;
  float lr, c1, c2;
};

__device__ __forceinline__ void grad_out(const GradsArgs& a, int64_t i, float g) {
  if (a.G) a.G[i] = g;
  if (a.P) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float m = b1 * a.m[i] + (1.f - b1) * g;
    const float v = b2 * a.v[i] + (1.f - b2) * g * g;
    a.m[i] = m;
    a.v[i] = v;
    a.P[i] -= a.lr * (m / a.c1) / (sqrtf(v / a.c2) + eps);
  }
}

__global__ void __launch_bounds__(kGradThreads) grads_kernel(const __grid_constant__ GradsArgs a) {
  __shared__ float left[2][kGradChunk][kGradRows];
  __shared__ float right[2][kGradChunk][kGradCols];
  __shared__ float red[2][kGradThreads / 32];
  const int F = a.F, H = a.H, C = a.C;
  const Off o = offsets(F, H, C);
  // this CTA's block: W3 = dy^T h2, then W2 = dz2^T h1, then W1 = dz1^T X
  auto blocks = [](int rows, int cols) { return (rows + kGradRows - 1) / kGradRows * ((cols + kGradCols - 1) / kGradCols); };
  int blk = blockIdx.x;
  const float *L = a.dy, *R = a.h2;
  int rows = C, cols = H;
  int64_t w = o.w3, bias = o.b3;
  if (blk >= blocks(C, H)) {
    blk -= blocks(C, H);
    L = a.dz2;
    R = a.h1;
    rows = H;
    w = o.w2;
    bias = o.b2;
    if (blk >= blocks(H, H)) {
      blk -= blocks(H, H);
      L = a.dz1;
      R = a.X;
      cols = F;
      w = o.w1;
      bias = o.b1;
    }
  }
  const int cblocks = (cols + kGradCols - 1) / kGradCols;
  const int r0 = blk / cblocks * kGradRows, c0 = blk % cblocks * kGradCols;
  const int tid = threadIdx.x, r = tid / kGradCols, c = tid % kGradCols;
  sm100::grid_dependency_wait();
  sm100::allow_dependents();
  auto load = [&](int chunk) {
    const int b0 = chunk * kGradChunk, buf = chunk & 1;
#pragma unroll
    for (int e = 0; e < kGradChunk * kGradRows / kGradThreads; ++e) {
      const int i = e * kGradThreads + tid, bb = i / kGradRows, rr = i % kGradRows;
      const bool ok = b0 + bb < a.B && r0 + rr < rows;
      copy4_async(&left[buf][bb][rr], ok ? L + (int64_t)(b0 + bb) * rows + r0 + rr : L, ok);
    }
#pragma unroll
    for (int e = 0; e < kGradChunk * kGradCols / kGradThreads; ++e) {
      const int bb = e * (kGradThreads / kGradCols) + r;
      const bool ok = b0 + bb < a.B && c0 + c < cols;
      copy4_async(&right[buf][bb][c], ok ? R + (int64_t)(b0 + bb) * cols + c0 + c : R, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int chunks = (a.B + kGradChunk - 1) / kGradChunk;
  load(0);
  if (chunks > 1) load(1);
  // the divisor max(1, sum V) and the loss, from the rows kernel's partial
  // sums in a fixed order
  float sv = 0.f, se = 0.f;
  for (int i = tid; i < a.parts; i += kGradThreads) {
    sv += a.part[2 * (int64_t)i];
    se += a.part[2 * (int64_t)i + 1];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sv += __shfl_xor_sync(0xffffffffu, sv, off);
    se += __shfl_xor_sync(0xffffffffu, se, off);
  }
  if ((tid & 31) == 0) {
    red[0][tid / 32] = sv;
    red[1][tid / 32] = se;
  }
  float s = 0.f, sb = 0.f;
  for (int chunk = 0; chunk < chunks; ++chunk) {
    const int buf = chunk & 1;
    if (chunk + 1 < chunks) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int n = min(kGradChunk, a.B - chunk * kGradChunk);
#pragma unroll 8
    for (int bb = 0; bb < n; ++bb) {
      const float l = left[buf][bb][r];
      s = fmaf(l, right[buf][bb][c], s);
      sb += l;
    }
    __syncthreads();
    if (chunk + 2 < chunks) load(chunk + 2);
  }
  float tv = 0.f, te = 0.f;
  for (int q = 0; q < kGradThreads / 32; ++q) {
    tv += red[0][q];
    te += red[1][q];
  }
  const float den = fmaxf(1.f, tv);
  if (blockIdx.x == 0 && tid == 0 && a.loss) *a.loss = te / den;
  if (r0 + r < rows) {
    if (c0 + c < cols) grad_out(a, w + (int64_t)(r0 + r) * cols + c0 + c, s / den);
    if (c0 + c == 0) grad_out(a, bias + r0 + r, sb / den);
  }
}

// Shared memory of the rows kernel that the weights may take part in.
constexpr size_t kRowsSmem = 200 * 1024;

template <auto K, typename A>
cudaError_t launch_pdl(const A& a, int grid, int threads, size_t smem, cudaStream_t st) {
  if (smem > 48 * 1024) {
    cudaError_t e = allow_smem<K>((int)kRowsSmem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, K, a);
}

int row_ctas(int B) { return (B + kRowsPerCta - 1) / kRowsPerCta; }

cudaError_t launch_rows(tp_mlp* n, const float* X, const float* T, const float* V, int B, float* Y, cudaStream_t st) {
  RowsArgs a{};
  a.P = n->params;
  a.X = X;
  a.T = T;
  a.V = V;
  a.B = B;
  a.F = n->in;
  a.H = n->hidden;
  a.C = n->out;
  a.Y = Y;
  a.h1 = n->h1;
  a.h2 = n->h2;
  a.dz1 = n->dz1;
  a.dz2 = n->dz2;
  a.dy = n->dy;
  a.part = n->part;
  // the weights stay in global memory when they do not fit beside the
  // activations (32 KB at most)
  const int64_t params = rows_params(a.F, a.H, a.C), acts = rows_acts(a.H, a.C);
  a.staged = (params + acts) * sizeof(float) <= kRowsSmem ? 1 : 0;
  a.ld1 = a.staged ? a.F | 1 : a.F;
  a.ld2 = a.staged ? a.H | 1 : a.H;
  const size_t smem = (size_t)(acts + (a.staged ? params : 0)) * sizeof(float);
  const int threads = kRowThreads * kRowsPerCta;
  return T ? launch_pdl<rows_kernel<true>>(a, row_ctas(B), threads, smem, st)
           : launch_pdl<rows_kernel<false>>(a, row_ctas(B), threads, smem, st);
}

// An output over the bytes of X: the kernels write outputs while other CTAs
// read X, so it is written to the network's own buffer and copied out last.
bool overlap(const float* out, size_t bytes, const float* x, size_t xbytes) {
  const uintptr_t o = reinterpret_cast<uintptr_t>(out), i = reinterpret_cast<uintptr_t>(x);
  return o < i + xbytes && i < o + bytes;
}

tp_status launch_forward(tp_mlp* n, const float* X, int B, float* Y, cudaStream_t st) {
  const cudaError_t e = launch_rows(n, X, nullptr, nullptr, B, Y, st);
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "mlp forward");
}

// Forward, loss and gradients (to G when not null); step > 0 takes Adam step
// `step` at learning rate lr.
tp_status launch_loss_grad(tp_mlp* n, const float* X, const float* T, const float* V, int B, float* loss, float* G,
                           int64_t step, float lr, cudaStream_t st) {
  cudaError_t e = launch_rows(n, X, T, V, B, nullptr, st);
  if (e != cudaSuccess) return cuda_fail(e, "mlp forward");
  GradsArgs a{};
  a.B = B;
  a.F = n->in;
  a.H = n->hidden;
  a.C = n->out;
  a.parts = row_ctas(B);
  a.X = X;
  a.h1 = n->h1;
  a.h2 = n->h2;
  a.dz1 = n->dz1;
  a.dz2 = n->dz2;
  a.dy = n->dy;
  a.part = n->part;
  a.G = G;
  a.loss = loss;
  if (step > 0) {
    a.P = n->params;
    a.m = n->m;
    a.v = n->v;
    a.lr = lr;
    a.c1 = 1.f - (float)std::pow(0.9, (double)step);
    a.c2 = 1.f - (float)std::pow(0.999, (double)step);
  }
  auto blocks = [](int rows, int cols) { return (rows + kGradRows - 1) / kGradRows * ((cols + kGradCols - 1) / kGradCols); };
  const int grid = blocks(a.C, a.H) + blocks(a.H, a.H) + blocks(a.H, a.F);
  e = launch_pdl<grads_kernel>(a, grid, kGradThreads, 0, st);
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "mlp backward");
}

}  // namespace
}  // namespace tp

using namespace tp;

extern "C" {

tp_status tp_mlp_create(tp_ctx* ctx, int32_t in, int32_t hidden, int32_t out, int32_t max_batch,
                        const float* init_params, tp_mlp** mlp) {
  if (!ctx || !mlp || !init_params) return fail(TP_ERR_INVALID, "null argument");
  *mlp = nullptr;
  DeviceGuard guard(ctx);
  if (in < 1 || hidden < 1 || out < 1 || hidden > 1024 || out > 1024 || max_batch < 1)
    return fail(TP_ERR_INVALID, "need 1 <= in, 1 <= hidden, out <= 1024, max_batch >= 1");
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (ctx->capturing) return fail(TP_ERR_CAPTURE, "creating an MLP allocates device memory");
  }
  auto* n = new tp_mlp();
  n->ctx = ctx;
  n->in = in;
  n->hidden = hidden;
  n->out = out;
  n->max_batch = max_batch;
  n->nparams = offsets(in, hidden, out).n;
  const size_t P = n->nparams * sizeof(float), BH = (size_t)max_batch * hidden * sizeof(float),
               BC = (size_t)max_batch * out * sizeof(float);
  cudaError_t e = cudaSuccess;
  for (auto pr : {std::make_pair(&n->params, P), std::make_pair(&n->grads, P), std::make_pair(&n->m, P),
                  std::make_pair(&n->v, P),
                  std::make_pair(&n->h1, BH), std::make_pair(&n->h2, BH), std::make_pair(&n->y, BC),
                  std::make_pair(&n->dy, BC), std::make_pair(&n->dz1, BH), std::make_pair(&n->dz2, BH),
                  std::make_pair(&n->part, 2 * (size_t)row_ctas(max_batch) * sizeof(float)),
                  std::make_pair(&n->xbuf, (size_t)max_batch * in * sizeof(float))})
    if (e == cudaSuccess) e = cudaMalloc(pr.first, pr.second);
  if (e == cudaSuccess) e = cudaMemcpy(n->params, init_params, P, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, P);
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, P);
  if (e != cudaSuccess) {
    for (float* p : {n->params, n->grads, n->m, n->v, n->h1, n->h2, n->y, n->dy, n->dz1, n->dz2, n->part, n->xbuf}) cudaFree(p);
    delete n;
    return cuda_fail(e, "allocating the MLP");
  }
  *mlp = n;
  return TP_OK;
}

tp_status tp_mlp_destroy(tp_mlp* n) {
  if (!n) return fail(TP_ERR_INVALID, "null mlp");
  for (float* p : {n->params, n->grads, n->m, n->v, n->h1, n->h2, n->y, n->dy, n->dz1, n->dz2, n->part, n->xbuf}) cudaFree(p);
  delete n;
  return TP_OK;
}

tp_status tp_mlp_num_params(const tp_mlp* n, int64_t* count) {
  if (!n || !count) return fail(TP_ERR_INVALID, "null argument");
  *count = n->nparams;
  return TP_OK;
}

tp_status tp_mlp_get_params(const tp_mlp* n, float* host_out) {
  if (!n || !host_out) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  cudaError_t e = cudaMemcpy(host_out, n->params, n->nparams * sizeof(float), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "reading MLP parameters");
}

tp_status tp_mlp_set_params(tp_mlp* n, const float* host_in) {
  if (!n || !host_in) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  cudaError_t e = cudaMemcpy(n->params, host_in, n->nparams * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, n->nparams * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, n->nparams * sizeof(float));
  n->step = 0;
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "writing MLP parameters");
}

tp_status tp_mlp_forward(tp_mlp* n, const float* X, int32_t batch, float* Y, const tp_exec* ex) {
  if (!n || !X || !Y || !ex) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  if (batch < 1 || batch > n->max_batch) return fail(TP_ERR_SHAPE, "batch must be 1..max_batch");
  cudaStream_t st = static_cast<cudaStream_t>(ex->stream);
  const size_t bytes = (size_t)batch * n->out * sizeof(float);
  const bool over = overlap(Y, bytes, X, (size_t)batch * n->in * sizeof(float));
  tp_status s = launch_forward(n, X, batch, over ? n->y : Y, st);
  if (s != TP_OK) return s;
  cudaError_t e = over ? cudaMemcpyAsync(Y, n->y, bytes, cudaMemcpyDeviceToDevice, st) : cudaSuccess;
  if (e == cudaSuccess && ex->mode == TP_SYNC) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "mlp forward output");
}

tp_status tp_mlp_loss_grad(tp_mlp* n, const float* X, const float* T, const float* V, int32_t batch, float* loss,
                           float* grads, const tp_exec* ex) {
  if (!n || !X || !T || !V || !ex) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  if (batch < 1 || batch > n->max_batch) return fail(TP_ERR_SHAPE, "batch must be 1..max_batch");
  cudaStream_t st = static_cast<cudaStream_t>(ex->stream);
  const size_t bytes = n->nparams * sizeof(float);
  const bool over = grads && overlap(grads, bytes, X, (size_t)batch * n->in * sizeof(float));
  tp_status s = launch_loss_grad(n, X, T, V, batch, loss, over ? n->grads : grads, 0, 0.f, st);
  if (s != TP_OK) return s;
  cudaError_t e = over ? cudaMemcpyAsync(grads, n->grads, bytes, cudaMemcpyDeviceToDevice, st) : cudaSuccess;
  if (e == cudaSuccess && ex->mode == TP_SYNC) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "mlp gradients");
}

tp_status tp_mlp_train_step(tp_mlp* n, const float* X, const float* T, const float* V, int32_t batch, float lr,
                            float* loss, const tp_exec* ex) {
  if (!n || !X || !T || !V || !ex) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  if (batch < 1 || batch > n->max_batch) return fail(TP_ERR_SHAPE, "batch must be 1..max_batch");
  cudaStream_t st = static_cast<cudaStream_t>(ex->stream);
  tp_status s = launch_loss_grad(n, X, T, V, batch, loss, nullptr, n->step + 1, lr, st);
  if (s != TP_OK) return s;
  n->step += 1;
  cudaError_t e = cudaSuccess;
  if (ex->mode == TP_SYNC) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? TP_OK : cuda_fail(e, "mlp train step");
}

tp_status tp_mlp_save(const tp_mlp* n, const char* path) {
  if (!n || !path) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  std::vector<float> h(n->nparams);
  tp_status s = tp_mlp_get_params(n, h.data());
  if (s != TP_OK) return s;
  FILE* f = std::fopen(path, "w");
  if (!f) return fail(TP_ERR_INVALID, std::string("cannot write ") + path);
  std::fprintf(f, "tp-mlp v1 %d %d %d\n", n->in, n->hidden, n->out);
  for (float v : h) std::fprintf(f, "%.9g\n", v);
  std::fclose(f);
  return TP_OK;
}

tp_status tp_mlp_load(tp_mlp* n, const char* path) {
  if (!n || !path) return fail(TP_ERR_INVALID, "null argument");
  DeviceGuard guard(n->ctx);
  FILE* f = std::fopen(path, "r");
  if (!f) return fail(TP_ERR_INVALID, std::string("cannot read ") + path);
  int a = 0, b = 0, c = 0;
  if (std::fscanf(f, "tp-mlp v1 %d %d %d", &a, &b, &c) != 3 || a != n->in || b != n->hidden || c != n->out) {
    std::fclose(f);
    return fail(TP_ERR_SHAPE, "MLP file does not match this network");
  }
  std::vector<float> h(n->nparams);
  for (auto& v : h)
    if (std::fscanf(f, "%f", &v) != 1) {
      std::fclose(f);
      return fail(TP_ERR_INVALID, "truncated MLP file");
    }
  std::fclose(f);
  return tp_mlp_set_params(n, h.data());
}

tp_status tp_mlp_features(int64_t M, int64_t N, int64_t K, int32_t dtype, float* out) {
  if (!out) return fail(TP_ERR_INVALID, "null output");
  if (M < 1 || N < 1 || K < 1) return fail(TP_ERR_SHAPE, "dimensions must be >= 1");
  if (dtype != TP_BF16 && dtype != TP_F8E4M3) return fail(TP_ERR_UNSUPPORTED, "dtype must be BF16 or F8E4M3");
  out[0] = (float)std::log2((double)M);
  out[1] = (float)std::log2((double)N);
  out[2] = (float)std::log2((double)K);
  out[3] = dtype == TP_BF16 ? 1.f : 0.f;
  out[4] = dtype == TP_BF16 ? 0.f : 1.f;
  return TP_OK;
}

tp_status tp_mlp_targets(const float* tflops, int32_t count, float* target, float* mask) {
  if (!tflops || !target || !mask || count < 1) return fail(TP_ERR_INVALID, "null argument or empty table");
  float best = 0.f;
  for (int i = 0; i < count; ++i) best = std::max(best, tflops[i]);
  // a config that did not run on the shape is its worst proposal: target 0,
  // still trained (an untrained output could otherwise win the arg-max)
  for (int i = 0; i < count; ++i) {
    mask[i] = best > 0.f ? 1.f : 0.f;
    target[i] = best > 0.f ? std::max(tflops[i], 0.f) / best : 0.f;
  }
  return TP_OK;
}

tp_status tp_propose(tp_ctx* ctx, tp_mlp* n, int64_t M, int64_t N, int64_t K, int32_t dtype, float min_score,
                     tp_gemm_config* out, float* score, int32_t* used_fallback) {
  if (!ctx || !n || !out) return fail(TP_ERR_INVALID, "null argument");
  if (n->in != 5) return fail(TP_ERR_SHAPE, "the proposer takes 5 features");
  int32_t count = 0;
  tp_status s = tp_autotune_space(dtype, 0, nullptr, 0, &count);
  if (s != TP_OK) return s;
  if (count != n->out) return fail(TP_ERR_SHAPE, "MLP outputs differ from the autotuner's single-pass config count");
  std::vector<tp_gemm_config> cfgs(count);
  tp_autotune_space(dtype, 0, cfgs.data(), count, &count);
  float x[5];
  s = tp_mlp_features(M, N, K, dtype, x);
  if (s != TP_OK) return s;
  cudaError_t e = cudaMemcpy(n->xbuf, x, sizeof(x), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "proposer features");
  s = launch_forward(n, n->xbuf, 1, n->y, nullptr);
  if (s != TP_OK) return s;
  std::vector<float> y(count);
  e = cudaMemcpy(y.data(), n->y, count * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "proposer scores");
  // arg-max over the single-pass configs the autotuner would try on this
  // shape (ties keep the lower index)
  int best = -1;
  for (int i = 0; i < count; ++i)
    if (autotune_config_runs(ctx, M, N, K, dtype, cfgs[i]) && (best < 0 || y[i] > y[best])) best = i;
  if (best < 0) return fail(TP_ERR_UNSUPPORTED, "no config of the space runs on this shape");
  const bool in_range = M <= 16384 && N <= 16384 && K <= 16384;
  if (score) *score = y[best];
  if (y[best] >= min_score && in_range) {
    *out = cfgs[best];
    if (used_fallback) *used_fallback = 0;
    return TP_OK;
  }
  if (used_fallback) *used_fallback = 1;
  int32_t found = 0;
  s = tp_autotune_lookup(ctx, M, N, K, dtype, 0, out, &found);
  if (s != TP_OK || found) return s;
  return tp_autotune(ctx, M, N, K, dtype, 0, 0, out, nullptr, nullptr);
}

}  // extern "C"

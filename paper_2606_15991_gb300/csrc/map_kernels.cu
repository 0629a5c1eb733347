// Element-wise map kernels: one tile program per output tile (plain
// partition, §3.4) or persistent programs walking a bounded sequence of tiles
// (mapped partition, §3.6). The rank-1 path moves 16 bytes per load/store
// (4 fp32 or 8 bf16) with streaming cache hints; other tilings move the rows
// of a tile as runs of 16-byte slots; tensors whose alignments differ take a
// scalar path. Each program stores only inside its tile.
#include <cuda_bf16.h>

#include "tile_claim.cuh"
#include "tp_internal.h"

namespace tp {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxThreads = 1024;  // of a block whose threads are dealt to tiles in groups (rank-1 vector path)
constexpr int kSegUnroll = 2;      // 16-byte slots in flight per thread of the segment path
constexpr int kSegRounds = 4;      // and its rounds over a tile, when there are tiles enough

struct MapArgs {
  void* out;
  const void* x;
  const void* y;
  float alpha;
  int32_t kind;      // tp_map_kind
  int64_t n;         // elements of the output
  int64_t ntiles;
  int64_t tile;      // rank-1 tile length
  unsigned* queue;   // TP_MAP_QUEUE counter
  uint32_t* counts;  // write-count instrumentation (optional)
  int32_t* owner;
  int64_t shape[3];  // general path, padded to rank 3 (leading 1s)
  int64_t tshape[3];
  int64_t grid[3];
  int32_t group;         // threads per tile (a power of two from 32 to the block's size)
  int32_t mis;           // elements from each base pointer down to a 16-byte boundary (segment path)
  uint32_t* claims;      // checked launch: tile-claim bitmap (null = release)
  unsigned* claim_done;  // checked launch: finished-CTA counter
  int* err;              // the operation's error word
};

// 2^a by the hardware base-2 exponential (flush-to-zero).
__device__ __forceinline__ float ex2_approx(float a) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

// gelu_tanh(x) = 0.5 x (1 + tanh(u)), u = sqrt(2/pi) (x + 0.044715 x^3),
// evaluated as x / (1 + exp(-2u)) (0.5 (1 + tanh u) = 1 / (1 + exp(-2u))),
// with exp(-2u) = 2^t, t = -2 log2(e) u = x (c0 + c1 x^2): one polynomial,
// one base-2 exponential, one fast division. t is capped at 125 so 1 + 2^t
// stays below 2^126, the range where the fast division is defined; the
// result there is ~0.
__device__ __forceinline__ float gelu_tanh(float x) {
  const float c0 = -2.f * 1.4426950408889634f * 0.7978845608028654f;  // -2 log2(e) sqrt(2/pi)
  const float c1 = c0 * 0.044715f;
  const float t = fminf(x * fmaf(c1, x * x, c0), 125.f);
  return __fdividef(x, 1.f + ex2_approx(t));
}

template <int OP>
__device__ __forceinline__ float apply(float x, float y, float c, float alpha) {
  if constexpr (OP == kMapAxpy) return fmaf(alpha, x, y);
  else if constexpr (OP == kMapGeluMul) return gelu_tanh(x) * y;
  else if constexpr (OP == kMapScale) return x * y;
  else return c + x + y;  // kMapAddAccum: c <- c + a + b
}

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Tile -> program schedule of §3.4 / §3.6, walked by groups of `group`
// threads, each on its own tile. Identity: the block's groups are consecutive
// programs (one tile each); strided: the block is one program and its groups
// take every G-th of its tiles; queue: the block dequeues one tile per group
// at a time, the next lot while it works on this one.
// `t` may lie past the last tile for a group of the block's last queue round;
// queue rounds are the block's, the other two loops each group's own.
// QUEUE: the instance serves queue-mapped partitions too.
template <bool GROUPED, bool QUEUE = true>
struct Schedule {
  int64_t t;      // this group's tile
  int tid;        // the thread's index in its group
  int nthr;       // threads of a group
  int grp, G;     // the group's index in the block, and their number
  unsigned ahead; // queue: the next lot (thread 0)
  int round;
  __device__ __forceinline__ bool first(const MapArgs& a, int64_t* slot) {
    if constexpr (GROUPED) {
      nthr = a.group;
      tid = (int)threadIdx.x & (nthr - 1);
      G = (int)blockDim.x / nthr;
      grp = (int)threadIdx.x / nthr;
    } else {
      nthr = kThreads;
      tid = (int)threadIdx.x;
      G = 1;
      grp = 0;
    }
    if (QUEUE && a.kind == TP_MAP_QUEUE) {
      round = 0;
      if (threadIdx.x == 0) ahead = atomicAdd(a.queue, (unsigned)G);
      return dequeue(a, slot);
    }
    t = a.kind == TP_MAP_IDENTITY ? (int64_t)blockIdx.x * G + grp : (int64_t)blockIdx.x + (int64_t)grp * gridDim.x;
    return t < a.ntiles;
  }
  __device__ __forceinline__ bool next(const MapArgs& a, int64_t* slot) {
    if (QUEUE && a.kind == TP_MAP_QUEUE) return dequeue(a, slot);
    if (a.kind == TP_MAP_IDENTITY) return false;
    t += (int64_t)G * gridDim.x;
    return t < a.ntiles;
  }
  // the two slots take turns, so one barrier a round is enough; a block asks
  // for no more once it has seen the end of the queue
  __device__ __forceinline__ bool dequeue(const MapArgs& a, int64_t* slot) {
    if (threadIdx.x == 0) slot[round & 1] = (int64_t)ahead;
    __syncthreads();
    const int64_t base = slot[round & 1];
    ++round;
    t = base + grp;
    if (base >= a.ntiles) return false;
    if (threadIdx.x == 0) ahead = atomicAdd(a.queue, (unsigned)G);
    return true;
  }
  // the tile program that runs this group's tile
  __device__ __forceinline__ int32_t program(const MapArgs& a) const {
    return a.kind == TP_MAP_IDENTITY ? (int32_t)t : (int32_t)blockIdx.x;
  }
};

template <bool COUNT>
__device__ __forceinline__ void count_write(const MapArgs& a, int32_t program, int64_t i) {
  if constexpr (COUNT) {
    atomicAdd(a.counts + i, 1u);
    a.owner[i] = program;
  }
}

// Checked launch: before storing tile t the program validates it against
// the map (a tile of the grid, and for a strided map one of this program's
// slots) and claims it; a refused claim skips the tile. Block-uniform.
template <bool kCheck = true>
__device__ __forceinline__ bool claim_map_tile(const MapArgs& a, int64_t t) {
  if constexpr (!kCheck) return true;
  if (a.claims == nullptr) return true;
  int won = 0;
  if (threadIdx.x == 0) {
    bool on_map = t >= 0 && t < a.ntiles;
    if (a.kind == TP_MAP_IDENTITY) on_map = on_map && t == (int64_t)blockIdx.x;
    if (a.kind == TP_MAP_STRIDED) on_map = on_map && (t - (int64_t)blockIdx.x) % gridDim.x == 0;
    if (!on_map) record_device_error(a.err, kDevRace);
    won = on_map && claim_tile(a.claims, t, a.err) ? 1 : 0;
  }
  return __syncthreads_or(won) != 0;
}

template <bool kCheck = true>
__device__ __forceinline__ void finish_map_claims(const MapArgs& a) {
  if constexpr (kCheck) {
    if (a.claims != nullptr) claims_finish(a.claims, a.ntiles, a.claim_done, gridDim.x);
  }
}

template <typename T> struct Vec;
template <> struct Vec<float> { using V = float4; static constexpr int N = 4; };
template <> struct Vec<__nv_bfloat16> { using V = uint4; static constexpr int N = 8; };

template <typename T>
__device__ __forceinline__ void unpack(const typename Vec<T>::V& v, float* f) {
  if constexpr (sizeof(T) == 4) {
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
  } else {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 t = __bfloat1622float2(h[i]);
      f[2 * i] = t.x;
      f[2 * i + 1] = t.y;
    }
  }
}

template <typename T>
__device__ __forceinline__ typename Vec<T>::V pack(const float* f) {
  typename Vec<T>::V v;
  if constexpr (sizeof(T) == 4) {
    v.x = f[0]; v.y = f[1]; v.z = f[2]; v.w = f[3];
  } else {
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  }
  return v;
}

// Rank-1 path: tile length is a multiple of the vector width and all three
// pointers are 16-byte aligned, so every tile starts on a vector boundary.
// Programmatic dependent launch: map launches carry the programmatic
// stream-serialization attribute, so the next launch on the stream may be
// scheduled while this one runs. Each map kernel first waits until the grid
// it depends on has completed and its memory is visible (a no-op when it was
// not launched early), then lets its own dependents be scheduled.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Vectors in flight per thread: 4 (f32) or 2 (bf16) of one tile per block;
// 2 where more threads of a block share them out.
template <typename T, bool GROUPED>
constexpr int vec_unroll() {
  return GROUPED || Vec<T>::N == 8 ? 2 : 4;
}

// Blocks per SM that the registers must leave room for: as many as the loads
// in flight allow without spilling (bf16 32 registers, f32 40; 40 and 64 where
// the output is read too; 64 with instrumentation and in the blocks of 1024).
template <int OP, typename T>
constexpr int vec_min_blocks(bool instrumented, bool grouped) {
  return grouped ? 1 : instrumented ? 4 : Vec<T>::N == 8 ? (OP == kMapAddAccum ? 6 : 8) : (OP == kMapAddAccum ? 4 : 6);
}

// A tile is the work of one group of threads (Schedule). GROUPED: groups and
// block sized to the tiles and the programs (group_shape); otherwise one block
// of 256 threads per tile, whose strides are constants.
template <int OP, typename T, bool COUNT, bool CHECKED, bool GROUPED>
__global__ void __launch_bounds__(GROUPED ? kMaxThreads : kThreads,
                                  vec_min_blocks<OP, T>(COUNT || CHECKED, GROUPED))
    map_vec_kernel(const __grid_constant__ MapArgs a) {
  using V = typename Vec<T>::V;
  constexpr int W = Vec<T>::N;
  constexpr int U = vec_unroll<T, GROUPED>();  // vectors per thread per round
  __shared__ int64_t slot[2];
  pdl_enter();
  T* __restrict__ out = static_cast<T*>(a.out);
  const T* __restrict__ x = static_cast<const T*>(a.x);
  const T* __restrict__ y = static_cast<const T*>(a.y);
  Schedule<GROUPED, GROUPED || CHECKED> s;
  for (bool more = s.first(a, slot); more; more = s.next(a, slot)) {
    const int64_t t = s.t;
    if (GROUPED && t >= a.ntiles) continue;
    if (!claim_map_tile<CHECKED>(a, t)) continue;
    const int nthr = GROUPED ? s.nthr : kThreads;
    const int32_t prog = s.program(a);
    const int64_t start = t * a.tile;
    const int64_t len = min(a.tile, a.n - start);
    const int64_t nv = len / W;
    const V* xv = reinterpret_cast<const V*>(x + start);
    const V* yv = reinterpret_cast<const V*>(y + start);
    V* ov = reinterpret_cast<V*>(out + start);
    // output vector w from its inputs
    auto move = [&](const V& xr, const V& yr, const V& cr, int64_t w) {
      float fx[W], fy[W], fc[W], fo[W];
      unpack<T>(xr, fx);
      unpack<T>(yr, fy);
      if constexpr (OP == kMapAddAccum) unpack<T>(cr, fc);
#pragma unroll
      for (int i = 0; i < W; ++i) fo[i] = apply<OP>(fx[i], fy[i], OP == kMapAddAccum ? fc[i] : 0.f, a.alpha);
      __stcs(ov + w, pack<T>(fo));
      if constexpr (COUNT) {
#pragma unroll
        for (int i = 0; i < W; ++i) count_write<COUNT>(a, prog, start + w * W + i);
      }
    };
    if constexpr (GROUPED) {
      // up to U vectors per thread and round, all loads first
#pragma unroll 1
      for (int64_t v = s.tid; v < nv; v += U * nthr) {
        V xr[U], yr[U], cr[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int64_t w = v + u * nthr;
          if (w < nv) {
            xr[u] = __ldcs(xv + w);
            yr[u] = __ldcs(yv + w);
            if constexpr (OP == kMapAddAccum) cr[u] = ov[w];
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int64_t w = v + u * nthr;
          if (w < nv) move(xr[u], yr[u], cr[u], w);
        }
      }
    } else {
      int64_t v = threadIdx.x;
      for (; v + (U - 1) * kThreads < nv; v += U * kThreads) {
        V xr[U], yr[U], cr[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          xr[u] = __ldcs(xv + v + u * kThreads);
          yr[u] = __ldcs(yv + v + u * kThreads);
          if constexpr (OP == kMapAddAccum) cr[u] = ov[v + u * kThreads];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) move(xr[u], yr[u], cr[u], v + u * kThreads);
      }
      for (; v < nv; v += kThreads) {
        V cr = {};
        if constexpr (OP == kMapAddAccum) cr = ov[v];
        move(__ldcs(xv + v), __ldcs(yv + v), cr, v);
      }
    }
    // ragged tail of the last tile (fewer than W elements)
    for (int64_t i = nv * W + s.tid; i < len; i += nthr) {
      const int64_t g = start + i;
      float c = OP == kMapAddAccum ? to_f<T>(out[g]) : 0.f;
      out[g] = from_f<T>(apply<OP>(to_f<T>(x[g]), to_f<T>(y[g]), c, a.alpha));
      count_write<COUNT>(a, prog, g);
    }
  }
  finish_map_claims<CHECKED>(a);
}

// n / d and n % d of non-negative values, in 32 bits where both fit (a 64-bit
// division costs hundreds of cycles).
__device__ __forceinline__ void divmod(int64_t n, int64_t d, int64_t* q, int64_t* r) {
  if (((n | d) >> 32) == 0) {
    const uint32_t q32 = (uint32_t)n / (uint32_t)d;
    *q = q32;
    *r = (uint32_t)n - q32 * (uint32_t)d;
  } else {
    *q = n / d;
    *r = n - *q * d;
  }
}

// Tiles made of row segments: any rank-1..3 partition whose three tensors are
// equally aligned (`mis` = elements from each base pointer down to a 16-byte
// boundary). A tile row is one contiguous run of elements, the same run in
// every tensor, so it is covered by 16-byte slots on the address grid. The
// inputs of a slot are loaded as one vector each, also where the run only
// touches it (its other elements are the neighbouring program's inputs, which
// nothing writes); what is stored are the run's elements, as one vector or one
// by one, so a program stores only inside its tile. Only a slot that reaches
// past the tensor's own first or last element is read element by element. The
// slots of all rows of the tile are dealt to the tile's threads in one flat
// sequence, so rows shorter than a warp leave no lane idle; a thread's
// (row, slot) advances by a fixed step, without a division per access.
// GROUPED as in map_vec_kernel, which stays for rank-1 tiles of whole
// vectors, where it needs no run arithmetic.
// Bound by HBM where the tile's columns are whole slots: y = gelu_tanh(x) * w
// over 4001 x 9728 bf16 (234 MB) takes 38.2 us in 128 x 256 tiles and 43.6 us
// in 16 x 64 ones; with one block per tile, and the run's end slots element by
// element, 37.6 and 100 us (one element per access with two 64-bit divisions
// each: 267 us). With 9729 columns every row has end slots, whose stores bound
// it: 45.6 and 59.5 us, 66.9 and 179 us before. Rank 1, 2^26 f32 elements in
// tiles of 1001 / 100: 122 / 191 us, 295 / 678 before.
template <int OP, typename T, bool COUNT, bool GROUPED>
__global__ void __launch_bounds__(kThreads) map_segment_kernel(const __grid_constant__ MapArgs a) {
  using V = typename Vec<T>::V;
  constexpr int W = Vec<T>::N;
  constexpr int U = kSegUnroll;  // slots in flight per thread
  __shared__ int64_t slot[2];
  pdl_enter();
  T* out = static_cast<T*>(a.out);
  const T* x = static_cast<const T*>(a.x);
  const T* y = static_cast<const T*>(a.y);
  Schedule<GROUPED> s;
  for (bool more = s.first(a, slot); more; more = s.next(a, slot)) {
    const int64_t t = s.t;
    if (GROUPED && t >= a.ntiles) continue;
    if (!claim_map_tile<!GROUPED>(a, t)) continue;
    const uint32_t nthr = GROUPED ? (uint32_t)s.nthr : (uint32_t)kThreads;
    const int32_t prog = s.program(a);
    int64_t t0, t1, t2, q;
    divmod(t, a.grid[2], &q, &t2);
    divmod(q, a.grid[1], &t0, &t1);
    // the tile clipped to the tensor: e0 x e1 rows of e2 elements
    const int64_t b0 = t0 * a.tshape[0], b1 = t1 * a.tshape[1], b2 = t2 * a.tshape[2];
    const int32_t e0 = (int32_t)min(a.tshape[0], a.shape[0] - b0), e1 = (int32_t)min(a.tshape[1], a.shape[1] - b1);
    const int32_t e2 = (int32_t)min(a.tshape[2], a.shape[2] - b2);
    const int64_t origin = (b0 * a.shape[1] + b1) * a.shape[2] + b2;
    // slots a row may touch; every row starts at the same place of a slot
    // when the row pitch is whole slots
    const int32_t ph0 = (int32_t)((uint64_t)(origin + a.mis) % W);
    const uint32_t per = (uint32_t)(a.shape[2] % W == 0 ? ph0 + e2 + W - 1 : e2 + 2 * W - 2) / W;
    const uint32_t rows = (uint32_t)e0 * (uint32_t)e1;
    const uint32_t dr = nthr / per, dc = nthr % per;
    uint32_t r = (uint32_t)s.tid / per, c = (uint32_t)s.tid % per;
    while (r < rows) {
      int64_t at[U];   // the slot's first element (may lie before the run's)
      int32_t i0[U], i1[U];  // its elements [i0, i1) are the run's; none when i0 >= i1
      bool vec[U];     // the slot lies inside the tensor: loaded as vectors
      V xr[U], yr[U], cr[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        i0[u] = i1[u] = 0;
        vec[u] = false;
        if (r < rows) {
          const uint32_t r0 = e0 > 1 ? r / (uint32_t)e1 : 0u;
          const uint32_t r1 = r - r0 * (uint32_t)e1;
          const int64_t g = origin + ((int64_t)r0 * a.shape[1] + r1) * a.shape[2];  // the run's first element
          const int32_t lo = (int32_t)c * W - (int32_t)((uint64_t)(g + a.mis) % W);
          at[u] = g + lo;
          i0[u] = max(-lo, 0);
          i1[u] = min(W, e2 - lo);
          vec[u] = i0[u] < i1[u] && at[u] >= 0 && at[u] + W <= a.n;
          if (vec[u]) {
            xr[u] = __ldcs(reinterpret_cast<const V*>(x + at[u]));
            yr[u] = __ldcs(reinterpret_cast<const V*>(y + at[u]));
            if constexpr (OP == kMapAddAccum)
              if (i0[u] == 0 && i1[u] == W) cr[u] = *reinterpret_cast<const V*>(out + at[u]);
          }
        }
        r += dr;
        c += dc;
        if (c >= per) {
          c -= per;
          ++r;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (vec[u]) {
          float fx[W], fy[W], fc[W], fo[W];
          const bool whole = i0[u] == 0 && i1[u] == W;
          unpack<T>(xr[u], fx);
          unpack<T>(yr[u], fy);
          if constexpr (OP == kMapAddAccum) {
            // of the output only the run's own elements are read: the others
            // may be being written by their program
            if (whole) unpack<T>(cr[u], fc);
            else {
#pragma unroll
              for (int i = 0; i < W; ++i) fc[i] = i >= i0[u] && i < i1[u] ? to_f<T>(out[at[u] + i]) : 0.f;
            }
          }
#pragma unroll
          for (int i = 0; i < W; ++i) fo[i] = apply<OP>(fx[i], fy[i], OP == kMapAddAccum ? fc[i] : 0.f, a.alpha);
          if (whole) __stcs(reinterpret_cast<V*>(out + at[u]), pack<T>(fo));
          else {
#pragma unroll
            for (int i = 0; i < W; ++i)
              if (i >= i0[u] && i < i1[u]) out[at[u] + i] = from_f<T>(fo[i]);
          }
          if constexpr (COUNT)
            for (int32_t i = i0[u]; i < i1[u]; ++i) count_write<COUNT>(a, prog, at[u] + i);
        } else {
          for (int32_t i = i0[u]; i < i1[u]; ++i) {
            const int64_t g = at[u] + i;
            const float cv = OP == kMapAddAccum ? to_f<T>(out[g]) : 0.f;
            out[g] = from_f<T>(apply<OP>(to_f<T>(x[g]), to_f<T>(y[g]), cv, a.alpha));
            count_write<COUNT>(a, prog, g);
          }
        }
      }
    }
  }
  finish_map_claims<!GROUPED>(a);
}

// General path: any rank-1..3 partition of a contiguous output, scalar
// accesses, elements of the tile outside the tensor are skipped. Taken only
// when the three tensors' base pointers differ in their offset from a 16-byte
// boundary, so that no 16-byte access fits all of them.
template <int OP, typename T, bool COUNT>
__global__ void __launch_bounds__(kThreads) map_generic_kernel(const __grid_constant__ MapArgs a) {
  __shared__ int64_t slot[2];
  pdl_enter();
  T* out = static_cast<T*>(a.out);
  const T* x = static_cast<const T*>(a.x);
  const T* y = static_cast<const T*>(a.y);
  const int64_t tile_elems = a.tshape[0] * a.tshape[1] * a.tshape[2];
  Schedule<false> s;
  for (bool more = s.first(a, slot); more; more = s.next(a, slot)) {
    const int64_t t = s.t;
    if (!claim_map_tile(a, t)) continue;
    const int64_t t2 = t % a.grid[2];
    const int64_t t1 = (t / a.grid[2]) % a.grid[1];
    const int64_t t0 = t / (a.grid[2] * a.grid[1]);
    for (int64_t e = threadIdx.x; e < tile_elems; e += kThreads) {
      const int64_t l2 = e % a.tshape[2];
      const int64_t l1 = (e / a.tshape[2]) % a.tshape[1];
      const int64_t l0 = e / (a.tshape[2] * a.tshape[1]);
      const int64_t g0 = t0 * a.tshape[0] + l0, g1 = t1 * a.tshape[1] + l1, g2 = t2 * a.tshape[2] + l2;
      if (g0 >= a.shape[0] || g1 >= a.shape[1] || g2 >= a.shape[2]) continue;
      const int64_t g = (g0 * a.shape[1] + g1) * a.shape[2] + g2;
      float c = OP == kMapAddAccum ? to_f<T>(out[g]) : 0.f;
      out[g] = from_f<T>(apply<OP>(to_f<T>(x[g]), to_f<T>(y[g]), c, a.alpha));
      count_write<COUNT>(a, s.program(a), g);
    }
  }
  finish_map_claims(a);
}

template <typename K>
cudaError_t launch_pdl(K kernel, const MapArgs& a, int64_t grid, int threads, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// How a map's tiles are accessed, fastest first.
enum Path : int {
  kVector,   // rank 1, tiles of whole vectors from a 16-byte boundary on
  kSegment,  // row segments on the 16-byte grid
  kScalar,   // one element at a time
};

// The path for `a`. The segment path counts a tile's rows and slots in 32
// bits, so tiles of 2^30 elements or more stay on the scalar path.
template <typename T>
Path map_path(MapArgs* a, bool rank1) {
  constexpr int W = Vec<T>::N;
  auto off = [](const void* p) { return reinterpret_cast<uintptr_t>(p) & 15u; };
  const uintptr_t m = off(a->out);
  if (off(a->x) != m || off(a->y) != m || m % sizeof(T)) return kScalar;
  if (rank1 && m == 0 && a->tile % W == 0) return kVector;
  int64_t elems = 1;
  for (int i = 0; i < 3; ++i) {
    const int64_t e = a->tshape[i] < a->shape[i] ? a->tshape[i] : a->shape[i];
    if (e >= (int64_t(1) << 30) / elems) return kScalar;
    elems *= e;
  }
  a->mis = (int32_t)(m / sizeof(T));
  return kSegment;
}

// Threads per tile, threads per block and blocks of a launch.
struct Shape {
  int group = kThreads, threads = kThreads;
  int64_t grid = 0;
  bool grouped() const { return group != kThreads || threads != kThreads; }
};

// A tile of `items` vectors, of which a thread has `unroll` in flight, gets as
// many threads as take it in `rounds` rounds (at least a warp), and a block as
// many groups as keep the chip's threads in use:
//  - identity: consecutive programs share a block of 256 threads, as long as
//    that leaves two blocks per SM;
//  - strided and queue: the blocks are the programs, whose number the caller
//    chose; with fewer than fill the SMs a block takes up to max_threads and
//    works on several of its tiles at once, as far as it has several (queue:
//    twice as many, so that the dynamic order still balances).
// More than one round pays only where there are tiles enough for every thread
// slot of the chip twice over; with fewer a tile is taken in one.
// The checked launch's claims are a block's, not a group's: one tile at a time.
// Measured on z = a x + y over 2^26 elements, one block of 256 threads per
// program and tile -> this: bf16 tiles of 1000, identity / strided over 608
// programs / queue, 71.4 / 110 / 150 -> 62.9 / 62.0 / 64.4 us; tiles of 2048
// from the queue 86.1 -> 63.3 us; f32 tiles of 1000 122 / 140 / 164 -> 116 /
// 128 / 119 us. Rounds: 16 x 64 bf16 tiles of 4001 x 9728 in one round 75.1
// us, in up to four 43.6 (a tile's index arithmetic is then spread over more
// of its elements).
Shape group_shape(const MapArgs& a, int64_t programs, int64_t items, int unroll, int rounds, int sms, int max_threads) {
  constexpr int64_t kSmThreads = 1024;  // resident threads per SM at 64 registers
  Shape s;
  s.grid = programs;
  if (a.claims) return s;
  const bool identity = a.kind == TP_MAP_IDENTITY;
  int threads = kThreads;
  while (threads < max_threads && programs * threads * 2 <= sms * kSmThreads) threads *= 2;
  int group = 32;
  while (group < threads && (int64_t)group * unroll < items) group *= 2;
  while (group > 32 && (int64_t)group * unroll * rounds >= 2 * items && a.ntiles * group >= 4 * sms * kSmThreads)
    group /= 2;
  int groups = threads / group;
  if (identity) {
    while (groups > 1 && a.ntiles / groups < 2 * (int64_t)sms) groups /= 2;
    s.grid = (a.ntiles + groups - 1) / groups;
  } else {
    const int64_t lots = a.kind == TP_MAP_QUEUE ? a.ntiles / (2 * programs) : (a.ntiles + programs - 1) / programs;
    while (groups > 1 && groups > lots) groups /= 2;
  }
  s.group = group;
  s.threads = group * groups;
  return s;
}

template <int OP, typename T>
cudaError_t launch_typed(MapArgs a, Path path, bool count, int64_t grid, int sms, cudaStream_t st) {
  constexpr int W = Vec<T>::N;
  if (path == kSegment) {
    const int64_t e2 = std::min(a.tshape[2], a.shape[2]);
    const int64_t rows = std::min(a.tshape[0], a.shape[0]) * std::min(a.tshape[1], a.shape[1]);
    const bool whole = a.mis == 0 && a.shape[2] % W == 0 && a.tshape[2] % W == 0;  // no slot is shared by two tiles
    const int64_t slots = rows * ((e2 + (whole ? W - 1 : 2 * W - 2)) / W);  // a row's at most
    const Shape s = group_shape(a, grid, slots, kSegUnroll, kSegRounds, sms, kThreads);
    a.group = s.group;
    if (s.grouped()) return count ? launch_pdl(map_segment_kernel<OP, T, true, true>, a, s.grid, s.threads, st)
                                  : launch_pdl(map_segment_kernel<OP, T, false, true>, a, s.grid, s.threads, st);
    return count ? launch_pdl(map_segment_kernel<OP, T, true, false>, a, s.grid, s.threads, st)
                 : launch_pdl(map_segment_kernel<OP, T, false, false>, a, s.grid, s.threads, st);
  }
  if (path == kVector) {
    constexpr int U = vec_unroll<T, true>();
    const int64_t vectors = std::min(a.tile, a.n) / W;
    Shape s;
    s.grid = grid;
    // tiles that give every thread of a plain block a vector stay there (bf16
    // tiles of 2048: 58.8 us, 61.4 in groups of 128 threads)
    if (a.kind != TP_MAP_IDENTITY || vectors < kThreads) s = group_shape(a, grid, vectors, U, 1, sms, kMaxThreads);
    a.group = s.group;
    if (a.claims) return count ? launch_pdl(map_vec_kernel<OP, T, true, true, false>, a, s.grid, s.threads, st)
                               : launch_pdl(map_vec_kernel<OP, T, false, true, false>, a, s.grid, s.threads, st);
    if (s.grouped() || a.kind == TP_MAP_QUEUE)
      return count ? launch_pdl(map_vec_kernel<OP, T, true, false, true>, a, s.grid, s.threads, st)
                   : launch_pdl(map_vec_kernel<OP, T, false, false, true>, a, s.grid, s.threads, st);
    return count ? launch_pdl(map_vec_kernel<OP, T, true, false, false>, a, s.grid, s.threads, st)
                 : launch_pdl(map_vec_kernel<OP, T, false, false, false>, a, s.grid, s.threads, st);
  }
  return count ? launch_pdl(map_generic_kernel<OP, T, true>, a, grid, kThreads, st)
               : launch_pdl(map_generic_kernel<OP, T, false>, a, grid, kThreads, st);
}

template <typename T>
cudaError_t launch_op(int op, MapArgs a, bool rank1, bool count, int64_t grid, int sms, cudaStream_t st) {
  const Path path = map_path<T>(&a, rank1);
  switch (op) {
    case kMapAxpy: return launch_typed<kMapAxpy, T>(a, path, count, grid, sms, st);
    case kMapGeluMul: return launch_typed<kMapGeluMul, T>(a, path, count, grid, sms, st);
    case kMapScale: return launch_typed<kMapScale, T>(a, path, count, grid, sms, st);
    default: return launch_typed<kMapAddAccum, T>(a, path, count, grid, sms, st);
  }
}

}  // namespace

tp_status launch_map(tp_ctx* ctx, tp_partition* out, int op, float alpha, const tp_tensor* x,
                     const tp_tensor* y, const tp_exec* ex, cudaStream_t stream, unsigned* queue, int* err) {
  MapArgs a{};
  a.out = out->t.ptr;
  a.x = x->ptr;
  a.y = y->ptr;
  a.alpha = alpha;
  a.kind = out->kind;
  a.n = numel(out->t);
  a.ntiles = out->num_tiles;
  a.tile = out->tile[0];
  a.queue = queue;
  a.counts = ex->write_counts;
  a.owner = ex->write_owner;
  if ((a.counts == nullptr) != (a.owner == nullptr))
    return fail(TP_ERR_INVALID, "write_counts and write_owner must be given together");
  if (ex->flags & TP_EXEC_CHECKED) {
    tp_status cs = claims_for(ctx, out->num_tiles, &a.claims, &a.claim_done);
    if (cs != TP_OK) return cs;
    a.err = err;
  }
  const int pad = 3 - out->rank;
  for (int i = 0; i < 3; ++i) {
    a.shape[i] = i < pad ? 1 : out->shape[i - pad];
    a.tshape[i] = i < pad ? 1 : out->tile[i - pad];
    a.grid[i] = i < pad ? 1 : out->grid[i - pad];
  }
  if (a.n == 0 || a.ntiles == 0) return TP_OK;
  const int64_t grid = out->kind == TP_MAP_IDENTITY ? out->num_tiles : out->num_programs;
  if (grid > 0x7fffffff) return fail(TP_ERR_UNSUPPORTED, "more than 2^31-1 tile programs");
  const bool count = a.counts != nullptr;
  cudaError_t e = out->t.dtype == TP_F32 ? launch_op<float>(op, a, out->rank == 1, count, grid, ctx->sm_count, stream)
                                         : launch_op<__nv_bfloat16>(op, a, out->rank == 1, count, grid, ctx->sm_count, stream);
  if (e != cudaSuccess) return cuda_fail(e, "map kernel launch");
  return TP_OK;
}

}  // namespace tp

// ---------------------------------------------------------------------------
// Allocation-free queue-mapped axpy (tp_map_axpy_queue_noalloc).
//
// Its only scratch is the device queue's tile counter. It lives in the static
// device array below, so the entry point needs no context and allocates
// nothing; every GPU that loads this library holds the array until exit.
#include <mutex>

namespace tp {
namespace {

constexpr int64_t kNoallocMaxTiles = int64_t(1) << 31;  // the 32-bit counter never wraps
constexpr int kNoallocMaxDevices = 64;

// One 32-bit tile counter (4 bytes used of a 256-byte-aligned array).
static __device__ __align__(256) unsigned int g_noalloc_tile_queue[1];

// Device address of g_noalloc_tile_queue per device, looked up once per
// device with that device current. In host code the array's name is only a
// host-side stand-in; only this looked-up address may be given to a kernel.
void* g_noalloc_queue_addr[kNoallocMaxDevices] = {};
int g_noalloc_sms[kNoallocMaxDevices] = {};
std::mutex g_noalloc_mu;

// Set-up of a device, on the entry point's first call there: the scratch
// array's device address, and every kernel instance the entry point can
// launch loaded now (with lazy module loading a kernel is otherwise loaded
// at its first launch), so later calls only enqueue work.
tp_status noalloc_queue_address(void** out, int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kNoallocMaxDevices) return fail(TP_ERR_UNSUPPORTED, "device index above 63");
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_queue_addr[dev]) {
    const void* kernels[] = {reinterpret_cast<const void*>(map_vec_kernel<kMapAxpy, float, false, false, false>),
                             reinterpret_cast<const void*>(map_vec_kernel<kMapAxpy, float, false, false, true>),
                             reinterpret_cast<const void*>(map_vec_kernel<kMapAxpy, __nv_bfloat16, false, false, false>),
                             reinterpret_cast<const void*>(map_vec_kernel<kMapAxpy, __nv_bfloat16, false, false, true>),
                             reinterpret_cast<const void*>(map_segment_kernel<kMapAxpy, float, false, false>),
                             reinterpret_cast<const void*>(map_segment_kernel<kMapAxpy, float, false, true>),
                             reinterpret_cast<const void*>(map_segment_kernel<kMapAxpy, __nv_bfloat16, false, false>),
                             reinterpret_cast<const void*>(map_segment_kernel<kMapAxpy, __nv_bfloat16, false, true>),
                             reinterpret_cast<const void*>(map_generic_kernel<kMapAxpy, float, false>),
                             reinterpret_cast<const void*>(map_generic_kernel<kMapAxpy, __nv_bfloat16, false>)};
    for (const void* k : kernels) {
      cudaFuncAttributes fa;
      e = cudaFuncGetAttributes(&fa, k);
      if (e != cudaSuccess) return cuda_fail(e, "loading the queue-mapped axpy kernels");
    }
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_tile_queue);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress of the tile-queue scratch");
    e = cudaDeviceGetAttribute(&g_noalloc_sms[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    g_noalloc_queue_addr[dev] = p;
  }
  *out = g_noalloc_queue_addr[dev];
  *sms = g_noalloc_sms[dev];
  return TP_OK;
}

}  // namespace
}  // namespace tp

extern "C" tp_status tp_map_axpy_queue_noalloc(void* z, const void* x, const void* y, int32_t dtype, int64_t n,
                                               int64_t tile, int32_t num_programs, float alpha, void* stream) {
  using namespace tp;
  if (dtype != TP_F32 && dtype != TP_BF16) return fail(TP_ERR_UNSUPPORTED, "dtype must be TP_F32 or TP_BF16");
  if (n < 0 || tile < 1) return fail(TP_ERR_INVALID, "need n >= 0 and tile >= 1");
  const int64_t ntiles = (n + tile - 1) / tile;
  if (ntiles > kNoallocMaxTiles)
    return fail(TP_ERR_INVALID, "more than 2^31 tiles: the allocation-free tile queue holds a 32-bit counter");
  if (n == 0) return TP_OK;
  if (!z || !x || !y) return fail(TP_ERR_INVALID, "null pointer");
  if (num_programs < 1 || num_programs > ntiles)
    return fail(TP_ERR_INVALID, "num_programs must be 1..number of tiles");
  const size_t es = dtype_size(dtype);
  const uintptr_t z0 = reinterpret_cast<uintptr_t>(z), z1 = z0 + (uintptr_t)n * es;
  for (const void* in : {x, y}) {
    const uintptr_t i0 = reinterpret_cast<uintptr_t>(in), i1 = i0 + (uintptr_t)n * es;
    if (i0 < z1 && z0 < i1) return fail(TP_ERR_ALIAS, "an input overlaps the output");
  }
  void* queue = nullptr;
  int sms = 0;
  tp_status s = noalloc_queue_address(&queue, &sms);
  if (s != TP_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(unsigned int), st);  // the queue starts at slot 0
  if (e != cudaSuccess) return cuda_fail(e, "clearing the tile-queue scratch");
  MapArgs a{};
  a.out = z;
  a.x = x;
  a.y = y;
  a.alpha = alpha;
  a.kind = TP_MAP_QUEUE;
  a.n = n;
  a.ntiles = ntiles;
  a.tile = tile;
  a.queue = static_cast<unsigned*>(queue);
  for (int i = 0; i < 3; ++i) {
    a.shape[i] = i < 2 ? 1 : n;
    a.tshape[i] = i < 2 ? 1 : tile;
    a.grid[i] = i < 2 ? 1 : ntiles;
  }
  e = dtype == TP_F32 ? launch_op<float>(kMapAxpy, a, true, false, num_programs, sms, st)
                      : launch_op<__nv_bfloat16>(kMapAxpy, a, true, false, num_programs, sms, st);
  if (e != cudaSuccess) return cuda_fail(e, "map kernel launch");
  return TP_OK;
}

// Deterministic one-launch global sums in FP64: warp shuffles, then shared memory, one
// partial per block, and the last block to finish (atomic ticket) adds the partials in
// a fixed order.  The result therefore does not depend on block scheduling.
#pragma once
#include <tuple>
#include <utility>

#include "pfmp_internal.cuh"

namespace pfmp {

// Kernels that follow each other on a stream without the launch gap between them: a kernel
// launched with launch_chained may become resident while its predecessor drains, and
// chain_enter, its first statement, waits until the predecessor has completed (its writes
// are then visible) after letting its own successor come up in the same way.  A successor
// launched in the ordinary way waits for completion as always.  Such a kernel is resident
// while its predecessor still writes, so it must not read what a predecessor writes through
// the read-only path (__ldg, const __restrict__ parameters: data that stay the same for as
// long as the kernel lives, which the compiler may also load above the wait): it takes ld_live,
// or plain loads of pointers without those qualifiers.  The links and clover blocks of an
// operator are exempt: clover_build waits for the stream before any kernel may use them.
// K at 4^3x8 (four launches of k_hop_pair) 16.4 -> 10.7 us.  The FP64 stencils and force
// contractions gain nothing (the FP64 force at 6x10x14x18 +2%), nor do the one-thread-per-site
// stencils (K at 32^3x64 +2%): those are launched in the ordinary way.  Inside a CUDA graph
// these edges cost more than they hide (mixed solve at 16^3x32 6.1 -> 6.9 ms), so a captured or
// recorded launch is an ordinary one; kernels that run on both sides are told (chained) where they can
// be without a cost.
__device__ __forceinline__ void chain_enter() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void chain_enter(bool chained) {
  if (chained) chain_enter();
}
// An ordinary coherent load, written so that it stays below chain_enter (volatile assembly keeps
// its order) without holding back the loads after it.
__device__ __forceinline__ float ld_live(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ld_live(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_live(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_live(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_live(const double2* p) {
  double2 v;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
// A chunk of launches as a CUDA graph, node after node: while a LaunchRecord of this thread is
// current, launch_plain and launch_chained add to its graph instead of launching.  A stream
// capture makes the same graph, but a cudaDeviceSynchronize in any other thread fails while a
// stream captures, and the capture with it.
struct LaunchRecord {
  cudaGraph_t graph = nullptr;
  cudaGraphNode_t last = nullptr;
  long long kernels = 0;
  static LaunchRecord*& current() {
    static thread_local LaunchRecord* r = nullptr;
    return r;
  }
  LaunchRecord() {
    PFMP_CUDA(cudaGraphCreate(&graph, 0));
    current() = this;
  }
  LaunchRecord(const LaunchRecord&) = delete;
  ~LaunchRecord() {
    current() = nullptr;
    cudaGraphDestroy(graph);
  }
  template <typename... P, size_t... I>
  void add(void (*kernel)(P...), dim3 grid, dim3 block, std::tuple<P...> args, std::index_sequence<I...>) {
    void* at[] = {(void*)&std::get<I>(args)...};
    cudaKernelNodeParams p{};
    p.func = (void*)kernel;
    p.gridDim = grid;
    p.blockDim = block;
    p.kernelParams = at;
    cudaGraphNode_t node;
    PFMP_CUDA(cudaGraphAddKernelNode(&node, graph, &last, last ? 1 : 0, &p));
    last = node;
    ++kernels;
  }
};
template <typename... P, typename... A>
void launch_plain(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args) {
  if (LaunchRecord* r = LaunchRecord::current())
    r->add(kernel, grid, block, std::tuple<P...>(static_cast<P>(args)...), std::index_sequence_for<P...>());
  else
    kernel<<<grid, block, 0, st>>>(static_cast<P>(args)...);
}

// whether launches on st are chained
inline bool chain_launches(cudaStream_t st) {
  if (LaunchRecord::current()) return false;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  PFMP_CUDA(cudaStreamIsCapturing(st, &capture));
  return capture == cudaStreamCaptureStatusNone;
}
template <typename... P, typename... A>
void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args) {
  if (LaunchRecord::current()) return launch_plain(kernel, grid, block, st, args...);
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = chain_launches(st) ? 1 : 0;
  PFMP_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
}

struct ReduceBuf {
  double* partials;   // [max_blocks * kMaxSums]
  unsigned* counter;  // one ticket counter, left at 0 after each use
};
constexpr int kMaxSums = 4;
constexpr int kMaxReduceBlocks = 65536;

// A thread's sum of FP32 values without the FP64 pipe, turned into FP64 once: an FP64 add and
// a conversion per value cost 16 cycles of the SM's FP64 pipe per warp each (22 us of a 77 us
// stencil with a norm at 24^3x48), thirteen FP32 operations under half a cycle each.  The sum is an
// unevaluated hi + mid + lo: Knuth's TwoSum adds the value to hi and the error of that to mid,
// and only the error of the second sum is rounded when it is added to lo, a 2^-72 of the
// running sum.  So value() is the sum of the values rounded to FP64 about once, where FP64
// additions in turn round at each (a pair hi + lo would stop at 2^-48).  ok() is false when the
// sum left the range of FP32 or a value was not finite: the caller then adds in FP64.
struct TripleSum {
  float hi = 0.f, mid = 0.f, lo = 0.f;
  // a + b = s + the return value exactly
  static __device__ __forceinline__ float two_sum(float a, float b, float& s) {
    s = __fadd_rn(a, b);
    const float c = __fsub_rn(s, a);
    return __fadd_rn(__fsub_rn(a, __fsub_rn(s, c)), __fsub_rn(b, c));
  }
  __device__ __forceinline__ void add(float v) {
    lo = __fadd_rn(lo, two_sum(mid, two_sum(hi, v, hi), mid));
  }
  __device__ __forceinline__ bool ok() const { return fabsf(hi) < 3e38f; }
  __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};

template <int N>
__device__ __forceinline__ void block_sum(double v[N], double* sh /* [N][32] */) {
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) sh[k * 32 + warp] = v[k];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      double w = lane < nw ? sh[k * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
      v[k] = w;
    }
  }
  __syncthreads();
}

// Adds v[0..N) over the whole grid.  Returns true in exactly one thread (thread 0 of the
// last block), whose out[0..N) then holds the grid totals.  Every thread of every block
// must call this (no early return before it).
template <int N>
__device__ __forceinline__ bool grid_sum(double v[N], ReduceBuf rb, double out[N]) {
  __shared__ double sh[N * 32];
  __shared__ bool last;
  const unsigned nblk = gridDim.x * gridDim.y * gridDim.z;
  const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  block_sum<N>(v, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) rb.partials[(size_t)bid * N + k] = v[k];
    __threadfence();
    unsigned t = atomicAdd(rb.counter, 1u);
    last = (t == nblk - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double w[N];
#pragma unroll
  for (int k = 0; k < N; ++k) w[k] = 0.0;
  for (unsigned b = threadIdx.x; b < nblk; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < N; ++k) w[k] += ((volatile double*)rb.partials)[(size_t)b * N + k];
  block_sum<N>(w, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) out[k] = w[k];
    *rb.counter = 0u;
    return true;
  }
  return false;
}

// The same sum for a finisher that needs the whole last block: true in every thread of the
// last block, each of which holds the totals in out[]; false in all other blocks.
template <int N>
__device__ __forceinline__ bool grid_sum_last(double v[N], ReduceBuf rb, double out[N]) {
  __shared__ double sh[N * 32];
  __shared__ double tot[N];
  __shared__ bool last;
  const unsigned nblk = gridDim.x * gridDim.y * gridDim.z;
  const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  block_sum<N>(v, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) rb.partials[(size_t)bid * N + k] = v[k];
    __threadfence();
    unsigned t = atomicAdd(rb.counter, 1u);
    last = (t == nblk - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double w[N];
#pragma unroll
  for (int k = 0; k < N; ++k) w[k] = 0.0;
  for (unsigned b = threadIdx.x; b < nblk; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < N; ++k) w[k] += ((volatile double*)rb.partials)[(size_t)b * N + k];
  block_sum<N>(w, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) tot[k] = w[k];
    *rb.counter = 0u;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) out[k] = tot[k];
  return true;
}

}  // namespace pfmp

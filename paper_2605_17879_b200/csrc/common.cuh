// Shared declarations of the B200 straggler-scoring kernels: parameter block, status
// bits, the order-preserving key map and small warp helpers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace guard {

constexpr int kMaxMetrics = 32;
constexpr uint32_t kStatNonFinite = 1u;
constexpr uint32_t kStatTimeout = 2u;
constexpr uint32_t kStatInternal = 4u;

// Per-metric detector parameters, passed to kernels by value (no device copy needed).
struct MetricParams {
    int M;
    int primary;
    int min_signals;
    int n_consec;
    int k;
    float tier_moderate;
    float tier_severe;
    int8_t dir[kMaxMetrics];
    float thrp[kMaxMetrics];      // (float)(thr / 0.6745): cut-off moved to the right-hand side
    float floor_rel[kMaxMetrics];
    float floor_abs[kMaxMetrics];
};

// float32 -> uint32 such that the IEEE total order of finite floats is the unsigned
// order of the keys: negative values have all bits flipped, others only the sign bit.
__host__ __device__ __forceinline__ uint32_t key_of_bits(uint32_t b) {
    return b ^ ((b & 0x80000000u) ? 0xFFFFFFFFu : 0x80000000u);
}
__host__ __device__ __forceinline__ uint32_t bits_of_key(uint32_t k) {
    return k ^ ((k & 0x80000000u) ? 0x80000000u : 0xFFFFFFFFu);
}
__device__ __forceinline__ uint32_t f2key(float x) { return key_of_bits(__float_as_uint(x)); }
__device__ __forceinline__ float key2f(uint32_t k) { return __uint_as_float(bits_of_key(k)); }
__device__ __forceinline__ bool nonfinite_bits(uint32_t b) { return (b & 0x7F800000u) == 0x7F800000u; }

// Median of n values from the two middle order statistics (keys): lower middle for odd
// n (then lo == hi), midpoint with one add and one exact halving for even n.
__device__ __forceinline__ float median_from_keys(uint32_t klo, uint32_t khi, bool even) {
    float a = key2f(klo);
    if (!even) return a;
    return __fmul_rn(0.5f, __fadd_rn(a, key2f(khi)));
}

// Spread used by every robust-z test: the MAD floored relative to |median| and absolutely.
__device__ __forceinline__ float scale_of(float mad, float med, float floor_rel, float floor_abs) {
    float s = mad;
    float rel = __fmul_rn(floor_rel, fabsf(med));
    if (rel > s) s = rel;
    if (floor_abs > s) s = floor_abs;
    return s;
}

// One-sided exceedance in the metric's bad direction: dir * (x - med) > thrp * scale,
// with the right-hand side precomputed (rhs = thrp * scale).
__device__ __forceinline__ bool exceeds(float x, float med, int dir, float rhs) {
    float dev = __fsub_rn(x, med);
    if (dir < 0) dev = -dev;
    return dev > rhs;
}

// A kernel launched by launch_after may start as soon as every CTA of the kernel in front of it in the stream has called
// pdl_trigger or exited; pdl_wait returns when that kernel has ended and its writes are visible.  What the kernel reads or
// writes before pdl_wait must therefore not be touched by the kernel in front, and be complete when that one starts.
// Kernels that have nothing to do before it call it first (a kernel must not end without it: the next one in the stream
// relies on it), and save a part of the launch latency: 1 to 2 us per launch.  pdl_trigger only where the next kernel
// has such work: CTAs that merely wait keep SMs from other streams (a pass of 16 384 ranks x 8 x 200 448 us with the
// split path's kernels triggering early, 442 without; 8 192 x 8 with ties 150 / 136).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_after_smem(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const A &...args) {
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &early;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, kernel, args...);
    if (e != cudaSuccess) (void)cudaGetLastError();   // the caller gets it; the thread's next CUDA call must not find it again
    return e;
}
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, const A &...args) {
    return launch_after_smem(kernel, grid, block, 0, st, args...);
}

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }

}  // namespace guard

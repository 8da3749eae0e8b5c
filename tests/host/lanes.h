// lanes.h -- CUDA blocks on the CPU, for tests: every thread of a block is a fiber that runs until it meets a
// collective, in an order that the test chooses, so a lane may be as far ahead of another as the programming model
// allows.  Included in front of a .cu file's text (compiled as C++ with -fsanitize=thread, whose hooks lanes.cpp takes
// for itself: every access to memory outside the fibers' stacks is checked for a conflicting one that no
// __syncwarp or __syncthreads orders; shuffles, votes and reductions order nothing).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>

#define __device__
#define __host__
#define __global__
#define __constant__
#define __shared__ static  // blocks run one after another
#define __launch_bounds__(...)
#define __grid_constant__
#include <cuda_runtime.h>
#undef __noinline__
#define __noinline__ __attribute__((noinline))

extern uint3 threadIdx, blockIdx;
extern dim3 blockDim, gridDim;

namespace lanes {
// one value per thread in, the values of the thread's warp or block out
const uint64_t* warp_exchange(uint64_t v);
uint64_t block_or(uint64_t v);
void warp_order();  // __syncwarp
void launch(int64_t blocks, int threads, size_t dynamic_bytes, const std::function<void()>& thread);
void* dynamic_shared();

template <typename T>
uint64_t bits(T v)
{
    uint64_t b = 0;
    std::memcpy(&b, &v, sizeof(T));
    return b;
}
template <typename T>
T from(uint64_t b)
{
    T v;
    std::memcpy(&v, &b, sizeof(T));
    return v;
}
inline int lane() { return threadIdx.x & 31; }
}  // namespace lanes

// the runtime's overloads for kernels, which only nvcc sees: a kernel may use what it asks for, one block at a time
template <typename... A>
cudaError_t cudaFuncSetAttribute(void (*)(A...), cudaFuncAttribute, int) { return cudaSuccess; }
template <typename... A>
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, void (*)(A...), int, size_t)
{
    *n = 1;
    return cudaSuccess;
}

inline void __syncwarp(unsigned = ~0u) { lanes::warp_order(); }
inline void __syncthreads() { lanes::block_or(0); }
inline int __syncthreads_or(int v) { return lanes::block_or(v != 0) != 0; }
template <typename T>
T __shfl_sync(unsigned, T v, int src, int width = 32)
{
    return lanes::from<T>(lanes::warp_exchange(lanes::bits(v))[(lanes::lane() & ~(width - 1)) + (src & (width - 1))]);
}
template <typename T>
T __shfl_xor_sync(unsigned, T v, int off, int width = 32)
{
    (void)width;  // offsets below the width only
    return lanes::from<T>(lanes::warp_exchange(lanes::bits(v))[lanes::lane() ^ off]);
}
template <typename T>
T __shfl_up_sync(unsigned, T v, int off)
{
    const uint64_t* x = lanes::warp_exchange(lanes::bits(v));
    return lanes::from<T>(x[lanes::lane() >= off ? lanes::lane() - off : lanes::lane()]);
}
inline unsigned __ballot_sync(unsigned, int v)
{
    const uint64_t* x = lanes::warp_exchange(v != 0);
    unsigned m = 0;
    for (int i = 0; i < 32; ++i) m |= (unsigned)x[i] << i;
    return m;
}
inline int __any_sync(unsigned m, int v) { return __ballot_sync(m, v) != 0; }
inline int __all_sync(unsigned m, int v) { return __ballot_sync(m, v) == ~0u; }
inline unsigned __reduce_min_sync(unsigned, unsigned v)
{
    const uint64_t* x = lanes::warp_exchange(v);
    unsigned m = ~0u;
    for (int i = 0; i < 32; ++i) m = (unsigned)x[i] < m ? (unsigned)x[i] : m;
    return m;
}
uint32_t atomicAdd(uint32_t* p, uint32_t v);
template <typename T>
T __ldg(const T* p) { return *p; }
template <typename T>
T __ldcs(const T* p) { return *p; }
inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline int __clzll(long long v) { return v == 0 ? 64 : __builtin_clzll((unsigned long long)v); }
inline uint32_t __float_as_uint(float v) { return lanes::from<uint32_t>(lanes::bits(v)); }
inline float __uint_as_float(uint32_t v) { return lanes::from<float>(v); }
inline float __uint2float_rz(uint32_t v)
{
    const float f = (float)v;
    return (double)f > (double)v ? std::nextafterf(f, 0.0f) : f;
}
inline float __int2float_rn(int v) { return (float)v; }
inline float __uint2float_rn(unsigned v) { return (float)v; }
inline int __float2int_rz(float v)
{
    return v != v ? 0 : v >= 2147483648.0f ? INT32_MAX : v <= -2147483648.0f ? INT32_MIN : (int)v;
}

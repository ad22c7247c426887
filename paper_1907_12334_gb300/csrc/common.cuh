// common.cuh -- internal helpers of the MSG-MIMC CUDA library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/msg_mimc.h"

namespace msg {

// thread-local last error, set by every failing entry point
void set_error(const std::string& what);
void clear_error();

#define MSG_CUDA_TRY(expr)                                                                        \
    do {                                                                                          \
        cudaError_t _e = (expr);                                                                  \
        if (_e != cudaSuccess) {                                                                  \
            ::msg::set_error(std::string(#expr) + ": " + cudaGetErrorString(_e));                 \
            return MSG_ERR_CUDA;                                                                  \
        }                                                                                         \
    } while (0)

#define MSG_CHECK_LAUNCH()                                                                        \
    do {                                                                                          \
        cudaError_t _e = cudaGetLastError();                                                      \
        if (_e != cudaSuccess) {                                                                  \
            ::msg::set_error(std::string("kernel launch: ") + cudaGetErrorString(_e));            \
            return MSG_ERR_CUDA;                                                                  \
        }                                                                                         \
    } while (0)

// Pinned host staging for the host-side tables an entry point uploads, so that
// the upload is a true asynchronous copy and the call returns without waiting
// for the stream.  staging_acquire hands out a slot of at least `bytes`;
// staging_release records an event on `st` after the copies from the slot were
// enqueued, and the slot is handed out again only once that event has completed.
int staging_acquire(size_t bytes, void** ptr, int* token);
int staging_release(int token, cudaStream_t st);

// Stream-ordered temporary (freed with cudaFreeAsync on the same stream) from a pool of
// this library's own, one per device, made on first use.  It keeps up to kTempKeep bytes
// between calls: the device's default pool gives everything back at each
// synchronisation, and mapping it again cost a call 200 us.  Returns the CUDA error, and
// leaves none pending.
constexpr uint64_t kTempKeep = uint64_t(64) << 20;
cudaError_t temp_alloc(void** p, size_t bytes, cudaStream_t st);

// (TZ)x of FP32 results, exact.  The conversion instruction to FP64 runs at the FP64
// pipe's rate (two a clock and SM), a limit of its own for kernels that write FP64 fields
// from FP32 sums; a normal number is widened by moving its IEEE-754 fields instead: the
// exponent's bias grows by 1023 - 127 = 896, the 23-bit fraction moves to the top of 52 bits.
__device__ __forceinline__ bool widens(float x)  // neither zero, subnormal, infinite nor NaN
{
    return (__float_as_uint(x) & 0x7fffffffu) - 0x00800000u < 0x7f000000u;
}
__device__ __forceinline__ double widen_normal(float x)
{
    const uint32_t u = __float_as_uint(x);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}
// N results at p, p + stride, ..; one test for all of them keeps the stores free of branches
template <int N>
__device__ __forceinline__ void store_wide(float* p, int64_t stride, const float (&v)[N], int n)
{
#pragma unroll
    for (int k = 0; k < N; ++k, p += stride)
        if (k < n) *p = v[k];
}
template <int N>
__device__ __forceinline__ void store_wide(double* p, int64_t stride, const float (&v)[N], int n)
{
    bool all = n >= N;
#pragma unroll
    for (int k = 0; k < N; ++k) all &= widens(v[k]);
    if (all) {
#pragma unroll
        for (int k = 0; k < N; ++k, p += stride) *p = widen_normal(v[k]);
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k, p += stride)
            if (k < n) *p = (double)v[k];
    }
}

// ---------------------------------------------------------------------------
// Hierarchy layout.
//
// Grid (p,q) of the semi-coarsened hierarchy (Eq. (2.1)) has nx = 2^p,
// ny = 2^q cells and (nx+1)(ny+1) nodes including the boundary, stored row by
// row (x fastest).  All grids (p',q') with p' <= P, q' <= Q of one rectangle
// are stored back to back in (p' major, q' minor) order, so with
//   T(n) = sum_{k=1..n} (2^k + 1) = 2^(n+1) - 2 + n
// grid (p',q') starts at node T(p'-1) T(Q) + (2^p' + 1) T(q'-1) and the whole
// rectangle holds T(P) T(Q) nodes.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int64_t tsum(int n) { return (int64_t(2) << n) - 2 + n; }
__host__ __device__ __forceinline__ int64_t grid_offset(int p, int q, int Qtop)
{
    return tsum(p - 1) * tsum(Qtop) + (int64_t)((1 << p) + 1) * tsum(q - 1);
}
// the same in 32 bits (a rectangle holds at most T(12)^2 < 2^27 nodes)
__host__ __device__ __forceinline__ int grid_offset32(int p, int q, int Qtop)
{
    auto t = [](int n) { return (2 << n) - 2 + n; };
    return t(p - 1) * t(Qtop) + ((1 << p) + 1) * t(q - 1);
}
__host__ __device__ __forceinline__ int64_t rect_nodes(int P, int Q) { return tsum(P) * tsum(Q); }
__host__ __device__ __forceinline__ int64_t field_nodes(int P, int Q)
{
    return (int64_t)((1 << (P + 1)) + 1) * ((1 << (Q + 1)) + 1);
}

}  // namespace msg

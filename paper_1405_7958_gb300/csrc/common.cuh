// Shared device helpers of the segmentation kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rt.h"

#define RT_CUDA_TRY(expr)                                   \
    do {                                                    \
        cudaError_t _e = (expr);                            \
        if (_e != cudaSuccess) return RT_ECUDA;             \
    } while (0)

namespace rtk {

constexpr int kMaxSide = 32768;

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int32_t ld_relaxed_i32(const int32_t *p)
{
    int32_t v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Record the first error code raised on the device (0 = RT_OK stays until an
// error arrives). Never traps.
__device__ __forceinline__ void raise_status(int32_t *st, int code)
{
    if (st) atomicCAS(st, 0, code);
}

// Grid-wide barrier for a cooperative launch (all CTAs co-resident).
// bar[0] = arrival count, bar[1] = generation. The wait is bounded by
// `timeout_ns`; on expiry the CTA records RT_ETIMEOUT in *err and returns
// false so the caller can leave the loop.
__device__ __forceinline__ bool grid_barrier(uint32_t *bar, uint32_t nblocks, int32_t *err,
                                             uint64_t timeout_ns)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        s_ok = 1;
        uint32_t gen = ld_acquire(bar + 1);
        __threadfence();
        uint32_t arrived = atomicAdd(bar, 1u);
        if (arrived == nblocks - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            uint64_t t0 = globaltimer_ns();
            uint32_t spins = 0;
            while (ld_acquire(bar + 1) == gen) {
                if (++spins > 64) __nanosleep(64);
                if ((spins & 255u) == 0 && globaltimer_ns() - t0 > timeout_ns) {
                    raise_status(err, RT_ETIMEOUT);
                    s_ok = 0;
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

// 16 bytes of a row of W bytes from column c, of which n exist (<= 0: none;
// the others are 0). Rows that are not 16-byte aligned: the aligned words
// around them, shifted, while these lie in the row; else byte by byte.
__device__ __forceinline__ void load_row16(const uint8_t *row, int c, int n, int W, uint32_t (&w)[4])
{
    const uint8_t *p = row + c;
    const uint32_t off = (uint32_t)(uintptr_t)p & 3u;
    w[0] = w[1] = w[2] = w[3] = 0u;
    if (n == 16 && ((uintptr_t)p & 15u) == 0) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        w[0] = v.x;
        w[1] = v.y;
        w[2] = v.z;
        w[3] = v.w;
    } else if (n == 16 && (off == 0 || (c >= 4 && c + 20 <= W))) {
        const uint32_t *q = reinterpret_cast<const uint32_t *>(p - off);
        uint32_t v[5];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = q[k];
        v[4] = off ? q[4] : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = __funnelshift_r(v[k], v[k + 1], 8u * off);
    } else {
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (k < n) w[k >> 2] |= (uint32_t)p[k] << (8 * (k & 3));
    }
}

// The first n of 4 N bytes (w) to o, in the widest stores its alignment allows.
template <int N>
__device__ __forceinline__ void store_bytes(uint8_t *o, int n, const uint32_t (&w)[N])
{
    if (n == 4 * N && ((uintptr_t)o & 15u) == 0) {
#pragma unroll
        for (int k = 0; k < N / 4; ++k)
            reinterpret_cast<uint4 *>(o)[k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
    } else if (n == 4 * N && ((uintptr_t)o & 3u) == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) reinterpret_cast<uint32_t *>(o)[k] = w[k];
    } else {
#pragma unroll
        for (int k = 0; k < 4 * N; ++k)
            if (k < n) o[k] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
    }
}

// 64 ints of a row, value(c) for column c, by 16 threads (q = 0 .. 15): the
// aligned quads of the row, whatever its alignment, and its ends one by one.
template <class V>
__device__ __forceinline__ void store_row64(int32_t *row, int q, V &&value)
{
    const int head = (int)((0u - (uint32_t)(uintptr_t)row) >> 2) & 3, at = head + 4 * q;
    if (at + 4 <= 64) {
        *reinterpret_cast<int4 *>(row + at) = make_int4(value(at), value(at + 1), value(at + 2), value(at + 3));
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (at + k < 64) row[at + k] = value(at + k);
    }
    if (q < head) row[q] = value(q);
}

// First statement of a kernel launched by launch_early: lets the next such
// kernel of the stream take its place on the SMs as soon as all blocks of
// this one have theirs, and waits until the kernels before this one are
// complete and their writes visible.
// Such a kernel reads no buffer of a stream by __ldg or through __restrict__:
// non-coherent loads want memory that nothing writes while the kernel lives,
// and it lives beside the kernel before it. (Plain loads cost nothing here:
// the chain and its operations within 0.2 %.)
__device__ __forceinline__ void start_early()
{
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

// kernel<<<grid, block, smem, s>>>(args...) whose blocks may be placed before
// the stream's previous kernel has ended (they wait in start_early), so that
// the launch's latency lies behind it: 1 to 2 us a kernel (a 1K chain of 14
// kernels 133 -> 110 us, labeling 700 x 700 in 4 of them 31 -> 24).
template <class... P, class... A>
inline cudaError_t launch_early(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

__host__ __device__ __forceinline__ int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
__host__ __device__ __forceinline__ int64_t round_up(int64_t a, int64_t b) { return ceil_div(a, b) * b; }

}  // namespace rtk

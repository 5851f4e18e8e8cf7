/*
 * A state in and out of a handle or a grid of a batch, from and to the caller's
 * device memory.
 *
 * Bound by DRAM bandwidth (large grids) or by launches (small ones), so each
 * direction is one kernel: in, the FP64 state and its FP32 shadow from one
 * read of the caller's arrays, and the status word cleared; out, the averages
 * copied and the gradients widened from the shadow into the caller's array
 * without a stop in the handle's.  Against two copies, a shadow pass over the
 * copied state and a memory set (in), and a widening pass and two copies (out),
 * a 2D mixed state moves 64 + 40 bytes a cell and variable instead of 88 + 72.
 * GB300, a pass with a state in and out: 12 grids 2.92 to 2.48 ms, 2048^2 0.16 ms
 * and 256^3 1.08 ms less, 64^2 20 us less.
 *
 * The kernels take the place of copies that accept any address, so they are
 * used only where both arrays lie, over their whole length, in one allocation
 * of the current device; host and managed memory, another device's and
 * anything the driver does not describe keep the copies.
 */
#pragma once
#include <cuda.h>

#include "internal.h"

namespace gks {

/* M the dimension: gradients are M arrays of n, averages one.  MIXED: into the shadow too. */
template <int M, bool MIXED>
__global__ void __launch_bounds__(256) state_in_kernel(const double *__restrict__ Wu, const double *__restrict__ Gu,
                                                       double *__restrict__ W, double *__restrict__ G, Shadow s, long n,
                                                       int *__restrict__ status)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *status = 0;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const double w = Wu[i];
        double g[M];
#pragma unroll
        for (int a = 0; a < M; ++a) g[a] = Gu[a * n + i];
        W[i] = w;
        if (MIXED) split_store(w, s.hi, s.lo, i);
#pragma unroll
        for (int a = 0; a < M; ++a) {
            G[a * n + i] = g[a];
            if (MIXED) s.g[a * n + i] = (float)g[a];
        }
    }
}

/* g: the gradients' FP32 shadow, or nullptr for the FP64 array G */
template <int M>
__global__ void __launch_bounds__(256) state_out_kernel(const double *__restrict__ W, const double *__restrict__ G,
                                                        const float *__restrict__ g, double *__restrict__ Wu,
                                                        double *__restrict__ Gu, long n)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const double w = W[i];
        double d[M];
#pragma unroll
        for (int a = 0; a < M; ++a) d[a] = g ? (double)g[a * n + i] : G[a * n + i];
        Wu[i] = w;
#pragma unroll
        for (int a = 0; a < M; ++a) Gu[a * n + i] = d[a];
    }
}

/* Whether [p, p + bytes) lies in one allocation of the current device (and is
 * aligned for doubles). */
inline bool in_device_memory(const void *p, size_t bytes)
{
    using Range = CUresult (*)(CUdeviceptr *, size_t *, CUdeviceptr);
    static const Range range = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) != cudaSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return (Range)f;
    }();
    if (!range || !p || ((size_t)p & 7)) return false;
    int dev = -1;
    cudaPointerAttributes a{};
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type != cudaMemoryTypeDevice || a.device != dev) return false;
    CUdeviceptr base = 0;
    size_t size = 0;
    if (range(&base, &size, (CUdeviceptr)(size_t)p) != CUDA_SUCCESS) return false;
    return (size_t)p - (size_t)base <= size && bytes <= size - ((size_t)p - (size_t)base);
}

inline unsigned state_blocks(long n) { return (unsigned)((n + 255) / 256 < 65536 ? (n + 255) / 256 : 65536); }

/* n doubles of averages and M n of gradients into W, G (and, with s.hi, the shadow) */
template <int M>
cudaError_t state_in(const double *Wu, const double *Gu, double *W, double *G, const Shadow &s, long n, int *status, cudaStream_t st)
{
    if (s.hi) state_in_kernel<M, true><<<state_blocks(n), 256, 0, st>>>(Wu, Gu, W, G, s, n, status);
    else state_in_kernel<M, false><<<state_blocks(n), 256, 0, st>>>(Wu, Gu, W, G, s, n, status);
    return cudaGetLastError();
}

template <int M>
cudaError_t state_out(const double *W, const double *G, const float *g, double *Wu, double *Gu, long n, cudaStream_t st)
{
    state_out_kernel<M><<<state_blocks(n), 256, 0, st>>>(W, G, g, Wu, Gu, n);
    return cudaGetLastError();
}

/* The status word after everything enqueued on the stream: the copy and the wait in one stop of the host. */
inline cudaError_t read_status(const int *status, int *out, cudaStream_t st)
{
    const cudaError_t e = cudaMemcpyAsync(out, status, sizeof(int), cudaMemcpyDeviceToHost, st);
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

} // namespace gks

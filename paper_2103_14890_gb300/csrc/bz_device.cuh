// bz_device.cuh -- small device helpers shared by the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bz {

template <typename T> struct C2;
template <> struct C2<double> { using type = double2; };
template <> struct C2<float> { using type = float2; };

template <typename V> __device__ __forceinline__ V cmk(decltype(V::x) a, decltype(V::x) b) {
    V r;
    r.x = a;
    r.y = b;
    return r;
}

// acc += a * b (complex)
template <typename V> __device__ __forceinline__ void cmac(V &acc, V a, V b) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}

// FP64 quotients that spare the FP64 pipe, on which a warp instruction takes 16
// cycles of an SM.  rcp64: the hardware's approximate reciprocal y of b (relative
// error e below 2^-17) and one step of the cubic iteration y (1 + e + e^2), e = 1 -
// b y (Householder's method of order 2): three operations, relative error below
// 2^-51 plus a rounding, for 2^-1021 < |b| < 2^1021 (measured: 1 ulp).  div64: a / b from y =
// rcp64(b) with the remainder's correction (Markstein 1990), three more, within
// half an ulp in all but rare cases, one ulp in those (none in 2^20).  The full
// division takes about three times as many.
__device__ __forceinline__ double rcp64(double b) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    double e = fma(-b, y, 1.0);
    e = fma(e, e, e);
    return fma(y, e, y);
}
__device__ __forceinline__ double div64(double a, double b, double y) {
    const double q = a * y;
    return fma(fma(-b, q, a), y, q);
}

// 2^e / b for a finite b >= 2^e, e given as scale = e << 20: rcp64 of b with the
// power of two taken off its exponent, off the FP64 pipe (below 2^-1022: that).
__device__ __forceinline__ double scaled_rcp(double b, int scale) {
    const unsigned hi = min((unsigned)(__double2hiint(b) - scale), 0x7fd00000u);
    return rcp64(__hiloint2double((int)hi, __double2loint(b)));
}

// Tiled half-spectrum layout: [cell / 32][mode][cell % 32].
__host__ __device__ __forceinline__ int64_t tiled_index(int64_t cell, int64_t mode, int64_t nhalf) {
    return (cell >> 5) * nhalf * 32 + mode * 32 + (cell & 31);
}

// Block-wide sum of up to 5 doubles; every thread receives the totals.
// `red` must hold 32 * 5 doubles of shared memory.
template <int K> __device__ __forceinline__ void block_sum(double (&v)[K], double *red) {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) red[warp * K + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) s += red[w * K + k];   // same order in every thread
        v[k] = s;
    }
    __syncthreads();
}

// Programmatic dependent launch.  griddep_launch: the next kernel of the stream,
// if launched with the attribute (launch_after), may start its prologue once
// every CTA of this grid has called it; griddep_wait: returns when the kernel
// before has completed and its writes are visible (at once without the
// attribute).  A kernel launched that way waits before it touches anything the
// kernels before it read or write, and reads what they wrote by __ldcg or
// cp.async: those memory changes while the kernel runs, so a pointer to it must
// not be `const __restrict__` (the compiler would take it as read-only for the
// kernel's lifetime and may read it by the non-coherent path, ahead of the wait).
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch `kernel`; pdl: as a programmatic dependent of the kernel before it.
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, bool pdl,
                         A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Velocity of flat grid index `idx` along dimension i (j_1 slowest).
__device__ __forceinline__ double grid_velocity(int64_t idx, int i, int dim, int N, double L,
                                                double dv) {
    int64_t t = idx;
    for (int q = dim - 1; q > i; --q) t /= N;
    return -L + (double)(t % N) * dv;
}

// Latch the first device-side error of a call into the library's error word.
__device__ __forceinline__ void raise_device_error(int *err, int code) {
    if (err) atomicCAS(err, 0, code);
}

}  // namespace bz

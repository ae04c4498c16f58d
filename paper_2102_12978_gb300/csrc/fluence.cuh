// fluence.cuh -- read-out kernels: the fluence reducer, which turns the
// per-cell accumulator into a dense FP64 array (times 1 / (window length) it is
// the intensity (1/tau) integral |S| dt of Section 5 over a window of whole
// periods), and the dense copy of a pitched field array.
//
// Both are bound by HBM: one warp copies a row of the box at a time (no index
// division), by 16-byte accesses where the row length and the destination
// allow them.  411 x 411 x 738 FP32 cells, the read-outs whole (allocation and
// wait included): fluence 411 us, a field 182 us (4.9 and 5.5 TB/s); through a
// staging array and a copy, and as a 2-D copy of the runtime, 1263 and 300 us.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fdtd {

// double(f) from the bits: the FP64 pipe, which converts at 1/64 of the FP32
// rate, is left the one subtraction per cell (with the two conversions and a
// product on it the reducer was bound by the pipe: 964 us for 411 x 411 x 738
// cells).  Zeros and normal numbers by integer operations, the rest converted.
__device__ __forceinline__ double widen(float f)
{
    const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
    if (e - 1u >= 254u && (u << 1) != 0u) return double(f);
    const unsigned hi = (u & 0x80000000u) | ((u << 1) ? ((u & 0x7fffffffu) >> 3) + (896u << 20) : 0u);
    return __hiloint2double(int(hi), int(u << 29));
}
__device__ __forceinline__ double flu_value(double v) { return v; }
__device__ __forceinline__ double flu_value(float2 v) { return widen(v.x) - widen(v.y); }

// V cells per access: 2 (16-byte stores; nx even, out 16-byte aligned) or 1.
template <typename acc_t, int V>
__global__ void __launch_bounds__(256)
fluence_export(const acc_t* __restrict__ F, double* __restrict__ out, int nx, long long rows, int pitch)
{
    const int lane = threadIdx.x & 31;
    for (long long r = (blockIdx.x * 256ll + threadIdx.x) >> 5; r < rows; r += gridDim.x * 8ll) {
        const acc_t* f = F + r * pitch;
        double* o = out + r * nx;
        #pragma unroll 4
        for (int i = lane * V; i < nx; i += 32 * V) {
            if constexpr (V == 2) {
                struct alignas(16) Two { double a, b; };
                struct alignas(2 * sizeof(acc_t)) In { acc_t a, b; };
                const In v = *reinterpret_cast<const In*>(f + i);
                *reinterpret_cast<Two*>(o + i) = Two{flu_value(v.a), flu_value(v.b)};
            } else {
                o[i] = flu_value(f[i]);
            }
        }
    }
}

// Rows of nx elements, `pitch` apart, to dense rows.  V elements per access:
// 16 / sizeof(T) (nx a multiple of it, out 16-byte aligned) or 1.
template <typename T, int V>
__global__ void __launch_bounds__(256)
field_export(const T* __restrict__ f, T* __restrict__ out, int nx, long long rows, int pitch)
{
    const int lane = threadIdx.x & 31;
    for (long long r = (blockIdx.x * 256ll + threadIdx.x) >> 5; r < rows; r += gridDim.x * 8ll) {
        const T* s = f + r * pitch;
        T* o = out + r * nx;
        #pragma unroll 4
        for (int i = lane * V; i < nx; i += 32 * V) {
            if constexpr (V > 1) {
                struct alignas(V * sizeof(T)) Vec { T e[V]; };
                *reinterpret_cast<Vec*>(o + i) = *reinterpret_cast<const Vec*>(s + i);
            } else {
                o[i] = s[i];
            }
        }
    }
}

// CTAs of either kernel: one warp per row, at most `most` CTAs.
inline unsigned export_blocks(long long rows, int sm_count)
{
    const long long want = (rows + 7) / 8, most = 16ll * (sm_count > 0 ? sm_count : 152);
    return unsigned(want < most ? want : most);
}

template <typename acc_t>
inline cudaError_t launch_fluence_export(const acc_t* F, double* out, int nx, long long rows, int pitch, int sm_count,
                                         cudaStream_t s)
{
    const unsigned b = export_blocks(rows, sm_count);
    if (nx % 2 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0)
        fluence_export<acc_t, 2><<<b, 256, 0, s>>>(F, out, nx, rows, pitch);
    else fluence_export<acc_t, 1><<<b, 256, 0, s>>>(F, out, nx, rows, pitch);
    return cudaGetLastError();
}

template <typename T>
inline cudaError_t launch_field_export(const void* f, void* out, int nx, long long rows, int pitch, int sm_count,
                                       cudaStream_t s)
{
    constexpr int V = 16 / int(sizeof(T));
    const unsigned b = export_blocks(rows, sm_count);
    if (nx % V == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0)
        field_export<T, V><<<b, 256, 0, s>>>(static_cast<const T*>(f), static_cast<T*>(out), nx, rows, pitch);
    else field_export<T, 1><<<b, 256, 0, s>>>(static_cast<const T*>(f), static_cast<T*>(out), nx, rows, pitch);
    return cudaGetLastError();
}

}  // namespace fdtd

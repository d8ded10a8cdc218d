// Packed float32 pairs and shared-memory staging of the CUDA-core kernels (the float32 dtype path).
//
// Every kernel of that path gives rows (routes or tokens) to threads and streams the other side's
// rows, which the block stages in shared memory and every thread of a warp reads at the same address.
// The multiply-adds themselves are not the bound (29 us of the encode below, 72 of the token pass of
// calls 3 and 2): shared-memory reads are, and the latency of a row's chain of products at eight to
// twelve warps per SM. So a row is read 16 bytes at a time (one access per four channels), it serves
// two rows of the thread where registers allow, and it is multiplied in pairs: fma.rn.f32x2 does two
// fused multiply-adds, each rounded as fmaf rounds, in one issue slot. The rows of the next step land
// (cp.async) while this step's are worked on. 8 x 16,384 tokens, M = 128, D = 32: encode 123 -> 62 us,
// decode 102 -> 70, route passes of calls 3, 2, 1 162, 130, 130 -> 108, 84, 84, token passes 232, 187
// -> 153, 120.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace flarepp {
namespace simt {

using f2 = uint64_t;  // two floats, the first in the low half

__device__ __forceinline__ f2 pack2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// a row of D floats in global memory (16-byte aligned), times s, as packed pairs; zeros when !in
template <int D>
__device__ __forceinline__ void load_row(f2* r, const float* p, float s, bool in) {
#pragma unroll
    for (int i = 0; i < D / 4; ++i) {
        const float4 v = in ? reinterpret_cast<const float4*>(p)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        r[2 * i] = pack2(v.x * s, v.y * s);
        r[2 * i + 1] = pack2(v.z * s, v.w * s);
    }
}
template <int D>
__device__ __forceinline__ void store_row(float* p, const f2* r, float s) {
#pragma unroll
    for (int i = 0; i < D / 4; ++i) {
        const float2 a = unpack2(r[2 * i]), b = unpack2(r[2 * i + 1]);
        reinterpret_cast<float4*>(p)[i] = make_float4(a.x * s, a.y * s, b.x * s, b.y * s);
    }
}

// <a, row> over D channels: four partial sums (two packed), added at the end
template <int D>
__device__ __forceinline__ float dot_row(const f2* a, const float* row) {
    f2 x = 0, y = 0;
#pragma unroll
    for (int i = 0; i < D / 4; ++i) {
        const ulonglong2 k = reinterpret_cast<const ulonglong2*>(row)[i];
        x = fma2(a[2 * i], k.x, x);
        y = fma2(a[2 * i + 1], k.y, y);
    }
    const float2 u = unpack2(x), v = unpack2(y);
    return (u.x + u.y) + (v.x + v.y);
}
// acc += w row
template <int D>
__device__ __forceinline__ void axpy_row(f2* acc, float w, const float* row) {
    const f2 w2 = pack2(w, w);
#pragma unroll
    for (int i = 0; i < D / 4; ++i) {
        const ulonglong2 v = reinterpret_cast<const ulonglong2*>(row)[i];
        acc[2 * i] = fma2(w2, v.x, acc[2 * i]);
        acc[2 * i + 1] = fma2(w2, v.y, acc[2 * i + 1]);
    }
}

// Half rows: two adjacent lanes share a row, lane h (0 or 1) of the pair taking the four-channel
// groups h, h + 2, ... (D / 2 channels, D / 4 pairs). A staged row's half is read once into registers
// for every product that takes it; the two halves of a warp's access lie side by side.
template <int D>
__device__ __forceinline__ void load_half(f2* r, const float* p, float s, int h) {
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
        const float4 v = reinterpret_cast<const float4*>(p)[2 * i + h];
        r[2 * i] = pack2(v.x * s, v.y * s);
        r[2 * i + 1] = pack2(v.z * s, v.w * s);
    }
}
template <int D>
__device__ __forceinline__ void read_half(f2* r, const float* row, int h) {
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
        const ulonglong2 v = reinterpret_cast<const ulonglong2*>(row)[2 * i + h];
        r[2 * i] = v.x;
        r[2 * i + 1] = v.y;
    }
}
template <int D>
__device__ __forceinline__ void store_half(float* p, const f2* r, float s, int h) {
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
        const float2 a = unpack2(r[2 * i]), b = unpack2(r[2 * i + 1]);
        reinterpret_cast<float4*>(p)[2 * i + h] = make_float4(a.x * s, a.y * s, b.x * s, b.y * s);
    }
}
// <a, b> over the pair's D channels (every lane of the warp takes part)
template <int D>
__device__ __forceinline__ float dot_half(const f2* a, const f2* b) {
    f2 x = 0, y = 0;
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
        x = fma2(a[2 * i], b[2 * i], x);
        y = fma2(a[2 * i + 1], b[2 * i + 1], y);
    }
    const float2 u = unpack2(x), v = unpack2(y);
    const float t = (u.x + u.y) + (v.x + v.y);
    return t + __shfl_xor_sync(0xffffffffu, t, 1);
}
// acc += w b
template <int D>
__device__ __forceinline__ void axpy_half(f2* acc, float w, const f2* b) {
    const f2 w2 = pack2(w, w);
#pragma unroll
    for (int i = 0; i < D / 4; ++i) acc[i] = fma2(w2, b[i], acc[i]);
}

// cp.async of 16 (4) bytes, zeros when !in (the source must still be a valid address)
__device__ __forceinline__ void copy16(void* dst, const void* src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 16u : 0u)
                 : "memory");
}
__device__ __forceinline__ void copy4(void* dst, const void* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 4u : 0u)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest N groups of this thread's copies have landed
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// stage rows [first, first + R) of a [rows][D] array (rows beyond `rows` as zeros) in dst
template <int D, int R>
__device__ __forceinline__ void stage_rows(float (*dst)[D], const float* src, int64_t first,
                                           int64_t rows) {
    for (int i = threadIdx.x; i < R * D / 4; i += blockDim.x) {
        const int64_t row = first + i / (D / 4);
        const bool in = row < rows;
        copy16(&dst[0][0] + 4 * i, src + (in ? row * D + 4 * (i % (D / 4)) : 0), in);
    }
}
// and of a [rows] array
template <int R>
__device__ __forceinline__ void stage_values(float* dst, const float* src, int64_t first,
                                             int64_t rows) {
    for (int i = threadIdx.x; i < R; i += blockDim.x) {
        const bool in = first + i < rows;
        copy4(dst + i, src + (in ? first + i : 0), in);
    }
}

}  // namespace simt
}  // namespace flarepp

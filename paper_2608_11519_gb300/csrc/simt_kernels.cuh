// CUDA-core kernels of the routing chain: the float32 dtype path (instantiated in
// simt_f32.cu). Products and accumulation in float32; tf32 tensor cores could not meet
// the float32 tolerance.
//
// Encode (calls 1 and 2, Sec. 3.2): one thread per one or two route rows streams a chunk of tokens
// through an online softmax (running max, running sum, weighted value sum) and writes
// the chunk's partials. Combine merges the partials of all chunks by the stable
// log-sum-exp reduction of App. A.3. Decode (call 3): one thread per one or two tokens streams the
// M routes through an online softmax over routes.
//
// Scores are kept in the base-2 domain: x = (scale * log2 e) <q, k>, weights 2^(x - max).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "flarepp_internal.h"
#include "simt_math.cuh"
#include "tc_ptx.cuh"

namespace flarepp {
namespace simt {

constexpr float kLog2e = 1.4426950408889634f;
// tokens (encode) or routes (decode) staged per step, by the rows per thread: their scores stay in
// registers, R x kTile of them
template <int R>
constexpr int kTile = R == 2 ? 8 : 16;

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One step of R rows' online softmax over kTile staged rows of the other side, cnt of them valid:
// scores with ks, weights 2^(score - max), and the weighted sums of vs in o. With R = 2 every staged
// row is read once for two rows.
template <int D, int R>
__device__ __forceinline__ void softmax_tile(const f2 (*q)[D / 2], f2 (*o)[D / 2], float* mx,
                                             float* l, const float (*ks)[D],
                                             const float (*vs)[D], int cnt) {
    float sc[R][kTile<R>];
    float tmax[R];
#pragma unroll
    for (int r = 0; r < R; ++r) tmax[r] = -INFINITY;
#pragma unroll
    for (int j = 0; j < kTile<R>; ++j) {
        f2 x[R] = {}, y[R] = {};
#pragma unroll
        for (int i = 0; i < D / 4; ++i) {
            const ulonglong2 k = reinterpret_cast<const ulonglong2*>(ks[j])[i];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                x[r] = fma2(q[r][2 * i], k.x, x[r]);
                y[r] = fma2(q[r][2 * i + 1], k.y, y[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 u = unpack2(x[r]), v = unpack2(y[r]);
            const float t = (u.x + u.y) + (v.x + v.y);
            sc[r][j] = j < cnt ? t : -INFINITY;
            tmax[r] = fmaxf(tmax[r], sc[r][j]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float mnew = fmaxf(mx[r], tmax[r]);
        const float corr = fast_exp2(mx[r] - mnew);  // 0 on the first tile
        l[r] *= corr;
        const f2 corr2 = pack2(corr, corr);
#pragma unroll
        for (int d = 0; d < D / 2; ++d) o[r][d] = mul2(o[r][d], corr2);
        mx[r] = mnew;
    }
#pragma unroll
    for (int j = 0; j < kTile<R>; ++j) {
        f2 w[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float p = fast_exp2(sc[r][j] - mx[r]);  // 0 for masked rows
            l[r] += p;
            w[r] = pack2(p, p);
        }
#pragma unroll
        for (int i = 0; i < D / 4; ++i) {
            const ulonglong2 v = reinterpret_cast<const ulonglong2*>(vs[j])[i];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                o[r][2 * i] = fma2(w[r], v.x, o[r][2 * i]);
                o[r][2 * i + 1] = fma2(w[r], v.y, o[r][2 * i + 1]);
            }
        }
    }
}

// grid.x = nchunk * n_mtiles * BH; block = m_tile / R threads, thread t with the routes t, t + block,
// ... of the tile.
template <int D, int R>
__global__ void __launch_bounds__(128 / R, simt_encode_warps(R, D) * R / 4) simt_encode_kernel(
    const float* __restrict__ k, const float* __restrict__ v, const float* __restrict__ q,
    int q_per_head, int64_t H, int64_t N, int64_t M, int64_t chunk_len, int64_t nchunk,
    int64_t n_mtiles, float sl2, float* __restrict__ pmax, float* __restrict__ psum,
    float* __restrict__ pacc) {
    __shared__ __align__(16) float ks[2][kTile<R>][D];
    __shared__ __align__(16) float vs[2][kTile<R>][D];
    tc::pdl_trigger();
    tc::pdl_wait();  // q and the partials belong to the kernels before this one

    int64_t bid = blockIdx.x;
    const int64_t c = bid % nchunk;
    bid /= nchunk;
    const int64_t mt = bid % n_mtiles;
    const int64_t bh = bid / n_mtiles;
    const int64_t m0 = mt * blockDim.x * R + threadIdx.x;

    const int64_t n_begin = c * chunk_len;
    const int64_t n_end = min(N, n_begin + chunk_len);
    const float* kb = k + bh * N * D;
    const float* vb = v + bh * N * D;
    auto stage = [&](int buf, int64_t n0) {
        stage_rows<D, kTile<R>>(ks[buf], kb, n0, n_end);
        stage_rows<D, kTile<R>>(vs[buf], vb, n0, n_end);
        copy_commit();
    };
    stage(0, n_begin);

    // query rows, pre-scaled into the base-2 domain
    f2 qr[R][D / 2], o[R][D / 2];
    float mx[R], l[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t m = m0 + r * blockDim.x;
        const bool active = m < M;
        load_row<D>(qr[r], q + ((q_per_head ? (bh % H) : bh) * M + (active ? m : 0)) * D, sl2,
                    active);
#pragma unroll
        for (int d = 0; d < D / 2; ++d) o[r][d] = 0;
        mx[r] = -INFINITY;
        l[r] = 0.f;
    }

    int buf = 0;
    for (int64_t n0 = n_begin; n0 < n_end; n0 += kTile<R>, buf ^= 1) {
        const bool more = n0 + kTile<R> < n_end;
        if (more) stage(buf ^ 1, n0 + kTile<R>);
        if (more)
            copy_wait<1>();
        else
            copy_wait<0>();
        __syncthreads();
        softmax_tile<D, R>(qr, o, mx, l, ks[buf], vs[buf], (int)min((int64_t)kTile<R>, n_end - n0));
        __syncthreads();  // this buffer is staged into again in the next step
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t m = m0 + r * blockDim.x;
        if (m < M) {
            const int64_t row = (bh * nchunk + c) * M + m;
            pmax[row] = mx[r];
            psum[row] = l[r];
            store_row<D>(pacc + row * D, o[r], 1.f);
        }
    }
}

// grid.x = ceil(N / 128) * BH; block = 128 / R threads, thread t with the tokens t, t + block, ... of
// the 128; routes staged kTile at a time.
template <int D, int R>
__global__ void __launch_bounds__(128 / R, R == 2 ? 4 : 1) simt_decode_kernel(
    const float* __restrict__ k, const float* __restrict__ q32, const float* __restrict__ z32,
    int64_t q_heads, int64_t N, int64_t M, float sl2, float* __restrict__ y,
    float* __restrict__ lse) {
    __shared__ __align__(16) float qs[2][kTile<R>][D];
    __shared__ __align__(16) float zs[2][kTile<R>][D];
    tc::pdl_trigger();
    tc::pdl_wait();  // Q and Z are written by the kernels before this one
    const int64_t ntiles = (N + 127) / 128;
    const int64_t bh = blockIdx.x / ntiles;
    const int64_t n0 = (blockIdx.x % ntiles) * 128 + threadIdx.x;
    const float* qb = q32 + bh % q_heads * M * D;  // q_heads: BH, or H when the batch shares Q
    const float* zb = z32 + bh * M * D;
    auto stage = [&](int buf, int64_t m0) {
        stage_rows<D, kTile<R>>(qs[buf], qb, m0, M);
        stage_rows<D, kTile<R>>(zs[buf], zb, m0, M);
        copy_commit();
    };
    stage(0, 0);
    f2 kr[R][D / 2], o[R][D / 2];
    float mx[R], l[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t n = n0 + r * blockDim.x;
        load_row<D>(kr[r], k + (bh * N + (n < N ? n : 0)) * D, sl2, n < N);
#pragma unroll
        for (int d = 0; d < D / 2; ++d) o[r][d] = 0;
        mx[r] = -INFINITY;
        l[r] = 0.f;
    }
    int buf = 0;
    for (int64_t m0 = 0; m0 < M; m0 += kTile<R>, buf ^= 1) {
        const bool more = m0 + kTile<R> < M;
        if (more) stage(buf ^ 1, m0 + kTile<R>);
        if (more)
            copy_wait<1>();
        else
            copy_wait<0>();
        __syncthreads();
        softmax_tile<D, R>(kr, o, mx, l, qs[buf], zs[buf], (int)min((int64_t)kTile<R>, M - m0));
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t n = n0 + r * blockDim.x;
        if (n < N) {
            store_row<D>(y + (bh * N + n) * D, o[r], 1.f / l[r]);
            if (lse) lse[bh * N + n] = mx[r] + log2f(l[r]);
        }
    }
}

inline cudaError_t encode_f32(const Plan& p, int call, const float* k, const float* v,
                              const float* seeds, float scale, char* ws, cudaStream_t st) {
    const int64_t blocks = p.nchunk * p.n_mtiles * p.BH;
    const float* q = call == 1 ? seeds : (const float*)(ws + p.off_q32);
    const int rows = simt_encode_rows(p.M, p.D);
    const auto run = [&](auto kernel) {
        return launch_pdl(kernel, dim3((unsigned)blocks), dim3((unsigned)(p.m_tile / rows)), 0, st,
                          k, v, q,
                          call == 1 ? 1 : 0, p.H, p.N, p.M, p.chunk_len, p.nchunk, p.n_mtiles,
                          scale * kLog2e, (float*)(ws + p.off_pmax), (float*)(ws + p.off_psum),
                          (float*)(ws + p.off_pacc));
    };
    switch (p.D) {
        case 16: return rows == 2 ? run(simt_encode_kernel<16, 2>) : run(simt_encode_kernel<16, 1>);
        case 32: return rows == 2 ? run(simt_encode_kernel<32, 2>) : run(simt_encode_kernel<32, 1>);
        case 64: return run(simt_encode_kernel<64, 1>);
        default: return cudaErrorInvalidValue;
    }
}

inline cudaError_t decode_f32(const Plan& p, const float* K, float scale, float* Y, char* ws,
                              cudaStream_t st, float* lse, const float* Qh) {
    const int64_t blocks = ((p.N + 127) / 128) * p.BH;
    const float* q32 = Qh ? Qh : (const float*)(ws + p.off_q32);
    // two tokens per thread (70 us for 8 x 16,384 tokens at M = 128, D = 32; one 87) once its blocks
    // take all four places that registers leave on every SM; at D = 64 two rows would spill
    const bool two = p.D <= 32 && blocks >= 4 * kNumSMs;
    const auto run = [&](auto kernel) {
        return launch_pdl(kernel, dim3((unsigned)blocks), dim3(two ? 64 : 128), 0, st, K, q32,
                          (const float*)(ws + p.off_z32), Qh ? p.H : p.BH, p.N, p.M,
                          scale * kLog2e, Y, lse);
    };
    switch (p.D) {
        case 16: return two ? run(simt_decode_kernel<16, 2>) : run(simt_decode_kernel<16, 1>);
        case 32: return two ? run(simt_decode_kernel<32, 2>) : run(simt_decode_kernel<32, 1>);
        case 64: return run(simt_decode_kernel<64, 1>);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace simt
}  // namespace flarepp

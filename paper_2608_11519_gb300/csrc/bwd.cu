// Backward of the routing chain (App. A.5): the CUDA-core passes (float32 inputs), the small
// kernels of both paths (c of call 3, the tensor-core path's prologue, the reduces of partial
// sums) and the launch sequence of both paths. The tensor-core passes are in tc_tok.cu (the token
// passes that also form dQ and dseeds), tc_kernels.cu (dZ, an encode with column statistics) and
// tc_bwd.cu (the separate passes).
//
// Every SDPA of the chain is differentiated from its saved output O and log-normaliser L:
//   P = 2^(x - L) with x = scale * log2(e) <a, b> (L kept in base 2 by the forward),
//   c = <dO, O>_D,  dS = P o (dO C^T - c),  dA = s dS B,  dB = s dS^T A,  dC = P^T dO
// for SDPA(A, B, C) with output O. The chain runs the three calls backwards:
//   call 3  Y = SDPA(K, Q, Z):   c3 per token;  dZ = P3^T dY,  dQ += s dS3^T K,  dK += s dS3 Q
//   call 2  Z = SDPA(Q, K, V):   c2 per route;  dV = P2^T dZ,  dQ += s dS2 K,    dK += s dS2^T Q
//   call 1  Q = SDPA(Qs, Kt, Vt) with the summed dQ (App. A.5: the decoder's query gradient is
//           added to the encoder's): c1 per route; dVt = P1^T dQ, dKt = s dS1^T Qs,
//           dQs = s dS1 Kt, summed over the batch for the shared seeds.
//
// Two kernel shapes cover it on CUDA cores. A route pass gives one thread per route and
// streams a chunk of tokens, accumulating the latent-side sums (dZ, dQ, dQs) into per-chunk
// partials that a reduce kernel adds in chunk order. A token pass gives two threads to one or two
// tokens and streams every route, producing that token's dK, dV (calls 2 and 3 together) or
// dKt, dVt (call 1). The tensor-core path works with bf16 copies of Q, Z, dZ and dQ as MMA operands:
// up to tok_max_routes(D) routes as dZ, the token pass of calls 3 and 2 with dQ, and the token pass of
// call 1 with dseeds; otherwise (D = 64, more routes, and heads whose log-normalisers spread too far)
// in the structure above, passes R3, T23, R2, T1, R1.
#include <cuda_bf16.h>
#include <math.h>

#include "flarepp_internal.h"
#include "simt_math.cuh"
#include "tc_ptx.cuh"

namespace flarepp {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr int kTok = 16;    // tokens staged per step of a route pass
constexpr int kRoute = 16;  // routes staged per step of a token pass

__device__ __forceinline__ float ld_f32(const float* p) { return *p; }
__device__ __forceinline__ float ld_f32(const __nv_bfloat16* p) { return __bfloat162float(*p); }

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// c3[n] = <dY_n, Y_n>: each thread reads one 16-byte vector of a row of dY and of Y (so a
// warp reads consecutive rows whole), and the D / V threads of a row add their partial dot
// products with shuffles. rows * D / V threads in all, t of them.
template <int D, typename T>
__device__ __forceinline__ void delta_token(const T* __restrict__ dY, const T* __restrict__ Y,
                                            int64_t rows, float* __restrict__ c3, int64_t t) {
    constexpr int V = 16 / (int)sizeof(T);  // elements per 16-byte vector
    constexpr int TPR = D / V;              // threads per row (2 .. 16, a power of two)
    const int64_t r = t / TPR;
    float acc = 0.f;
    if (r < rows) {
        const uint4 a = reinterpret_cast<const uint4*>(dY)[t];
        const uint4 b = reinterpret_cast<const uint4*>(Y)[t];
        const T* av = reinterpret_cast<const T*>(&a);
        const T* bv = reinterpret_cast<const T*>(&b);
#pragma unroll
        for (int e = 0; e < V; ++e) acc = fmaf(ld_f32(av + e), ld_f32(bv + e), acc);
    }
#pragma unroll
    for (int off = TPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (r < rows && (t % TPR) == 0) c3[r] = acc;
}
template <int D, typename T>
__global__ void __launch_bounds__(256) delta_tokens_kernel(const T* __restrict__ dY,
                                                           const T* __restrict__ Y, int64_t rows,
                                                           float* __restrict__ c3) {
    delta_token<D, T>(dY, Y, rows, c3, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

template <int D, typename T>
void launch_delta_tokens(const T* dY, const T* Y, int64_t rows, float* c3, cudaStream_t st) {
    constexpr int TPR = D / (16 / (int)sizeof(T));
    const int64_t threads = rows * TPR;
    delta_tokens_kernel<D, T><<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(dY, Y, rows, c3);
}

// Threads per route of the route passes: two at D = 64 in call 3, where one thread's two rows and two sums
// are 256 registers and spill (868 bytes; 8 x 16,384 tokens, M = 128: 789 us, with two 280).
constexpr int route_threads(int D, int mode) { return D == 64 && mode == 3 ? 2 : 1; }

constexpr int kFlush = 256;  // tokens that the route passes sum in registers

// Route pass of call MODE (3, 2 or 1) over one chunk of tokens, float32; thread, or pair, = route m.
//   MODE 3: a = Q, keys b = K, w = dY, g = Z, column statistics L3[n], c3[n];
//           pa += P w (dZ), pb += dS k (dQ / s)
//   MODE 2: a = Q, keys = K, w = V, g = dZ, row statistics L2[m], c2[m]; pb += dS k
//   MODE 1: a = seeds (per head), keys = Kt, w = Vt, g = dQ, row statistics L1[m], c1[m];
//           pb += dS kt
// dS here is P o (dP - c); the factor s is applied by the reduce.
// grid.x = nchunk * n_mtiles * BH; block = m_tile route_threads threads.
template <int D, int MODE>
__global__ void __launch_bounds__(128 * route_threads(D, MODE),
                                  simt_route_warps(D) / 4 / route_threads(D, MODE)) route_pass_kernel(
    const float* __restrict__ a, int a_per_head, const float* __restrict__ kb,
    const float* __restrict__ wb, const float* __restrict__ g, const float* __restrict__ Lrow,
    const float* __restrict__ crow, const float* __restrict__ Lcol,
    const float* __restrict__ ccol, int64_t H, int64_t N, int64_t M, int64_t chunk_len,
    int64_t nchunk, int64_t n_mtiles, float sl2, float* __restrict__ pa, float* __restrict__ pb) {
    using namespace simt;
    __shared__ __align__(16) float ks[2][kTok][D];
    __shared__ __align__(16) float ws[2][kTok][D];
    __shared__ float lc[2][kTok], cc[2][kTok];
    tc::pdl_trigger();
    tc::pdl_wait();

    int64_t bid = blockIdx.x;
    const int64_t c = bid % nchunk;
    bid /= nchunk;
    const int64_t mt = bid % n_mtiles;
    const int64_t bh = bid / n_mtiles;
    constexpr int P = route_threads(D, MODE);
    const int64_t m = (mt * blockDim.x + threadIdx.x) / P;
    const int h = (int)threadIdx.x % P;
    const bool active = m < M;
    const int64_t mm = active ? m : 0;
    const int64_t n_begin = c * chunk_len;
    const int64_t n_end = min(N, n_begin + chunk_len);
    auto stage = [&](int buf, int64_t n0) {
        stage_rows<D, kTok>(ks[buf], kb + bh * N * D, n0, n_end);
        stage_rows<D, kTok>(ws[buf], wb + bh * N * D, n0, n_end);
        if (MODE == 3) {
            stage_values<kTok>(lc[buf], Lcol + bh * N, n0, n_end);
            stage_values<kTok>(cc[buf], ccol + bh * N, n0, n_end);
        }
        copy_commit();
    };
    stage(0, n_begin);

    constexpr int W = D / 2 / P;  // packed pairs of channels per thread
    f2 ar[W], gr[W], accA[MODE == 3 ? W : 1], accB[W];
    const float* ap = a + ((a_per_head ? bh % H : bh) * M + mm) * D;
    const float* gp = g + (bh * M + mm) * D;
    if constexpr (P == 2) {
        load_half<D>(ar, ap, sl2, h);
        load_half<D>(gr, gp, 1.f, h);
    } else {
        load_row<D>(ar, ap, sl2, true);
        load_row<D>(gr, gp, 1.f, true);
    }
#pragma unroll
    for (int d = 0; d < W; ++d) {
        accB[d] = 0;
        if (MODE == 3) accA[d] = 0;
    }
    const float Lr = MODE == 3 ? 0.f : Lrow[bh * M + mm];
    const float cr = MODE == 3 ? 0.f : crow[bh * M + mm];

    // The sums go to the chunk's partials every kFlush tokens and start afresh: a float32 sum of hundreds
    // of terms after one another loses more than the sum of its parts (dseeds of 25 x 4,000 tokens,
    // M = 150, D = 64, in chunks of 672: 17 % more error than in chunks of 320, with this 3 % less). It
    // costs 1 % of a training step (8 x 16,384 tokens, M = 128, D = 32: 785 -> 794 us).
    const int64_t row = (bh * nchunk + c) * M + m;
    auto put = [&](float* part, f2* acc, bool first) {
        float* dst = part + row * D;
#pragma unroll
        for (int i = 0; i < W / 2; ++i) {
            float4* q = reinterpret_cast<float4*>(dst) + (P == 2 ? 2 * i + h : i);
            float4 v = first ? make_float4(0.f, 0.f, 0.f, 0.f) : *q;
            const float2 x = unpack2(acc[2 * i]), y = unpack2(acc[2 * i + 1]);
            *q = make_float4(v.x + x.x, v.y + x.y, v.z + y.x, v.w + y.y);
            acc[2 * i] = acc[2 * i + 1] = 0;
        }
    };
    int buf = 0, left = kFlush / kTok;
    bool first = true;
    for (int64_t n0 = n_begin; n0 < n_end; n0 += kTok, buf ^= 1) {
        const int cnt = (int)min((int64_t)kTok, n_end - n0);
        const bool more = n0 + kTok < n_end;
        if (more) stage(buf ^ 1, n0 + kTok);
        if (more)
            copy_wait<1>();
        else
            copy_wait<0>();
        __syncthreads();
#pragma unroll(D == 64 ? 1 : (MODE == 3 ? 2 : 8))
        for (int j = 0; j < kTok; ++j) {
            const auto weights = [&](float x, float dp, float& p, float& ds) {
                p = j < cnt ? ex2(x - (MODE == 3 ? lc[buf][j] : Lr)) : 0.f;
                ds = p * (dp - (MODE == 3 ? cc[buf][j] : cr));
            };
            float p, ds;
            if constexpr (P == 2) {
                f2 kj[W], wj[W];
                read_half<D>(kj, ks[buf][j], h);
                read_half<D>(wj, ws[buf][j], h);
                weights(dot_half<D>(ar, kj), dot_half<D>(gr, wj), p, ds);
                axpy_half<D>(accB, ds, kj);
                if (MODE == 3) axpy_half<D>(accA, p, wj);
            } else {
                weights(dot_row<D>(ar, ks[buf][j]), dot_row<D>(gr, ws[buf][j]), p, ds);
                axpy_row<D>(accB, ds, ks[buf][j]);
                if (MODE == 3) axpy_row<D>(accA, p, ws[buf][j]);
            }
        }
        if (active && (--left == 0 || !more)) {
            put(pb, accB, first);
            if (MODE == 3) put(pa, accA, first);
            first = false;
            left = kFlush / kTok;
        }
        __syncthreads();  // this buffer is staged into again in the next step
    }
}

// ---- reduces of partial sums. A row's slots are shared out to `ways` groups of D / 4 threads (four
// channels a thread; reduce_ways), way w adding the slots w, w + ways, ... in ascending order; the ways'
// sums are then added in way order.
template <int D>
unsigned reduce_blocks(int64_t rows, int ways) {
    const int64_t per_block = kRedThreads / ways / (D / 4);
    return (unsigned)((rows + per_block - 1) / per_block);
}
// This thread's row, channel group and way.
template <int D>
struct RedThread {
    int64_t row;
    int g, way;
    __device__ __forceinline__ explicit RedThread(int ways) {
        const int per = kRedThreads / ways, i = (int)threadIdx.x % per;
        way = (int)threadIdx.x / per;
        row = (int64_t)blockIdx.x * (per / (D / 4)) + i / (D / 4);
        g = i % (D / 4);
    }
};
__device__ __forceinline__ void add4(float4& a, float4 v) {
    a.x += v.x;
    a.y += v.y;
    a.z += v.z;
    a.w += v.w;
}
// The sum over the slots that next() gives, one after the other (null: no more); four loads in flight.
template <typename Next>
__device__ __forceinline__ float4 sum_slots(Next next) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (;;) {
        const float4* p[4];
        float4 v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) p[e] = next();
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = p[e] ? *p[e] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4; ++e) add4(a, v[e]);
        if (!p[3]) return a;
    }
}
// The ways' sums added in way order: valid in the threads of way 0. Every thread of the block calls it.
__device__ __forceinline__ float4 add_ways(float4 a, int ways, float4* sums) {
    if (ways == 1) return a;
    const int per = kRedThreads / ways;
    sums[threadIdx.x] = a;
    __syncthreads();
    if ((int)threadIdx.x < per)
        for (int k = 1; k < ways; ++k) add4(a, sums[threadIdx.x + k * per]);
    __syncthreads();
    return a;
}
__device__ __forceinline__ float4 scaled(float s, float4 a) {
    return make_float4(s * a.x, s * a.y, s * a.z, s * a.w);
}
// four floats as four bf16 and back
__device__ __forceinline__ uint2 pack4(float4 v) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);
    const __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                      *reinterpret_cast<const uint32_t*>(&hi));
}
__device__ __forceinline__ float4 unpack4(uint2 p) {
    const float2 f0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&p.x));
    const float2 f1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&p.y));
    return make_float4(f0.x, f0.y, f1.x, f1.y);
}
__device__ __forceinline__ void st_out4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st_out4(__nv_bfloat16* p, float4 v) {
    *reinterpret_cast<uint2*>(p) = pack4(v);
}
__device__ __forceinline__ float dot4(float4 a, float4 b) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
}
// the sum of x over a row's T threads (adjacent lanes)
template <int T>
__device__ __forceinline__ float row_sum(float x) {
    const unsigned lane = threadIdx.x & 31u;
    const unsigned mask = ((1u << T) - 1u) << (lane & ~(unsigned)(T - 1));
#pragma unroll
    for (int off = T / 2; off > 0; off >>= 1) x += __shfl_xor_sync(mask, x, off);
    return x;
}

// Reduce of the route passes' partials.
//   MODE 3: dZ = sum pa, dQ = s sum pb, c2 = <dZ, Z>
//   MODE 2: dQ += s sum pb, c1 = <dQ, Q>
//   MODE 1: dseeds[h, m] = s sum_b sum_chunks pb (rows = H * M)
// `op`, when not null, receives a bf16 copy of dZ (MODE 3) or dQ (MODE 2). In MODE 2 c1 is
// then taken from that copy: the passes of call 1 form dP = dQ K~^T from the bf16 dQ, and
// dS = P (dP - c1) cancels for a nearly one-hot P only when c1 = <dQ, Q> uses the same dQ.
template <int D, typename T, int MODE>
__global__ void __launch_bounds__(kRedThreads)
    bwd_reduce_kernel(const float* __restrict__ pa, const float* __restrict__ pb, int64_t rows,
                      int64_t B, int64_t H, int64_t M, int64_t nchunk, int ways, float scale,
                      const float* __restrict__ O, float* __restrict__ dz, float* __restrict__ dq,
                      float* __restrict__ cout, T* __restrict__ dseeds,
                      __nv_bfloat16* __restrict__ op) {
    __shared__ float4 sums[kRedThreads];
    const RedThread<D> t(ways);
    const bool in = t.row < rows;
    const int64_t bh = in ? t.row / M : 0, m = in ? t.row % M : 0;  // MODE 1: the head
    const int64_t st = M * (D / 4);
    const auto slots = [&](const float* part) {
        int64_t b = in ? 0 : B, c = t.way;
        return sum_slots([=]() mutable -> const float4* {
            if (MODE != 1) {
                if (!in || c >= nchunk) return nullptr;
            } else {
                for (; b < B && c >= nchunk; ++b) c -= nchunk;
                if (b >= B) return nullptr;
            }
            const int64_t slot = (MODE == 1 ? b * H + bh : bh) * nchunk + c;
            c += ways;
            return reinterpret_cast<const float4*>(part) + slot * st + m * (D / 4) + t.g;
        });
    };
    const float4 sb = add_ways(slots(pb), ways, sums);
    float4 sa = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MODE == 3) sa = add_ways(slots(pa), ways, sums);
    if (!in || t.way != 0) return;
    const int64_t at = t.row * D + 4 * t.g;
    if (MODE == 1) {
        st_out4(dseeds + at, scaled(scale, sb));
        return;
    }
    const float4 o = *reinterpret_cast<const float4*>(O + at);
    float4 v = scaled(scale, sb);
    float dot;
    if (MODE == 3) {
        st_out4(dz + at, sa);
        st_out4(dq + at, v);
        if (op) st_out4(op + at, sa);
        dot = dot4(sa, o);
    } else {
        add4(v, *reinterpret_cast<const float4*>(dq + at));
        st_out4(dq + at, v);
        if (op) {
            st_out4(op + at, v);
            v = unpack4(pack4(v));
        }
        dot = dot4(v, o);
    }
    dot = row_sum<D / 4>(dot);
    if (t.g == 0) cout[t.row] = dot;
}

// Token pass, float32; two threads per R tokens n, every route streamed.
//   MODE 23 (calls 3 and 2 together): keys k = K_n, w = V_n, y = dY_n; routes a = Q, g = dZ,
//     z = Z with L2, c2 per route and L3, c3 of the token:
//     x = s' <k, q_m>; P2 = 2^(x - L2_m); P3 = 2^(x - L3_n);
//     dS = P2 (<w, dz_m> - c2_m) + P3 (<y, z_m> - c3_n)
//     dK = s sum_m dS q_m;  dV = sum_m P2 dz_m
//   MODE 1: k = Kt_n, w = Vt_n; routes a = seeds (per head), g = dQ with L1, c1:
//     P1 = 2^(x - L1_m); dS = P1 (<w, dq_m> - c1_m); dKt = s sum_m dS a_m; dVt = sum_m P1 dq_m
// grid.x = ceil(N / 64 R) * BH; block = 128 threads, pair t with the tokens t, t + 64.
template <int D, int MODE, int R>
__global__ void __launch_bounds__(128) token_pass_kernel(
    const float* __restrict__ kb, const float* __restrict__ wb, const float* __restrict__ yb,
    const float* __restrict__ a, int a_per_head, const float* __restrict__ g,
    const float* __restrict__ z, const float* __restrict__ Lrow, const float* __restrict__ crow,
    const float* __restrict__ Lcol, const float* __restrict__ ccol, int64_t H, int64_t N,
    int64_t M, float sl2, float scale, float* __restrict__ dk_out, float* __restrict__ dv_out) {
    using namespace simt;
    constexpr bool kThree = MODE == 23;
    __shared__ __align__(16) float as_[2][kRoute][D];
    __shared__ __align__(16) float gs[2][kRoute][D];
    __shared__ __align__(16) float zs[2][kThree ? kRoute : 1][D];
    __shared__ float ls[2][kRoute], cs[2][kRoute];
    tc::pdl_trigger();
    tc::pdl_wait();
    const int64_t ntiles = (N + 64 * R - 1) / (64 * R);
    const int64_t bh = blockIdx.x / ntiles;
    const int h = threadIdx.x & 1;
    const int64_t nbase = (blockIdx.x % ntiles) * 64 * R + threadIdx.x / 2;
    const float* ab = a + (a_per_head ? bh % H : bh) * M * D;
    auto stage = [&](int buf, int64_t m0) {
        stage_rows<D, kRoute>(as_[buf], ab, m0, M);
        stage_rows<D, kRoute>(gs[buf], g + bh * M * D, m0, M);
        if constexpr (kThree) stage_rows<D, kRoute>(zs[buf], z + bh * M * D, m0, M);
        stage_values<kRoute>(ls[buf], Lrow + bh * M, m0, M);
        stage_values<kRoute>(cs[buf], crow + bh * M, m0, M);
        copy_commit();
    };
    stage(0, 0);
    f2 kr[R][D / 4], wr[R][D / 4], yr[R][kThree ? D / 4 : 1], dk[R][D / 4], dv[R][D / 4];
    float L3[R], c3[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t n = nbase + r * 64 < N ? nbase + r * 64 : 0;
        load_half<D>(kr[r], kb + (bh * N + n) * D, sl2, h);
        load_half<D>(wr[r], wb + (bh * N + n) * D, 1.f, h);
        if constexpr (kThree) load_half<D>(yr[r], yb + (bh * N + n) * D, 1.f, h);
#pragma unroll
        for (int d = 0; d < D / 4; ++d) dk[r][d] = dv[r][d] = 0;
        L3[r] = kThree ? Lcol[bh * N + n] : 0.f;
        c3[r] = kThree ? ccol[bh * N + n] : 0.f;
    }
    int buf = 0;
    for (int64_t m0 = 0; m0 < M; m0 += kRoute, buf ^= 1) {
        const int cnt = (int)min((int64_t)kRoute, M - m0);
        const bool more = m0 + kRoute < M;
        if (more) stage(buf ^ 1, m0 + kRoute);
        if (more)
            copy_wait<1>();
        else
            copy_wait<0>();
        __syncthreads();
#pragma unroll(D == 64 ? 1 : 8)
        for (int j = 0; j < kRoute; ++j) {
            const bool in = j < cnt;
            f2 aj[D / 4], gj[D / 4];
            read_half<D>(aj, as_[buf][j], h);
            read_half<D>(gj, gs[buf][j], h);
            float x[R], p[R], ds[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                x[r] = dot_half<D>(kr[r], aj);
                const float dp = dot_half<D>(wr[r], gj);
                p[r] = in ? ex2(x[r] - ls[buf][j]) : 0.f;
                ds[r] = p[r] * (dp - cs[buf][j]);
                axpy_half<D>(dv[r], p[r], gj);
            }
            if constexpr (kThree) {
                f2 zj[D / 4];
                read_half<D>(zj, zs[buf][j], h);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float dp3 = dot_half<D>(yr[r], zj);
                    ds[r] = fmaf(in ? ex2(x[r] - L3[r]) : 0.f, dp3 - c3[r], ds[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) axpy_half<D>(dk[r], ds[r], aj);
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t n = nbase + r * 64;
        if (n < N) {
            store_half<D>(dk_out + (bh * N + n) * D, dk[r], scale, h);
            store_half<D>(dv_out + (bh * N + n) * D, dv[r], 1.f, h);
        }
    }
}

template <int D>
cudaError_t route_bwd_d(const Plan& p, const BwdPlan& bp, const float* seeds, const float* Kt,
                        const float* Vt, const float* K, const float* V, float scale, const float* Y,
                        const float* dY, const char* saved, float* dseeds, float* dKt, float* dVt, float* dK,
                        float* dV, char* ws, cudaStream_t st) {
    const SavedLayout sl = saved_layout(p);
    const float* Q32 = (const float*)(saved + sl.off_q);
    const float* Z32 = (const float*)(saved + sl.off_z);
    const float* L1 = (const float*)(saved + sl.off_l1);
    const float* L2 = (const float*)(saved + sl.off_l2);
    const float* L3 = (const float*)(saved + sl.off_l3);
    float* pa = (float*)(ws + bp.off_pa);
    float* pb = (float*)(ws + bp.off_pb);
    float* dz = (float*)(ws + bp.off_dz);
    float* dq = (float*)(ws + bp.off_dq);
    float* c1 = (float*)(ws + bp.off_d1);
    float* c2 = (float*)(ws + bp.off_d2);
    float* c3 = (float*)(ws + bp.off_d3);
    const float sl2 = scale * kLog2e;
    const int64_t tok_rows = p.BH * p.N;
    const int64_t lat_rows = p.BH * p.M;
    const unsigned route_blocks = (unsigned)(bp.nchunk * bp.n_mtiles * p.BH);
    // One route per thread in the route passes: pairs of threads with one or two routes are slower (8 x
    // 16,384 tokens, M = 128, D = 32: 132 or 140 us for call 3, 98 or 93 for calls 2 and 1; this 108 and 84).
    constexpr int kTwo = D <= 32 ? 2 : 1;
    const bool two23 = simt_two_tokens(D, false, p.N, p.BH), two1 = simt_two_tokens(D, true, p.N, p.BH);
    const int64_t seed_rows = p.H * p.M;
    const int ways = reduce_ways(lat_rows, D, bp.nchunk);
    const int seed_ways = reduce_ways(seed_rows, D, p.B * bp.nchunk);
    const unsigned red_blocks = reduce_blocks<D>(lat_rows, ways);

    launch_delta_tokens<D, float>(dY, Y, tok_rows, c3, st);
    const auto route = [&](auto kernel, int per_route, const float* a, int per_head, const float* k,
                           const float* w, const float* g, const float* Lr, const float* cr) {
        return launch_pdl(kernel, dim3(route_blocks), dim3((unsigned)(bp.m_tile * per_route)), 0, st, a,
                          per_head, k, w, g, Lr, cr, (const float*)L3, (const float*)c3, p.H, p.N,
                          p.M, bp.chunk_len, bp.nchunk, bp.n_mtiles, sl2, pa, pb);
    };
    const auto token = [&](auto kernel, bool two, const float* k, const float* w, const float* y,
                           const float* a, int per_head, const float* g, const float* z,
                           const float* Lr, const float* cr, float* o0, float* o1) {
        const unsigned blocks = (unsigned)((two ? (p.N + 127) / 128 : (p.N + 63) / 64) * p.BH);
        return launch_pdl(kernel, dim3(blocks), dim3(128), 0, st, k, w, y, a, per_head, g, z,
                          Lr, cr, (const float*)L3, (const float*)c3, p.H, p.N, p.M, sl2, scale, o0,
                          o1);
    };
    const float* none = nullptr;
    cudaError_t e;
    // call 3: dZ and the decoder's dQ
    if ((e = route(route_pass_kernel<D, 3>, route_threads(D, 3), Q32, 0, K, dY, Z32, none, none)) !=
        cudaSuccess)
        return e;
    bwd_reduce_kernel<D, float, 3><<<red_blocks, kRedThreads, 0, st>>>(
        pa, pb, lat_rows, p.B, p.H, p.M, bp.nchunk, ways, scale, Z32, dz, dq, c2, nullptr, nullptr);
    // calls 3 and 2: dK and dV per token
    if ((e = token(two23 ? token_pass_kernel<D, 23, kTwo> : token_pass_kernel<D, 23, 1>, two23, K, V,
                   dY, Q32, 0, dz, Z32, L2, c2, dK, dV)) != cudaSuccess)
        return e;
    // call 2: the encoder's dQ, added to the decoder's
    if ((e = route(route_pass_kernel<D, 2>, route_threads(D, 2), Q32, 0, K, V, dz, L2, c2)) !=
        cudaSuccess)
        return e;
    bwd_reduce_kernel<D, float, 2><<<red_blocks, kRedThreads, 0, st>>>(
        nullptr, pb, lat_rows, p.B, p.H, p.M, bp.nchunk, ways, scale, Q32, nullptr, dq, c1, nullptr,
        nullptr);
    // call 1: dKt, dVt per token, then the seeds' gradient
    if ((e = token(two1 ? token_pass_kernel<D, 1, kTwo> : token_pass_kernel<D, 1, 1>, two1, Kt, Vt,
                   none, seeds, 1, dq, none, L1, c1, dKt, dVt)) != cudaSuccess)
        return e;
    if ((e = route(route_pass_kernel<D, 1>, route_threads(D, 1), seeds, 1, Kt, Vt, dq, L1, c1)) !=
        cudaSuccess)
        return e;
    bwd_reduce_kernel<D, float, 1>
        <<<reduce_blocks<D>(seed_rows, seed_ways), kRedThreads, 0, st>>>(
            nullptr, pb, seed_rows, p.B, p.H, p.M, bp.nchunk, seed_ways, scale, nullptr, nullptr,
            nullptr, nullptr, dseeds, nullptr);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- the merged T23 pass
// T23C (tc_bwd.cu) multiplies V and dZ scaled by u = 2^(L3[n] - R) and w = 2^(R - L2[m])
// for one shift R per (b, h). With R = min_m L2 both scales stay within 2^kMergeRange
// whenever max_n L3 - R and max_m L2 - R do; a (b, h) outside that range (scores spread
// over more than ~60 binary orders) is flagged and runs the unmerged T23 pass instead.
constexpr float kMergeRange = 60.f;

// part[bh][j] for j < parts: max of L3 over slice j of the tokens; part[bh][kRangeParts] and
// [kRangeParts + 1]: min and max of L2 (from slice 0's block). One block per (bh, j), block `id`.
__device__ __forceinline__ void merge_range(const float* __restrict__ L2,
                                            const float* __restrict__ L3, int64_t M, int64_t N,
                                            int parts, int64_t id, float* __restrict__ part) {
    __shared__ float red[3][8];
    const int64_t bh = id / parts;
    const int j = (int)(id % parts);
    const int64_t per = (N + parts - 1) / parts;
    const int64_t n0 = j * per, n1 = min(N, n0 + per);
    float mx3 = -INFINITY, mn2 = INFINITY, mx2 = -INFINITY;
#pragma unroll 8
    for (int64_t n = n0 + threadIdx.x; n < n1; n += blockDim.x) mx3 = fmaxf(mx3, L3[bh * N + n]);
    if (j == 0)
        for (int64_t m = threadIdx.x; m < M; m += blockDim.x) {
            const float x = L2[bh * M + m];
            mn2 = fminf(mn2, x);
            mx2 = fmaxf(mx2, x);
        }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        mx3 = fmaxf(mx3, __shfl_xor_sync(0xffffffffu, mx3, off));
        mn2 = fminf(mn2, __shfl_xor_sync(0xffffffffu, mn2, off));
        mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, off));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = mx3;
        red[1][w] = mn2;
        red[2][w] = mx2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            mx3 = fmaxf(mx3, red[0][k]);
            mn2 = fminf(mn2, red[1][k]);
            mx2 = fmaxf(mx2, red[2][k]);
        }
        float* o = part + bh * (kRangeParts + 2);
        o[j] = mx3;
        if (j == 0) {
            o[kRangeParts] = mn2;
            o[kRangeParts + 1] = mx2;
        }
    }
}
// slices of the tokens: 4096 each (16 loads per thread), at most kRangeParts
inline int range_parts(int64_t N) {
    const int64_t n = (N + 4095) / 4096;
    return (int)(n < kRangeParts ? n : kRangeParts);
}

// Everything that the tensor-core backward needs ahead of its passes, none of it depending on the
// rest: the slices' ranges for the merged pass (blocks [0, BH * parts); none when parts is 0), the
// bf16 operands of Q (with its lo part when lo is given, as the training forward took it) and Z (the
// next `cvt` blocks), and c3 (the rest, bound by the reads of dY and Y). Block 0 also clears the word
// behind the flags. One launch: as four they took 25 us at 32 (b, h) of 16,384 tokens, D = 32, this
// 13.
template <int D>
__global__ void __launch_bounds__(256) bwd_prologue_kernel(
    const __nv_bfloat16* __restrict__ dY, const __nv_bfloat16* __restrict__ Y, int64_t rows,
    float* __restrict__ c3, const float* __restrict__ Q, const float* __restrict__ Z, int64_t lat,
    __nv_bfloat16* __restrict__ qb, __nv_bfloat16* __restrict__ qlo, __nv_bfloat16* __restrict__ zb,
    unsigned cvt, const float* __restrict__ L2, const float* __restrict__ L3, int64_t BH, int64_t M,
    int64_t N, int parts, float* __restrict__ rpart, int* __restrict__ any) {
    tc::pdl_trigger();
    int64_t id = blockIdx.x;
    if (any != nullptr && id == 0 && threadIdx.x == 0) *any = 0;
    if (id < BH * parts) {
        merge_range(L2, L3, M, N, parts, id, rpart);
        return;
    }
    id -= BH * parts;
    if (id < cvt) {
        for (int64_t i = id * 256 + threadIdx.x; i < lat / 4; i += (int64_t)cvt * 256) {
            const float4 q = reinterpret_cast<const float4*>(Q)[i];
            const uint2 hi = pack4(q);
            reinterpret_cast<uint2*>(qb)[i] = hi;
            if (qlo != nullptr) {
                const float4 h = unpack4(hi);
                reinterpret_cast<uint2*>(qlo)[i] =
                    pack4(make_float4(q.x - h.x, q.y - h.y, q.z - h.z, q.w - h.w));
            }
            reinterpret_cast<uint2*>(zb)[i] = pack4(reinterpret_cast<const float4*>(Z)[i]);
        }
        return;
    }
    id -= cvt;
    delta_token<D>(dY, Y, rows, c3, id * 256 + threadIdx.x);
}

// R[bh] = min_m L2; flags[bh] = 1 when the (b, h) runs the unmerged pass, and then flags[BH] = 1.
__device__ __forceinline__ void merge_flag(const float* __restrict__ part, int parts, int64_t bh,
                                           int64_t BH, float* __restrict__ Rb,
                                           int* __restrict__ flags) {
    const float* o = part + bh * (kRangeParts + 2);
    float mx3 = -INFINITY;
#pragma unroll 8
    for (int j = 0; j < parts; ++j) mx3 = fmaxf(mx3, o[j]);
    const float R = o[kRangeParts], mx2 = o[kRangeParts + 1];
    Rb[bh] = R;
    const bool fits = mx3 - R <= kMergeRange && mx2 - R <= kMergeRange;
    flags[bh] = fits ? 0 : 1;
    if (!fits) atomicOr(flags + BH, 1);
}
__global__ void merge_flags_kernel(const float* __restrict__ part, int parts, int64_t BH,
                                   float* __restrict__ Rb, int* __restrict__ flags) {
    const int64_t bh = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (bh < BH) merge_flag(part, parts, bh, BH, Rb, flags);
}

// The merged pass's route operand w dZ: W[bh][m][:] = bf16(2^(R[bh] - L2[bh][m]) dZ[bh][m][:]), and
// c2 taken from it: c2w = <W, Z> / w. The pass forms w dP2 = W V^T, and dS2 = P2 (dP2 - c2)
// cancels for a nearly one-hot P2 only when c2 sees the same rounded dZ. v, z: this thread's four
// channels (group g of D / 4) of the row of dZ and Z.
template <int D>
__device__ __forceinline__ void merge_operand(float4 v, float4 z, float e, int64_t row, int g,
                                              __nv_bfloat16* W, float* c2w) {
    const float w = exp2f(e);
    const uint2 pk = pack4(make_float4(w * v.x, w * v.y, w * v.z, w * v.w));
    reinterpret_cast<uint2*>(W + row * D)[g] = pk;
    const float dot = row_sum<D / 4>(dot4(unpack4(pk), z));
    if (g == 0) c2w[row] = dot * exp2f(-e);
}

template <int D>
__global__ void __launch_bounds__(256)
    merge_operand_kernel(const float* __restrict__ dz, const float* __restrict__ Z,
                         const float* __restrict__ L2, const float* __restrict__ Rb, int64_t M,
                         int64_t rows, __nv_bfloat16* __restrict__ W, float* __restrict__ c2w) {
    constexpr int T = D / 4;
    const int64_t row = ((int64_t)blockIdx.x * 256 + threadIdx.x) / T;  // bh * M + m
    const int g = threadIdx.x % T;
    if (row >= rows) return;  // (rows in whole groups of T threads)
    merge_operand<D>(reinterpret_cast<const float4*>(dz + row * D)[g],
                     reinterpret_cast<const float4*>(Z + row * D)[g], Rb[row / M] - L2[row], row, g,
                     W, c2w);
}

// dZ from the partial sums of tc_dz_pass (a chunk's token-parity parts as the encode's plan cuts them: 4,
// 2 or 1 by the route tiles of the row's group of 512): its bf16 copy, c2 = <dZ, Z>, and the merged
// pass's operand; and the (b, h)'s shift and flag.
template <int D>
__global__ void __launch_bounds__(kRedThreads)
    dz_reduce_kernel(const float* __restrict__ part, int M, int nchunk, int64_t rows, int ways,
                     const float* __restrict__ Z, const float* __restrict__ L2,
                     const float* __restrict__ rpart, int parts, float* __restrict__ Rb,
                     int* __restrict__ flags, __nv_bfloat16* __restrict__ dzb,
                     float* __restrict__ c2, __nv_bfloat16* __restrict__ W,
                     float* __restrict__ c2w) {
    __shared__ float4 sums[kRedThreads];
    tc::pdl_trigger();
    tc::pdl_wait();
    const RedThread<D> t(ways);
    const bool in = t.row < rows;
    const int64_t bh = in ? t.row / M : 0;  // row = bh * M + m
    const int m = in ? (int)(t.row - bh * M) : 0;
    if (in && m == 0 && t.g == 0 && t.way == 0) merge_flag(rpart, parts, bh, rows / M, Rb, flags);
    const int left = M - (m & ~511);
    const int ul = left > 256 ? 0 : (left > 128 ? 1 : 2);  // log2 of the parts per chunk
    const int n = in ? nchunk << ul : 0, mask = (1 << ul) - 1;
    const float4* p = reinterpret_cast<const float4*>(part + (bh * nchunk * 4 * M + m) * D) + t.g;
    const int64_t st = (int64_t)M * (D / 4);
    int s = t.way;
    float4 a = sum_slots([=]() mutable -> const float4* {
        if (s >= n) return nullptr;
        const float4* q = p + ((int64_t)(s >> ul) * 4 + (s & mask)) * st;
        s += ways;
        return q;
    });
    a = add_ways(a, ways, sums);
    if (!in || t.way != 0) return;
    const int64_t at = t.row * D + 4 * t.g;
    const float4 z = *reinterpret_cast<const float4*>(Z + at);
    st_out4(dzb + at, a);
    const float dot = row_sum<D / 4>(dot4(a, z));
    if (t.g == 0) c2[t.row] = dot;
    merge_operand<D>(a, z, rpart[bh * (kRangeParts + 2) + kRangeParts] - L2[t.row], t.row, t.g, W,
                     c2w);
}

// Reduce of the partials dS^T K that the token passes of tc_tok.cu leave, a CTA's slot each, in CTA
// order.
//   DSEEDS false: dQ = s sum (of the flagged (b, h) s times the sum of the route passes' partials,
//     pb of R3 and pa of R2, nchunk each), as bf16, and c1 = <dQ, Q> from that copy (as
//     bwd_reduce_kernel's MODE 2)
//   DSEEDS true: dseeds[h, m] = s sum over the batch and the slots (rows = H * M)
template <int D, bool DSEEDS>
__global__ void __launch_bounds__(kRedThreads)
    tok_reduce_kernel(const float* __restrict__ part, int64_t rows, int64_t B, int64_t H, int64_t M,
                      int64_t nt, int64_t tiles, int64_t ctas, int64_t slots, int ways, float scale,
                      const int* __restrict__ flags, const float* __restrict__ pb,
                      const float* __restrict__ pa, int64_t nchunk, const float* __restrict__ Q,
                      float* __restrict__ c1, __nv_bfloat16* __restrict__ op) {
    __shared__ float4 sums[kRedThreads];
    tc::pdl_trigger();
    tc::pdl_wait();
    const RedThread<D> t(ways);
    const bool in = t.row < rows;
    const int64_t hb = in ? t.row / M : 0, m = in ? t.row % M : 0;  // DSEEDS: the head, else bh
    const int64_t st = M * (D / 4);
    // the slots of (b, h): one per CTA whose run of tiles reaches it
    const auto count = [=](int64_t bh) {
        return ((bh + 1) * nt * ctas - 1) / tiles - ((bh * nt + 1) * ctas - 1) / tiles + 1;
    };
    const auto at_slot = [=](const float* base, int64_t slot) {
        return reinterpret_cast<const float4*>(base) + slot * st + m * (D / 4) + t.g;
    };
    float4 a;
    if (DSEEDS) {
        int64_t b = 0, s = t.way, n = in ? count(hb) : 0;
        a = sum_slots([=]() mutable -> const float4* {
            while (s >= n) {  // on to the next batch element
                s -= n;
                if (!in || ++b >= B) {
                    n = 0;
                    s = 0;
                    return nullptr;
                }
                n = count(b * H + hb);
            }
            const float4* q = at_slot(part, (b * H + hb) * slots + s);
            s += ways;
            return q;
        });
    } else {
        const bool flagged = flags != nullptr && in && flags[hb] != 0;
        const int64_t n = !in ? 0 : (flagged ? 2 * nchunk : count(hb));
        int64_t s = t.way;
        a = sum_slots([=]() mutable -> const float4* {
            if (s >= n) return nullptr;
            const float4* q = !flagged ? at_slot(part, hb * slots + s)
                              : s < nchunk ? at_slot(pb, hb * nchunk + s)
                                           : at_slot(pa, hb * nchunk + s - nchunk);
            s += ways;
            return q;
        });
    }
    a = add_ways(a, ways, sums);
    if (!in || t.way != 0) return;
    const int64_t at = t.row * D + 4 * t.g;
    const uint2 pk = pack4(scaled(scale, a));
    *reinterpret_cast<uint2*>(op + at) = pk;
    if (!DSEEDS) {
        const float dot =
            row_sum<D / 4>(dot4(unpack4(pk), *reinterpret_cast<const float4*>(Q + at)));
        if (t.g == 0) c1[t.row] = dot;
    }
}

// The tensor-core path (bf16 inputs): the prologue, then R3 -> reduce (dZ, the decoder's dQ, c2) ->
// T23 (dK, dV) and R2 -> reduce (dQ, c1) -> T1 (dKt, dVt) and R1 -> reduce (dseeds). For D <= 32,
// T23 runs merged (T23C) for every (b, h) whose statistics allow it and unmerged for the rest; and
// where the routes fit (tok_max_routes), dZ comes from an encode and the token passes of tc_tok.cu
// form dQ and dseeds as well: R3, T23 and R2 then run for the flagged (b, h) alone.
template <int D>
cudaError_t route_bwd_tc_d(const Plan& p, const BwdPlan& bp, const void* seeds, const void* Kt,
                           const void* Vt, const void* K, const void* V, float scale,
                           const void* Y, const void* dY, const char* saved, void* dseeds,
                           void* dKt, void* dVt, void* dK, void* dV, char* ws, cudaStream_t st) {
    using T = __nv_bfloat16;
    const SavedLayout sl = saved_layout(p);
    const float* Q32 = (const float*)(saved + sl.off_q);
    const float* Z32 = (const float*)(saved + sl.off_z);
    const float* L1 = (const float*)(saved + sl.off_l1);
    const float* L2 = (const float*)(saved + sl.off_l2);
    const float* L3 = (const float*)(saved + sl.off_l3);
    float* pa = (float*)(ws + bp.off_pa);
    float* pb = (float*)(ws + bp.off_pb);
    float* dz = (float*)(ws + bp.off_dz);
    float* dq = (float*)(ws + bp.off_dq);
    float* c1 = (float*)(ws + bp.off_d1);
    float* c2 = (float*)(ws + bp.off_d2);
    float* c3 = (float*)(ws + bp.off_d3);
    T* qb = (T*)(ws + bp.off_qb);
    T* zb = (T*)(ws + bp.off_zb);
    T* dzb = (T*)(ws + bp.off_dzb);
    T* dqb = (T*)(ws + bp.off_dqb);
    T* wop = (T*)(ws + bp.off_w);
    float* c2w = (float*)(ws + bp.off_c2w);
    float* Rb = (float*)(ws + bp.off_rb);
    int* flags = (int*)(ws + bp.off_flags);
    float* rpart = (float*)(ws + bp.off_rpart);
    int* status = (int*)(ws + bp.off_status);
    const int64_t tok_rows = p.BH * p.N;
    const int64_t lat_rows = p.BH * p.M;
    const int64_t lat = lat_rows * p.D;
    const int64_t seed_rows = p.H * p.M;
    cudaError_t e;

    constexpr bool kMerged = D <= 32;
    // Q as the training forward gave it to calls 2 and 3: a hi/lo pair for D <= 32
    T* qlo = kMerged ? (T*)(ws + bp.off_qlo) : nullptr;
    const int parts = kMerged ? range_parts(p.N) : 0;
    const unsigned cvt = (unsigned)min((int64_t)kNumSMs, (lat / 4 + 255) / 256);
    const int64_t delta = (tok_rows * (D / 8) + 255) / 256;
    bwd_prologue_kernel<D><<<(unsigned)(p.BH * parts + cvt + delta), 256, 0, st>>>(
        (const T*)dY, (const T*)Y, tok_rows, c3, Q32, Z32, lat, qb, qlo, zb, cvt, L2, L3, p.BH, p.M,
        p.N, parts, rpart, kMerged ? flags + p.BH : nullptr);
    if (kMerged && bp.tok_slots == 0)
        merge_flags_kernel<<<(unsigned)((p.BH + 127) / 128), 128, 0, st>>>(rpart, parts, p.BH, Rb,
                                                                            flags);
    // R3: route rows; S = Q K^T, dP = Z dY^T; column statistics L3, c3 -> dQ3, dZ partials
    TcBwdOperands r3{{qb, zb, zb}, {K, dY, dY}, nullptr, nullptr, L3, c3, pa, pb, nullptr, nullptr};
    r3.lo = qlo;
    // T23: token rows; S = K Q^T, dP2 = V dZ^T, dP3 = dY Z^T -> dK, dV
    TcBwdOperands t23{{K, V, dY}, {qb, dzb, zb}, L3, c3, L2, c2, nullptr, nullptr, dK, dV};
    t23.lo = qlo;
    // R2: route rows; S = Q K^T, dP = dZ V^T; row statistics L2, c2 -> dQ2 partials
    TcBwdOperands r2{{qb, dzb, dzb}, {K, V, V}, L2, c2, nullptr, nullptr, nullptr, pb, nullptr,
                     nullptr};
    r2.lo = qlo;
    if constexpr (kMerged) {
        t23.flags = flags;  // the flagged (b, h) run the unmerged T23
        t23.want = 1;
        t23.any = flags + p.BH;
        if (bp.tok_slots > 0) {
            // dZ as an encode of K and dY, then the token passes that also form dQ and dseeds;
            // the flagged (b, h) take R3 (for its dQ3), T23 and R2 (its dQ2 partials go to pa,
            // which R3's dZ does not need here)
            float* pz = (float*)(ws + bp.off_pz);
            float* pt = (float*)(ws + bp.off_pt);
            const int64_t tiles = bp.tok_nt * p.BH;
            // (the slots that rows have at most: four token parities a chunk; the CTAs' in all)
            const int ways_z = reduce_ways(lat_rows, D, p.nchunk * 4);
            const int ways_q = reduce_ways(lat_rows, D, bp.tok_slots);
            const int ways_s = reduce_ways(seed_rows, D, bp.tok_slots * p.B);
            const dim3 threads(kRedThreads);
            r3.flags = r2.flags = flags;
            r3.want = r2.want = 1;
            r3.any = r2.any = flags + p.BH;
            r2.pb = pa;
            if ((e = tc_dz_pass(p, qb, qlo, K, dY, L3, scale, pz, status, st)) != cudaSuccess)
                return e;
            if ((e = launch_pdl(dz_reduce_kernel<D>, dim3(reduce_blocks<D>(lat_rows, ways_z)), threads,
                                0, st, (const float*)pz, (int)p.M, (int)p.nchunk, lat_rows, ways_z,
                                Z32, L2,
                                (const float*)rpart, parts, Rb, flags, dzb, c2, wop, c2w)) !=
                cudaSuccess)
                return e;
            TokOperands t{{K, V, dY}, {qb, wop, zb}, qlo, L3, c3, L2, c2w, Rb, flags, pt, dK, dV};
            if ((e = tc_tok_pass(p, bp, false, t, scale, status, st)) != cudaSuccess) return e;
            if ((e = tc_bwd_pass(p, bp, 0, r3, scale, status, st)) != cudaSuccess) return e;
            if ((e = tc_bwd_pass(p, bp, 3, t23, scale, status, st)) != cudaSuccess) return e;
            if ((e = tc_bwd_pass(p, bp, 1, r2, scale, status, st)) != cudaSuccess) return e;
            if ((e = launch_pdl(tok_reduce_kernel<D, false>,
                                dim3(reduce_blocks<D>(lat_rows, ways_q)), threads, 0, st,
                                (const float*)pt, lat_rows, p.B, p.H, p.M, bp.tok_nt, tiles,
                                bp.tok_ctas, bp.tok_slots, ways_q, scale, (const int*)flags,
                                (const float*)pb, (const float*)pa, bp.nchunk, Q32, c1, dqb)) !=
                cudaSuccess)
                return e;
            t = TokOperands{{Kt, Vt, Vt}, {seeds, dqb, dqb}, nullptr, nullptr, nullptr, L1, c1,
                            nullptr, nullptr, pt, dKt, dVt};
            if ((e = tc_tok_pass(p, bp, true, t, scale, status, st)) != cudaSuccess) return e;
            return launch_pdl(tok_reduce_kernel<D, true>,
                              dim3(reduce_blocks<D>(seed_rows, ways_s)), threads, 0, st,
                              (const float*)pt, seed_rows, p.B, p.H, p.M, bp.tok_nt, tiles,
                              bp.tok_ctas, bp.tok_slots, ways_s, scale, (const int*)nullptr,
                              (const float*)nullptr, (const float*)nullptr, (int64_t)0,
                              (const float*)nullptr, (float*)nullptr, (T*)dseeds);
        }
    }
    TcBwdOperands o{};
    if ((e = tc_bwd_pass(p, bp, 0, r3, scale, status, st)) != cudaSuccess) return e;
    const int ways = reduce_ways(lat_rows, D, bp.nchunk);
    const int seed_ways = reduce_ways(seed_rows, D, p.B * bp.nchunk);
    const unsigned red_blocks = reduce_blocks<D>(lat_rows, ways);
    bwd_reduce_kernel<D, T, 3><<<red_blocks, kRedThreads, 0, st>>>(
        pa, pb, lat_rows, p.B, p.H, p.M, bp.nchunk, ways, scale, Z32, dz, dq, c2, nullptr, dzb);
    if constexpr (kMerged) {
        merge_operand_kernel<D><<<(unsigned)((lat / 4 + 255) / 256), 256, 0, st>>>(
            dz, Z32, L2, Rb, p.M, lat_rows, wop, c2w);
        // T23C: S = K Q^T, T = dY Z^T + (u V) (w dZ)^T
        TcBwdOperands om{{K, dY, V}, {qb, wop, zb}, L3, c3, L2, c2w, nullptr, nullptr, dK, dV};
        om.Rb = Rb;
        om.flags = flags;
        om.want = 0;
        om.lo = qlo;
        if ((e = tc_bwd_pass(p, bp, 5, om, scale, status, st)) != cudaSuccess) return e;
    }
    if ((e = tc_bwd_pass(p, bp, 3, t23, scale, status, st)) != cudaSuccess) return e;
    if ((e = tc_bwd_pass(p, bp, 1, r2, scale, status, st)) != cudaSuccess) return e;
    bwd_reduce_kernel<D, T, 2><<<red_blocks, kRedThreads, 0, st>>>(
        nullptr, pb, lat_rows, p.B, p.H, p.M, bp.nchunk, ways, scale, Q32, nullptr, dq, c1, nullptr,
        dqb);
    // T1: token rows; S = Kt Qs^T, dP = Vt dQ^T; column statistics L1, c1 -> dKt, dVt
    o = TcBwdOperands{{Kt, Vt, Vt}, {seeds, dqb, dqb}, nullptr, nullptr, L1, c1, nullptr,
                      nullptr, dKt, dVt};
    if ((e = tc_bwd_pass(p, bp, 4, o, scale, status, st)) != cudaSuccess) return e;
    // R1: route rows; S = Qs Kt^T, dP = dQ Vt^T; row statistics L1, c1 -> dQs partials
    o = TcBwdOperands{{seeds, dqb, dqb}, {Kt, Vt, Vt}, L1, c1, nullptr, nullptr, nullptr, pb,
                      nullptr, nullptr};
    if ((e = tc_bwd_pass(p, bp, 2, o, scale, status, st)) != cudaSuccess) return e;
    bwd_reduce_kernel<D, T, 1><<<reduce_blocks<D>(seed_rows, seed_ways), kRedThreads, 0, st>>>(
        nullptr, pb, seed_rows, p.B, p.H, p.M, bp.nchunk, seed_ways, scale, nullptr, nullptr, nullptr,
        nullptr, (T*)dseeds, nullptr);
    return cudaGetLastError();
}

cudaError_t route_bwd_f32(const Plan& p, const BwdPlan& bp, const void* seeds, const void* Kt,
                          const void* Vt, const void* K, const void* V, float scale, const void* Y,
                          const void* dY, const char* saved, void* dseeds, void* dKt, void* dVt,
                          void* dK, void* dV, char* ws, cudaStream_t st) {
    const auto f = [](const void* x) { return (const float*)x; };
    const auto o = [](void* x) { return (float*)x; };
#define FLAREPP_BWD(DD)                                                                     \
    return route_bwd_d<DD>(p, bp, f(seeds), f(Kt), f(Vt), f(K), f(V), scale, f(Y), f(dY), saved, \
                           o(dseeds), o(dKt), o(dVt), o(dK), o(dV), ws, st);
    switch (p.D) {
        case 16: FLAREPP_BWD(16)
        case 32: FLAREPP_BWD(32)
        case 64: FLAREPP_BWD(64)
        default: return cudaErrorInvalidValue;
    }
#undef FLAREPP_BWD
}

}  // namespace

cudaError_t route_bwd(const Plan& p, const BwdPlan& bp, const void* seeds, const void* Kt,
                      const void* Vt, const void* K, const void* V, float scale, const void* Y,
                      const void* dY, const char* saved, void* dseeds, void* dKt, void* dVt,
                      void* dK, void* dV, char* ws, cudaStream_t st) {
    if (bp.path == kPathTc) {
#define FLAREPP_TCBWD(DD)                                                                     \
    return route_bwd_tc_d<DD>(p, bp, seeds, Kt, Vt, K, V, scale, Y, dY, saved, dseeds, dKt, \
                              dVt, dK, dV, ws, st);
        switch (p.D) {
            case 16: FLAREPP_TCBWD(16)
            case 32: FLAREPP_TCBWD(32)
            case 64: FLAREPP_TCBWD(64)
            default: return cudaErrorInvalidValue;
        }
#undef FLAREPP_TCBWD
    }
    return route_bwd_f32(p, bp, seeds, Kt, Vt, K, V, scale, Y, dY, saved, dseeds, dKt, dVt, dK, dV,
                         ws, st);
}

}  // namespace flarepp

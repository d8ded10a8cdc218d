// Tensor-core (tcgen05 / TMEM / TMA) weight-gradient GEMM of the mixer's backward:
//   dW[r][c] = sum over tokens t of A(t, r) B(t, c)
// (dWo = dO^T merge(Y), dW_in = dP^T X, the backward of O = merge(Y) Wo^T and of
// K, V, K~, V~ = X W_in^T in Fig. 1). Both operands are token-major in memory, so the
// contraction runs over tokens with MN-major operand tiles: each tile is a set of D-wide
// channel columns ("atoms") of 64 tokens x D channels each, swizzled to the D-wide row like
// every other operand of the library. A tile arrives as four-dimensional TMA boxes
// {D channels, 64 tokens, atoms, 1} (the atom dimension steps over heads, or over the D-wide
// column blocks of a plain matrix): one box per tile, or one per atom where a tile of a
// HEADS source would cross from one tensor into the next. Few large boxes instead of one
// per atom took dW_in from 1.20 to about 0.3 ms at mesh3d. A channel source is either
//   HEADS: up to four tensors [B*H][N][D] side by side (channel r: tensor r / C, head
//          (r % C) / D, column r % D), or
//   PLAIN: one matrix [B][N][C] (channel r: column r).
// A work item is (256 rows of dW, NT columns of dW, a chunk of the tokens: a run of 64-token stages that
// may reach over several batch elements), the rows as two halves of 128 that share B's tile, each with an accumulator of its own: the reads
// bound the kernel, and with 128 rows every tile of B is fetched twice as often (dW_in of 262,144
// tokens, C = 256, four projections: 164 -> 128 us; HBM's bytes alone 99). The item writes its
// float32 partial sum to part[chunk][R][Cc], and a reduce kernel adds the chunks (in a fixed order:
// deterministic).
//
// Roles (8 warps): warp 0 the TMA producer, warp 1 the MMA issuer, warps 4..7 the epilogue
// (TMEM lane = row of dW). There is about one item per SM where the tiles allow (wgrad_plan), so that
// nothing is left to overlap an item's epilogue with and the partial sums are few. Every wait is bounded (2 s of %globaltimer), as
// in the other kernels.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <math.h>
#include <mutex>

#include "flarepp_internal.h"
#include "tc_ptx.cuh"

namespace flarepp {
namespace {

using namespace tc;

constexpr int kThreads = 256;
constexpr int kFirstEpiWarp = 4;
constexpr int kRowsW = 128;   // rows of dW per half of an item (TMEM lanes, MMA M)
constexpr int kHalves = 2;    // halves per item, at most
constexpr int kMaxNT = 256;   // columns of dW per item, at most
constexpr int kTok = 64;      // tokens per pipeline stage (four K = 16 steps)
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr uint32_t kTmemCols = 512;

template <int D>
struct WCfg {
    static constexpr int kAtom = kTok * D * 2;  // one 64-token x D column, swizzled
    static constexpr int kAStage = (kRowsW / D) * kAtom;
    static constexpr int kBStage = (kMaxNT / D) * kAtom;
    static constexpr int kStage = kHalves * kAStage + kBStage;
    static constexpr int kStages = (192 * 1024) / kStage > 6 ? 6 : (192 * 1024) / kStage;
    static constexpr uint32_t kSwz = D == 16 ? kSw32 : (D == 32 ? kSw64 : kSw128);
    static constexpr uint32_t kSBO = 8 * D * 2;  // 8-token groups along K
    static constexpr int kNumBars = 2 * kStages + 4 + 1;
    static constexpr int kNeed = 1024 + kStages * kStage + kNumBars * 8 + 16;
    static constexpr int kSmem = kNeed > 122880 ? kNeed : 122880;  // one CTA per SM
    static_assert(kSmem <= 232448, "shared memory budget");
};

struct WgParams {
    int64_t B, N, H, C;
    int64_t R, Cc;         // rows and columns of dW
    int a_heads, b_heads;  // source kinds: 1 = HEADS, 0 = PLAIN
    int a_apb, b_apb;      // atoms per TMA box of each operand
    int NT;
    uint32_t idesc;
    int64_t stages_per_b, stages;  // 64-token stages of a batch element, and of all
    int64_t chunk_len, n_chunks;   // stages per chunk
    int64_t row_tiles, row_groups, col_tiles, n_items;
    float* part;  // [n_chunks][R][Cc]
    int* status;
};

struct WItem {
    int64_t rt, ct, g0, g1, chunk;  // stages [g0, g1)
    int halves;  // row tiles rt, rt + 1, ... of this item
};

__device__ __forceinline__ WItem witem(const WgParams& p, int64_t v) {
    WItem w;
    const int64_t tiles = p.row_groups * p.col_tiles;
    const int64_t t = v % tiles;  // tiles of one chunk run together (their tokens are shared)
    w.chunk = v / tiles;
    w.rt = t / p.col_tiles * kHalves;
    w.halves = (int)min((int64_t)kHalves, p.row_tiles - w.rt);
    w.ct = t % p.col_tiles;
    w.g0 = w.chunk * p.chunk_len;
    w.g1 = min(p.stages, w.g0 + p.chunk_len);
    return w;
}

__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                         int* status) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 0) {
            if (*abort_flag) return false;
            if (globaltimer_ns() - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                atomicExch(status, (int)FLAREPP_ERR_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* status) {
    const bool got = wait_bar(bar, parity, abort_flag, status);
    return __all_sync(0xffffffffu, got);
}

// Load the atoms of channels [c0, c0 + width) of one source for tokens [n0, n0 + kTok) of
// batch element b into consecutive atom slots at dst, in boxes of apb atoms (a box never
// crosses from one tensor of a HEADS source into the next).
template <int D>
__device__ __forceinline__ void load_atoms(uint32_t dst, int heads_kind, const CUtensorMap* m0,
                                           const CUtensorMap* m1, const CUtensorMap* m2,
                                           const CUtensorMap* m3, int64_t c0, int width, int apb,
                                           int64_t C, int64_t b, int n0, uint32_t bar) {
    using W = WCfg<D>;
    for (int k = 0; k < width / (apb * D); ++k) {
        const int64_t c = c0 + (int64_t)k * apb * D;
        const uint32_t d = dst + k * apb * W::kAtom;
        if (heads_kind) {
            const int64_t p = c / C;
            const CUtensorMap* m = p == 0 ? m0 : p == 1 ? m1 : p == 2 ? m2 : m3;
            tma_load_4d(d, m, 0, n0, (int)((c % C) / D), (int)b, bar);
        } else {
            tma_load_4d(d, m0, 0, n0, (int)(c / D), (int)b, bar);
        }
    }
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    tc_wgrad_kernel(const __grid_constant__ CUtensorMap tA0, const __grid_constant__ CUtensorMap tA1,
                    const __grid_constant__ CUtensorMap tA2, const __grid_constant__ CUtensorMap tA3,
                    const __grid_constant__ CUtensorMap tB0, const __grid_constant__ CUtensorMap tB1,
                    const __grid_constant__ CUtensorMap tB2, const __grid_constant__ CUtensorMap tB3,
                    const WgParams prm) {
    using W = WCfg<D>;
    constexpr int kS = W::kStages;
    pdl_trigger();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_shared<1024>(smem_raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kS * W::kStage);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + W::kNumBars);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t full0 = smem_u32(bars);
    const uint32_t empty0 = full0 + 8u * kS;
    const uint32_t accfull0 = empty0 + 8u * kS;
    const uint32_t accempty0 = accfull0 + 16u;
    const uint32_t fin = accempty0 + 16u;
    const int warp = warp_index();
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int st = 0; st < kS; ++st) {
            mbar_init(full0 + 8u * st, 1);
            mbar_init(empty0 + 8u * st, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accfull0 + 8u * b, 1);
            mbar_init(accempty0 + 8u * b, kRowsW);
        }
        mbar_init(fin, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);
    // every global access below may depend on the kernel before this one
    pdl_wait();

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        uint32_t it = 0;
        bool ok = true;
        for (int64_t v = blockIdx.x; v < prm.n_items && ok; v += gridDim.x) {
            const WItem I = witem(prm, v);
            const uint32_t bytes = (uint32_t)(I.halves * W::kAStage + (prm.NT / D) * W::kAtom);
            int64_t b = I.g0 / prm.stages_per_b, in_b = I.g0 % prm.stages_per_b;
            for (int64_t g = I.g0; g < I.g1; ++g, ++it) {
                const int st = it % kS;
                if (it >= (uint32_t)kS &&
                    !warp_wait(empty0 + 8u * st, ((it / kS) - 1) & 1, abort_flag, prm.status)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const uint32_t dst = smem_u32(smem + st * W::kStage);
                    mbar_expect_tx(full0 + 8u * st, bytes);
                    const int n = (int)(in_b * kTok);
                    for (int x = 0; x < I.halves; ++x)
                        load_atoms<D>(dst + x * W::kAStage, prm.a_heads, &tA0, &tA1, &tA2, &tA3,
                                      (I.rt + x) * kRowsW, kRowsW, prm.a_apb, prm.C, b, n,
                                      full0 + 8u * st);
                    load_atoms<D>(dst + kHalves * W::kAStage, prm.b_heads, &tB0, &tB1, &tB2, &tB3,
                                  I.ct * prm.NT, prm.NT, prm.b_apb, prm.C, b, n, full0 + 8u * st);
                }
                __syncwarp();
                if (++in_b == prm.stages_per_b) {
                    in_b = 0;
                    ++b;
                }
            }
        }
        if (!ok) {
            const uint64_t t0 = globaltimer_ns();
            for (int st = 0; st < kS && (uint32_t)st < it; ++st) {
                const uint32_t x = it - 1 - ((it - 1 - st) % kS);
                while (!mbar_try_wait(full0 + 8u * st, (x / kS) & 1) &&
                       globaltimer_ns() - t0 < kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        // row tile number seq of this CTA is summed in accumulator seq & 1
        uint32_t it = 0, seq = 0;
        bool ok = true;
        for (int64_t v = blockIdx.x; v < prm.n_items && ok; v += gridDim.x) {
            const WItem I = witem(prm, v);
            for (int x = 0; x < I.halves && ok; ++x)  // the accumulators are read out
                ok = seq + x < 2 ||
                     warp_wait(accempty0 + 8u * ((seq + x) & 1), (((seq + x) >> 1) - 1) & 1,
                               abort_flag, prm.status);
            if (!ok) break;
            for (int64_t g = I.g0; g < I.g1; ++g, ++it) {
                const int st = it % kS;
                if (!warp_wait(full0 + 8u * st, (it / kS) & 1, abort_flag, prm.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = smem_u32(smem + st * W::kStage);
                if (elect_one()) {
                    // MN-major operands: K steps of 16 tokens inside each atom (16 D 2 bytes on, in
                    // the descriptors' units of 16); atoms (D-wide channel columns) kAtom bytes
                    // apart along M and N
                    const uint64_t bd =
                        smem_desc(a0 + kHalves * W::kAStage, W::kAtom, W::kSBO, W::kSwz);
#pragma unroll
                    for (int x = 0; x < kHalves; ++x) {
                        if (x >= I.halves) break;
                        const uint32_t acc = tmem + ((seq + x) & 1) * kMaxNT;
                        const uint64_t ad = smem_desc(a0 + x * W::kAStage, W::kAtom, W::kSBO, W::kSwz);
#pragma unroll
                        for (int k = 0; k < kTok / 16; ++k)
                            mma_ss(acc, ad + 2 * D * k, bd + 2 * D * k, prm.idesc,
                                   (g == I.g0 && k == 0) ? 0u : 1u);
                    }
                    mma_commit(empty0 + 8u * st);
                }
                __syncwarp();
            }
            if (!ok) break;
            if (elect_one())
                for (int x = 0; x < I.halves; ++x) mma_commit(accfull0 + 8u * ((seq + x) & 1));
            __syncwarp();
            seq += I.halves;
        }
        if (elect_one()) mma_commit(fin);
        __syncwarp();
        const uint64_t tw = globaltimer_ns();
        while (!__all_sync(0xffffffffu, mbar_try_wait(fin, 0)) &&
               globaltimer_ns() - tw < kWaitLimitNs) {
        }
    } else if (warp >= kFirstEpiWarp) {
        // ------------------------------------------------------------ epilogue
        const int q = warp % 4;
        const int r = 32 * q + lane;
        const uint32_t lane_off = (uint32_t)(32 * q) << 16;
        uint32_t j = 0;
        bool ok = true;
        for (int64_t v = blockIdx.x; v < prm.n_items && ok; v += gridDim.x) {
            const WItem I = witem(prm, v);
            for (int x = 0; x < I.halves; ++x, ++j) {
                const int ab = j & 1;
                if (!warp_wait(accfull0 + 8u * ab, (j >> 1) & 1, abort_flag, prm.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + lane_off + ab * kMaxNT;
                const int64_t row = (I.rt + x) * kRowsW + r;
                float* dst = prm.part + (I.chunk * prm.R + row) * prm.Cc + I.ct * prm.NT;
                for (int c = 0; c < prm.NT; c += 16) {
                    uint32_t v16[16];
                    tmem_ld16(acc + c, v16);
                    tmem_wait_ld16(v16);
                    if (row < prm.R) {
                        float4* d4 = reinterpret_cast<float4*>(dst + c);
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            d4[g] = make_float4(
                                __uint_as_float(v16[4 * g]), __uint_as_float(v16[4 * g + 1]),
                                __uint_as_float(v16[4 * g + 2]), __uint_as_float(v16[4 * g + 3]));
                    }
                }
                tc_fence_before();
                mbar_arrive(accempty0 + 8u * ab);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// dW = sum of the chunks' partials; rows r < R_out take the sum of the rows r + k * R_out for
// k < fold (fold 2 adds the gradients of tied projections). A block of eight warps has 128 values of
// dW, four per lane; warp w adds the partials w, w + 8, ... of the fold * n_chunks, then the eight
// sums are added in warp order. (One thread per value going through all chunks was a chain of loads:
// 44 us for dWo and 26 for dW_in at 262,144 tokens, C = 256, four projections; now 10 and 12.)
constexpr int kReduceWarps = 8;
__global__ void __launch_bounds__(32 * kReduceWarps)
    wgrad_reduce_kernel(const float* __restrict__ part, int64_t n_chunks, int64_t R, int64_t Cc,
                        int64_t R_out, int fold, __nv_bfloat16* __restrict__ out) {
    __shared__ float4 sums[kReduceWarps][32];
    pdl_trigger();
    pdl_wait();
    const int w = threadIdx.x / 32, lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * 32 + lane) * 4;  // Cc is a multiple of 16
    const bool in = i < R_out * Cc;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) {
        for (int k = 0; k < fold; ++k) {
            const float* src = part + k * R_out * Cc + i;
#pragma unroll 4
            for (int64_t ch = w; ch < n_chunks; ch += kReduceWarps) {
                const float4 v = *reinterpret_cast<const float4*>(src + ch * R * Cc);
                acc.x += v.x;
                acc.y += v.y;
                acc.z += v.z;
                acc.w += v.w;
            }
        }
    }
    sums[w][lane] = acc;
    __syncthreads();
    if (w != 0 || !in) return;
    for (int g = 1; g < kReduceWarps; ++g) {
        const float4 v = sums[g][lane];
        acc.x += v.x;
        acc.y += v.y;
        acc.z += v.z;
        acc.w += v.w;
    }
    const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y);
    const __nv_bfloat162 hi = __floats2bfloat162_rn(acc.z, acc.w);
    uint2 o;
    o.x = *reinterpret_cast<const uint32_t*>(&lo);
    o.y = *reinterpret_cast<const uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(out + i) = o;
}

__global__ void transpose_bf16_kernel(const __nv_bfloat16* __restrict__ src, int64_t R,
                                      int64_t Cc, int rep, __nv_bfloat16* __restrict__ dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // index into dst
    const int64_t cols = rep * R;
    if (i >= Cc * cols) return;
    const int64_t c = i / cols, j = i % cols;
    dst[i] = src[(j % R) * Cc + c];
}

__global__ void add_bf16_kernel(__nv_bfloat16* __restrict__ dst,
                                const __nv_bfloat16* __restrict__ src, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16_rn(__bfloat162float(dst[i]) + __bfloat162float(src[i]));
}

// ------------------------------------------------------------------ host side

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// bf16 {D channels, N tokens, atoms, B} with the given byte strides of dimensions 1..3;
// boxes of D x kTok x `atoms` x 1, swizzled to the D-wide row. In shared memory a box is
// atom-major: atom a is the kTok x D block at a * kTok * D * 2.
bool make_map(CUtensorMap* m, const void* base, int64_t D, int64_t N, int64_t n_atoms,
              int64_t B, int64_t s_tok, int64_t s_atom, int64_t s_b, int atoms) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)N, (cuuint64_t)n_atoms, (cuuint64_t)B};
    cuuint64_t strides[3] = {(cuuint64_t)s_tok, (cuuint64_t)s_atom, (cuuint64_t)s_b};
    cuuint32_t box[4] = {(cuuint32_t)D, (cuuint32_t)kTok, (cuuint32_t)atoms, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapSwizzle sw = D == 16 ? CU_TENSOR_MAP_SWIZZLE_32B
                                          : (D == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                     : CU_TENSOR_MAP_SWIZZLE_128B);
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Atoms per box for tiles of `width` channels: the whole tile, unless a tile of a HEADS
// source could cross from one tensor into the next (C not a multiple of the width).
int atoms_per_box(const WgradSource& s, int64_t C, int64_t D, int width) {
    return (s.heads && C % width != 0) ? 1 : width / (int)D;
}

// the maps of one source, for boxes of `atoms` atoms: HEADS (n tensors [B*H][N][D], the
// atoms are heads) or PLAIN ([B][N][C], the atoms are the D-wide column blocks)
bool source_maps(CUtensorMap* m, const WgradSource& s, int64_t B, int64_t N, int64_t H,
                 int64_t D, int atoms) {
    for (int p = 0; p < 4; ++p) {
        const void* base = s.t[p < s.n ? p : 0];
        const bool ok = s.heads ? make_map(&m[p], base, D, N, H, B, D * 2, N * D * 2,
                                           H * N * D * 2, atoms)
                                : make_map(&m[p], base, D, N, H, B, H * D * 2, D * 2,
                                           N * H * D * 2, atoms);
        if (!ok) return false;
    }
    return true;
}

template <int D>
cudaError_t launch(const CUtensorMap* ma, const CUtensorMap* mb, const WgParams& prm,
                   cudaStream_t st) {
    using Wc = WCfg<D>;
    const cudaError_t attr = ensure_smem_limit((const void*)tc_wgrad_kernel<D>, Wc::kSmem);
    if (attr != cudaSuccess) return attr;
    if (prm.n_items == 0) return cudaSuccess;
    int dev = 0, sms = kNumSMs;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t grid = prm.n_items < sms ? prm.n_items : sms;
    return launch_pdl(tc_wgrad_kernel<D>, dim3((unsigned)grid), dim3(kThreads), Wc::kSmem, st, ma[0],
                      ma[1], ma[2], ma[3], mb[0], mb[1], mb[2], mb[3], prm);
}

}  // namespace

cudaError_t transpose_bf16(const void* src, int64_t R, int64_t Cc, int rep, void* dst,
                           cudaStream_t st) {
    const int64_t n = Cc * rep * R;
    if (n == 0) return cudaSuccess;
    transpose_bf16_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
        (const __nv_bfloat16*)src, R, Cc, rep, (__nv_bfloat16*)dst);
    return cudaGetLastError();
}

cudaError_t add_bf16(void* dst, const void* src, int64_t n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096;
    add_bf16_kernel<<<(unsigned)blocks, 256, 0, st>>>((__nv_bfloat16*)dst,
                                                      (const __nv_bfloat16*)src, n);
    return cudaGetLastError();
}

WgradPlan wgrad_plan(int64_t B, int64_t N, int64_t R, int64_t Cc) {
    WgradPlan w{};
    int nt = kMaxNT;
    while (nt > 16 && Cc % nt != 0) nt /= 2;
    w.NT = nt;
    w.row_tiles = (R + kRowsW - 1) / kRowsW;
    w.col_tiles = Cc / nt;
    // The chunk count of least time, in units of a stage (about 1.2 us with every SM at it): waves of
    // items, each its stages and an epilogue (256 KB of partial sums an item: about 8), and the reduce's
    // reads of the partial sums (5 for a full wave's). Chunks run over the batch: cut inside a batch
    // element, 10 of them at C = 512 are 160 items for the four projections on 152 SMs, two waves
    // (dW_in of 10 x 2,000 tokens 86 us, with chunks over the batch 52).
    w.row_groups = (w.row_tiles + kHalves - 1) / kHalves;
    w.stages_per_b = (N + kTok - 1) / kTok;
    const int64_t tiles = w.row_groups * w.col_tiles, stages = B * w.stages_per_b;
    double best = 1e300;
    int64_t n = 0, waves = cdiv(tiles, kNumSMs) - 1;
    for (int k = 0; k < 6 && n < stages; ++k) {
        n = ++waves * kNumSMs / tiles;  // the most chunks with these waves
        if (n > stages) n = stages;
        const int64_t len = cdiv(stages, n), chunks = cdiv(stages, len);
        const double cost = (double)cdiv(tiles * chunks, kNumSMs) * ((double)len + 8.0) +
                            5.0 * (double)(tiles * chunks) / kNumSMs;
        if (cost < best) {
            best = cost;
            w.chunk_len = len;
            w.n_chunks = chunks;
        }
    }
    w.part_bytes = (size_t)w.n_chunks * (size_t)R * (size_t)Cc * sizeof(float);
    return w;
}

cudaError_t tc_wgrad(int64_t B, int64_t N, int64_t H, int64_t D, const WgradSource& a,
                     const WgradSource& b, int64_t R, int64_t Cc, int64_t R_out, int fold,
                     float* part, void* dW, int* status, cudaStream_t st) {
    const WgradPlan w = wgrad_plan(B, N, R, Cc);
    if (w.NT % D != 0 || R % D != 0) return cudaErrorInvalidValue;
    WgParams prm{};
    prm.B = B;
    prm.N = N;
    prm.H = H;
    prm.C = H * D;
    prm.R = R;
    prm.Cc = Cc;
    prm.a_heads = a.heads;
    prm.b_heads = b.heads;
    prm.NT = w.NT;
    prm.idesc = idesc_bf16_f32(kRowsW, w.NT, true, true);
    prm.stages_per_b = w.stages_per_b;
    prm.stages = B * w.stages_per_b;
    prm.chunk_len = w.chunk_len;
    prm.n_chunks = w.n_chunks;
    prm.row_tiles = w.row_tiles;
    prm.col_tiles = w.col_tiles;
    prm.row_groups = w.row_groups;
    prm.n_items = w.n_chunks * w.row_groups * w.col_tiles;
    prm.part = part;
    prm.status = status;
    CUtensorMap ma[4], mb[4];
    prm.a_apb = atoms_per_box(a, H * D, D, kRowsW);
    prm.b_apb = atoms_per_box(b, H * D, D, w.NT);
    if (!source_maps(ma, a, B, N, H, D, prm.a_apb) || !source_maps(mb, b, B, N, H, D, prm.b_apb))
        return cudaErrorInvalidValue;
    cudaError_t e;
    switch (D) {
        case 16: e = launch<16>(ma, mb, prm, st); break;
        case 32: e = launch<32>(ma, mb, prm, st); break;
        case 64: e = launch<64>(ma, mb, prm, st); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int64_t n = R_out * Cc;
    return launch_pdl(wgrad_reduce_kernel, dim3((unsigned)((n + 127) / 128)), dim3(32 * kReduceWarps),
                      0, st, (const float*)part, w.n_chunks, R, Cc, R_out, fold, (__nv_bfloat16*)dW);
}

}  // namespace flarepp

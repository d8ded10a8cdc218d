// Tensor-core token passes of the chain's backward (App. A.5) that also form the route-side
// gradient: bf16 inputs, D = 16 and 32, up to tok_max_routes(D) routes.
//
// TMEM lanes are tokens. For a tile of 128 tokens and every item of 64 routes a pass forms the
// score tiles, turns them into P and dS (bf16), and accumulates
//   calls 3 and 2 (CALL1 false), with u = 2^(L3 - R), w = 2^(R - L2) for the shift R of the
//     (b, h) (the two calls' probabilities differ by the rank-one factor P2 / P3 = u w):
//       S = K Q^T,  T = [dY | u V] [Z | w dZ]^T,  P3 = 2^(c S - L3),
//     (u V as a bf16 pair hi + lo: V is exact in bf16, and with u V rounded once more dQ, and with it
//     dseeds, dKt and dVt, would be further off than with V itself: dVt's error by 17 to 40 %)
//       dS = P3 (T - c3 - u (w c2)),  E2 = P3 u
//       dK += dS Q,   dV += E2 (w dZ),   dQ += dS^T K (calls 3 and 2 together)
//   call 1:
//       S = Kt Qs^T,  T = Vt dQ^T,  P = 2^(c S - L1),  dS = P (T - c1)
//       dKt += dS Qs,  dVt += P dQ,   dQs += dS^T Kt
// The sums over the tokens (dQ, dQs) stay in TMEM for all tiles of a (b, h) that the CTA works
// on and leave as one float32 partial per CTA and (b, h), which a reduce adds in CTA order. So
// the scores of a call are formed, and their exponentials taken, once for both sides of the
// gradient; a separate route-row pass for dQ would do both again.
//
// dS goes to shared memory as [128 tokens][64 routes], one 128-byte row per token, swizzled: read
// K-major it is the A operand of dK += dS Q, read MN-major it is the transposed A operand of
// dQ += dS^T K. P (or E2) goes back to TMEM over the T columns its thread has read.
//
// Two streams share a token tile: stream s takes the route items s, s + 2, ..., so that the dS
// tiles of items 2b and 2b + 1 (block b) lie next to each other and one product of 128 routes
// serves both. Each stream has its own score tiles and two warpgroups of 32 columns each; the item ring
// and dK and dV are shared, the latter with two accumulators by the parity of the tile.
// Roles (20 warps): warp 0 issues every product, warp 3 loads (TMA) the token tiles, the items and
// the per-route statistics; warps 4..19 are the softmax warpgroups (stream w / 2, columns
// 32 (w % 2) ..). One issuer serves the streams in turn: for a stream's item it issues S, the dV
// product of the stream's item before (which frees the T columns), T, and one commit that the
// softmax waits on, then the dK product of the item before; after both streams the dQ product of
// the block before. Two issuers, one per stream, let the streams fall into step: both waited for
// the tensor pipe, then both worked on scores while it idled (3600 cycles per block of 128 x 128
// scores in call 1 on the 262,144-token shape).
// Persistent CTAs take equal, contiguous runs of the BH x ceil(N / 128) token tiles, so a CTA
// changes its (b, h) (and writes its dQ) as rarely as possible.
// Every wait is bounded as in the other tensor-core kernels: on expiry the kernel records
// FLAREPP_ERR_TIMEOUT in the status word, every role leaves its loops, the producer waits for its
// copies in flight, the MMA issuers for their products, and TMEM is freed.
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

constexpr int kRows = 128;   // tokens per tile (TMEM lanes, MMA M)
constexpr int kItem = 64;    // routes per item
constexpr int kThreads = 20 * 32;
constexpr int kSoftThreads = 512;
constexpr int kFirstSoftmaxWarp = 4;
constexpr uint32_t kTmemCols = 512;

// LO (calls 3 and 2): Q as the hi/lo pair of bf16 operands the training forward gave it; the item
// carries Q's lo tile, and S adds the product with it.
template <int D, bool CALL1, bool LO>
struct TokCfg {
    static_assert(D == 16 || D == 32, "D = 64 has no room for dQ beside its accumulators");
    static_assert(!(CALL1 && LO), "call 1's scores take the seeds, exact in bf16");
    static constexpr int kNT = CALL1 ? 2 : 3;        // token tiles: K, V (, dY) / Kt, Vt
    static constexpr int kNI = kNT + (LO ? 1 : 0);   // item tiles: Q, w dZ, Z (, lo) / Qs, dQ
    static constexpr int kATile = kRows * D * 2;
    // (calls 3 and 2: u V leaves its tile as a bf16 pair, the lo part in a tile behind the loaded ones)
    static constexpr int kABytes = (kNT + (CALL1 ? 0 : 1)) * kATile;
    static constexpr int kItemTile = kItem * D * 2;
    static constexpr int kStage = kNI * kItemTile;
    // ring stages, taken by the items of both streams in turn: at D = 32 the pair of u V leaves room
    // for five in calls 3 and 2 (two a stream: the training step of 262,144 tokens, M = 512, 2165 us
    // instead of 2104; u V rounded once, with three a stream, 2055)
    static constexpr int kStages = D == 32 && !CALL1 ? 5 : 6;
    static constexpr int kDsTile = kRows * kItem * 2;
    static constexpr int kMaxM = (int)tok_max_routes(D);
    static constexpr uint32_t kSwz = D == 16 ? kSw32 : kSw64;
    static constexpr uint32_t kSBO = 8 * D * 2;
    static constexpr uint32_t kDsSBO = 8 * kItem * 2;
    // TMEM columns: per stream S and T, then per tile parity dK and dV, then dQ (D per 128 routes)
    static constexpr uint32_t kColAcc = 4 * kItem;
    static constexpr uint32_t kColQ = kColAcc + 4 * D;
    static_assert(kColQ + (kMaxM / 128) * D <= kTmemCols, "TMEM budget");
    // shared memory: dS [buffer][stream], token tiles [2], the ring, statistics
    // [segment parity][2][kMaxM], barriers
    static constexpr int kOffA = 4 * kDsTile;
    static constexpr int kOffRing = kOffA + 2 * kABytes;
    static constexpr int kOffStat = kOffRing + kStages * kStage;
    static constexpr int kOffBars = kOffStat + 4 * kMaxM * 4;
    // full[stages], empty[stages], afull[2], aready[2], afree[2], sready[2], pready[2],
    // accdone[2], accfree[2], statfull[2], segfree[2], dqdone, fin
    static constexpr int kNumBars = 2 * kStages + 18 + 2;
    static constexpr int kNeed = 1024 + kOffBars + kNumBars * 8 + 16;
    static constexpr int kSmem = kNeed > 122880 ? kNeed : 122880;  // one CTA per SM
    static_assert(kSmem <= 232448, "shared memory budget");
    static constexpr uint32_t kIdescS = idesc_bf16_f32(128, kItem, false, false);
    static constexpr uint32_t kIdescAcc = idesc_bf16_f32(128, D, false, true);
    static constexpr uint32_t kIdescQ = idesc_bf16_f32(128, D, true, true);
};

struct TokParams {
    int64_t H, N, M;
    int64_t nt, tiles;   // token tiles per (b, h), and in all
    int64_t slots;       // partial slots per (b, h)
    int n_items, n_blocks;  // route items of 64 and blocks of 128
    int i0_per_head;     // call 1: item tile 0 (the seeds) is indexed by head
    float c;             // scale * log2(e), signed
    float scale;
    const float* Lrow;   // calls 3 and 2: L3, c3 per token
    const float* crow;
    const float* Lcol;   // per route: L2, c2 (calls 3 and 2) or L1, c1
    const float* ccol;
    const float* Rb;     // calls 3 and 2: the shift R of each (b, h)
    const int* flags;    // when not null: only the (b, h) with flags[bh] == 0
    float* part;         // [BH][slots][M][D]: the CTAs' dS^T K
    __nv_bfloat16* out0;  // s dS Q and P dQ (or E2 w dZ), [BH][N][D]
    __nv_bfloat16* out1;
    int* status;
    uint64_t wait_ns;
    int64_t withhold_it;  // test hook: ring item of CTA 0 the producer never loads (-1: none)
};

// The CTA's run of token tiles, (b, h) by (b, h), without the flagged ones.
struct TileIt {
    const TokParams& p;
    int t, t1, bh, tile;
    __device__ __forceinline__ TileIt(const TokParams& prm)
        : p(prm),
          t((int)((int64_t)blockIdx.x * prm.tiles / gridDim.x)),
          t1((int)((int64_t)(blockIdx.x + 1) * prm.tiles / gridDim.x)),
          bh(0),
          tile(0) {
        settle();
    }
    __device__ __forceinline__ void settle() {
        for (; t < t1; t = (int)min((int64_t)(bh + 1) * (int)p.nt, (int64_t)t1)) {
            bh = t / (int)p.nt;
            tile = t - bh * (int)p.nt;
            if (p.flags == nullptr || p.flags[bh] == 0) return;
        }
    }
    __device__ __forceinline__ bool valid() const { return t < t1; }
    __device__ __forceinline__ bool last_of_segment() const {
        return t + 1 >= t1 || tile + 1 == (int)p.nt;
    }
    __device__ __forceinline__ void next() {
        ++t;
        if (++tile == (int)p.nt) settle();
    }
};

// Partial slot of this CTA for (b, h): its distance from the first CTA whose run reaches it.
__device__ __forceinline__ int64_t first_cta(int64_t tile, int64_t tiles, int64_t ctas) {
    return ((tile + 1) * ctas - 1) / tiles;
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t ex2x2(uint64_t x) {
    float a, b;
    unpack_f32x2(x, a, b);
    return pack_f32x2(ex2(a), ex2(b));
}
// bf16 pair (lo in the low half) from a packed f32 pair
__device__ __forceinline__ uint32_t bf16x2(uint64_t v) {
    uint32_t r;
    asm("{\n\t.reg .f32 a, b;\n\tmov.b64 {a, b}, %1;\n\tcvt.rn.bf16x2.f32 %0, b, a;\n\t}"
        : "=r"(r)
        : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t ld_pair(const uint32_t* r, int k) {
    return pack_f32x2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
}

// Bounded wait on an mbarrier phase by a whole warp. False when the kernel is aborting.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                         int* status, uint64_t limit) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 0) {
            if (*abort_flag) return false;
            if (globaltimer_ns() - t0 > limit) {
                *abort_flag = 1;
                atomicExch(status, (int)FLAREPP_ERR_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, uint64_t limit) {
    const bool got = wait_bar(bar, parity, abort_flag, status, limit);
    return __all_sync(0xffffffffu, got);
}

__device__ __forceinline__ void tmem_wait_ld8(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
}

// This row's row statistics of a token tile: -L3, -c3 and u = 2^(L3 - R) (calls 3 and 2).
struct RowStats {
    float nL, nc, u;
};

// P (or E2) and dS of 16 columns for this thread's row, packed bf16 pairs. sr, tr: the columns of
// S and T; st0, st1: the per-route statistics of these columns (calls 3 and 2: -(w c2) in st0;
// call 1: -L1 in st0, -c1 in st1). Columns at or beyond nv are not routes: 0.
template <bool CALL1, bool FULL>
__device__ __forceinline__ void slice_math(const uint32_t* sr, const uint32_t* tr, uint32_t* pp,
                                           uint32_t* ds, int nv, uint64_t c2, uint64_t nL2,
                                           uint64_t nc2, uint64_t u2, const float* st0,
                                           const float* st1) {
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(st0 + 2 * k);
        ulonglong2 b{};
        if (CALL1) b = *reinterpret_cast<const ulonglong2*>(st1 + 2 * k);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint64_t x = ld_pair(sr, k + e), t = ld_pair(tr, k + e);
            const uint64_t s0 = e == 0 ? a.x : a.y, s1 = e == 0 ? b.x : b.y;
            uint64_t p, d;
            if (CALL1) {
                p = ex2x2(fma2(x, c2, s0));
                d = mul2(p, add2(t, s1));
            } else {
                const uint64_t p3 = ex2x2(fma2(x, c2, nL2));
                p = mul2(p3, u2);
                d = mul2(p3, fma2(u2, s0, add2(t, nc2)));
            }
            pp[k + e] = bf16x2(p);
            ds[k + e] = bf16x2(d);
            if (!FULL) {
                const int col = 2 * (k + e);
                const uint32_t m = (col < nv ? 0xffffu : 0u) | (col + 1 < nv ? 0xffff0000u : 0u);
                pp[k + e] &= m;
                ds[k + e] &= m;
            }
        }
    }
}

template <int D, bool CALL1, bool LO>
__global__ void __launch_bounds__(kThreads, 1)
    tc_tok_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmA1,
                  const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmI0,
                  const __grid_constant__ CUtensorMap tmI1, const __grid_constant__ CUtensorMap tmI2,
                  const __grid_constant__ CUtensorMap tmLo, const TokParams prm) {
    using C = TokCfg<D, CALL1, LO>;
    constexpr int kS = C::kStages;
    pdl_trigger();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_shared<1024>(smem_raw);
    uint8_t* ds_buf = smem;
    uint8_t* abuf = smem + C::kOffA;
    uint8_t* ring = smem + C::kOffRing;
    float* stats = reinterpret_cast<float*>(smem + C::kOffStat);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kOffBars);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::kNumBars);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const uint32_t full0 = smem_u32(bars);  // [stage]
    const uint32_t empty0 = full0 + 8u * kS;  // [stage]
    const uint32_t afull0 = empty0 + 8u * kS;
    const uint32_t aready0 = afull0 + 16u;
    const uint32_t afree0 = aready0 + 16u;
    const uint32_t sready0 = afree0 + 16u;
    const uint32_t pready0 = sready0 + 16u;
    const uint32_t accdone0 = pready0 + 16u;
    const uint32_t accfree0 = accdone0 + 16u;
    const uint32_t statfull0 = accfree0 + 16u;
    const uint32_t segfree0 = statfull0 + 16u;
    const uint32_t dqdone = segfree0 + 16u;
    const uint32_t fin = dqdone + 8u;

    const int warp = warp_index();
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int k = 0; k < kS; ++k) {
            mbar_init(full0 + 8u * k, 1);
            mbar_init(empty0 + 8u * k, 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(afull0 + 8u * k, 1);
            mbar_init(aready0 + 8u * k, kSoftThreads);
            mbar_init(afree0 + 8u * k, 1);
            mbar_init(sready0 + 8u * k, 1);
            mbar_init(pready0 + 8u * k, 8);
            mbar_init(accdone0 + 8u * k, 1);
            mbar_init(accfree0 + 8u * k, kSoftThreads);
            mbar_init(statfull0 + 8u * k, 32);
            mbar_init(segfree0 + 8u * k, kSoftThreads);
        }
        mbar_init(dqdone, 1);
        mbar_init(fin, 1);
        *abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmA0);
        prefetch_tmap(&tmA1);
        prefetch_tmap(&tmI0);
        prefetch_tmap(&tmI1);
        if (!CALL1) {
            prefetch_tmap(&tmA2);
            prefetch_tmap(&tmI2);
        }
        if (LO) prefetch_tmap(&tmLo);
    }
    if (warp == 2) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);
    // every global access below may depend on the kernel before this one
    pdl_wait();
    auto wait = [&](uint32_t bar, uint32_t parity) {
        return warp_wait(bar, parity & 1u, abort_flag, prm.status, prm.wait_ns);
    };

    if (warp == 3) {
        // ------------------------------------------------------------ TMA producer
        uint32_t tc = 0, seg = 0, it = 0;  // tiles, segments, items
        int prev_bh = -1;
        int64_t withheld = -1;
        bool ok = true;
        for (TileIt T(prm); T.valid() && ok; T.next(), ++tc) {
            if (T.bh != prev_bh) {
                // the statistics of the (b, h)'s routes, negated, for this segment
                prev_bh = T.bh;
                const uint32_t sb = seg & 1u;
                if (seg >= 2 && !wait(segfree0 + 8u * sb, (seg >> 1) - 1)) {
                    ok = false;
                    break;
                }
                float* s0 = stats + sb * 2 * C::kMaxM;
                float* s1 = s0 + C::kMaxM;
                const float R = CALL1 ? 0.f : prm.Rb[T.bh];
                for (int m = lane; m < prm.n_items * kItem; m += 32) {
                    const bool in = m < prm.M;
                    const int64_t idx = (int64_t)T.bh * prm.M + m;
                    const float L = in ? prm.Lcol[idx] : 0.f, cc = in ? prm.ccol[idx] : 0.f;
                    if (CALL1) {
                        s0[m] = -L;
                        s1[m] = -cc;
                    } else {
                        s0[m] = in ? -exp2f(R - L) * cc : 0.f;
                    }
                }
                mbar_arrive(statfull0 + 8u * sb);
                ++seg;
            }
            const uint32_t ab = tc & 1u;
            if (tc >= 2 && !wait(afree0 + 8u * ab, (tc >> 1) - 1)) {
                ok = false;
                break;
            }
            if (elect_one()) {
                const uint32_t bar = afull0 + 8u * ab;
                const uint32_t dst = smem_u32(abuf + ab * C::kABytes);
                const int row = T.tile * kRows;
                mbar_expect_tx(bar, C::kNT * C::kATile);
                tma_load_3d(dst, &tmA0, 0, row, T.bh, bar);
                tma_load_3d(dst + C::kATile, &tmA1, 0, row, T.bh, bar);
                if (!CALL1) tma_load_3d(dst + 2 * C::kATile, &tmA2, 0, row, T.bh, bar);
            }
            __syncwarp();
            const int z0 = (int)(prm.i0_per_head ? T.bh % prm.H : T.bh);
            for (int i = 0; i < prm.n_items; ++i) {
                const uint32_t st = it % kS;
                if (it >= (uint32_t)kS && !wait(empty0 + 8u * st, it / kS - 1)) {
                    ok = false;
                    break;
                }
                if (blockIdx.x == 0 && it == prm.withhold_it) {
                    withheld = it++;  // never loaded: the waits of its consumers run out
                    continue;
                }
                ++it;
                if (elect_one()) {
                    const uint32_t bar = full0 + 8u * st;
                    const uint32_t dst = smem_u32(ring + st * C::kStage);
                    const int row = i * kItem;
                    mbar_expect_tx(bar, C::kStage);
                    tma_load_3d(dst, &tmI0, 0, row, z0, bar);
                    tma_load_3d(dst + C::kItemTile, &tmI1, 0, row, T.bh, bar);
                    if (!CALL1)
                        tma_load_3d(dst + 2 * C::kItemTile, &tmI2, 0, row, T.bh, bar);
                    if (LO)
                        tma_load_3d(dst + C::kNT * C::kItemTile, &tmLo, 0, row, T.bh, bar);
                }
                __syncwarp();
            }
        }
        if (!ok) {
            // after an abort: wait (bounded) until the newest copy of every buffer has landed
            const uint64_t w0 = globaltimer_ns();
            for (uint32_t st = 0; st < (uint32_t)kS && st < it; ++st) {
                const uint32_t x = it - 1 - ((it - 1 - st) % kS);  // the newest item in this stage
                while (x != withheld && !mbar_try_wait(full0 + 8u * st, (x / kS) & 1) &&
                       globaltimer_ns() - w0 < prm.wait_ns) {
                }
            }
            // (the token tiles issued are those of the tiles before tc, and perhaps tc itself)
            for (uint32_t b = 0; b < 2 && b < tc; ++b) {
                const uint32_t x = tc - 1 - ((tc - 1 - b) & 1u);
                while (!mbar_try_wait(afull0 + 8u * b, (x >> 1) & 1) &&
                       globaltimer_ns() - w0 < prm.wait_ns) {
                }
            }
        }
    } else if (warp == 0) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t kHi = smem_desc_hi(C::kSBO, C::kSwz);
        constexpr uint32_t kHiDs = smem_desc_hi(C::kDsSBO, kSw128);
        const uint32_t a_u = smem_u32(abuf), ring_u = smem_u32(ring), ds_u = smem_u32(ds_buf);
        // the block before, whose dV, dK and dQ products are owed
        struct Block {
            bool any, two;              // it exists; stream 1 had an item in it
            bool first, last, seg_end;  // of its tile; the last tile of its segment
            bool fresh;                 // the first tile of its segment: dQ starts afresh
            uint32_t tc, st0, st1;      // its tile; ring stages of its items
        } o{};
        uint32_t it = 0;            // items
        uint32_t is0 = 0, is1 = 0;  // and per stream
        uint32_t bg = 0;            // blocks
        uint32_t n_fresh = 0;       // segments whose dQ products have begun
        // Stream s's turn: S and T of its item in stage st of token buffer ab (if `has`), and the
        // dV and dK products of its item of the block before (if `owed`).
        auto turn = [&](int s, bool has, uint32_t st, uint32_t ab, bool owed) {
            const uint32_t t0 = tmem + s * 2 * kItem;
            const uint32_t a = smem_desc_lo(a_u + ab * C::kABytes, 16);
            const uint32_t i = smem_desc_lo(ring_u + st * C::kStage, 16);
            const uint32_t o_st = s == 0 ? o.st0 : o.st1;
            const uint32_t acc = tmem + C::kColAcc + (o.tc & 1u) * 2 * D;
            const uint32_t im = smem_desc_lo(ring_u + o_st * C::kStage, C::kItemTile);
            const bool start = o.first && s == 0;  // the products that start dK and dV
            if (has) {
#pragma unroll
                for (int k = 0; k < D / 16; ++k)  // S = K Q^T
                    mma_ss(t0, desc_of(a + 2 * k, kHi), desc_of(i + 2 * k, kHi), C::kIdescS,
                           k > 0 ? 1u : 0u);
                if (LO) {
                    const uint32_t il = i + ((C::kNT * C::kItemTile) >> 4);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        mma_ss(t0, desc_of(a + 2 * k, kHi), desc_of(il + 2 * k, kHi), C::kIdescS,
                               1u);
                }
            }
            if (owed) {
#pragma unroll
                for (int k = 0; k < kItem / 16; ++k)  // dV += P dQ (E2 w dZ)
                    mma_ts(acc + D, t0 + kItem + 32 * (k / 2) + 8 * (k % 2),
                           desc_of(im + (C::kItemTile >> 4) + 2 * D * k, kHi), C::kIdescAcc,
                           (!start || k > 0) ? 1u : 0u);
            }
            if (has) {
                // T = Vt dQ^T, or (u V) (w dZ)^T + dY Z^T
                const uint32_t a1 = a + (C::kATile >> 4), i1 = i + (C::kItemTile >> 4);
#pragma unroll
                for (int k = 0; k < D / 16; ++k)
                    mma_ss(t0 + kItem, desc_of(a1 + 2 * k, kHi), desc_of(i1 + 2 * k, kHi),
                           C::kIdescS, k > 0 ? 1u : 0u);
                if (!CALL1) {
                    const uint32_t a2 = a + ((2 * C::kATile) >> 4), al = a + ((3 * C::kATile) >> 4);
                    const uint32_t i2 = i + ((2 * C::kItemTile) >> 4);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        mma_ss(t0 + kItem, desc_of(al + 2 * k, kHi), desc_of(i1 + 2 * k, kHi),
                               C::kIdescS, 1u);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        mma_ss(t0 + kItem, desc_of(a2 + 2 * k, kHi), desc_of(i2 + 2 * k, kHi),
                               C::kIdescS, 1u);
                }
                mma_commit(sready0 + 8u * s);
            }
            if (owed) {
                const uint32_t ds = smem_desc_lo(
                    ds_u + ((bg - 1) & 1u) * 2 * C::kDsTile + s * C::kDsTile, 16);
#pragma unroll
                for (int k = 0; k < kItem / 16; ++k)  // dK += dS Q
                    mma_ss(acc, desc_of(ds + 2 * k, kHiDs), desc_of(im + 2 * D * k, kHi),
                           C::kIdescAcc, (!start || k > 0) ? 1u : 0u);
                mma_commit(empty0 + 8u * o_st);
            }
        };
        // dQ += dS^T K of the block before, and what it frees.
        auto finish_block = [&](int b) {
            const uint32_t ab = o.tc & 1u, buf = (bg - 1) & 1u;
            const uint32_t d0 = smem_desc_lo(ds_u + buf * 2 * C::kDsTile, C::kDsTile);
            const uint32_t k0 = smem_desc_lo(a_u + ab * C::kABytes, C::kATile);
#pragma unroll
            for (int k = 0; k < kRows / 16; ++k)
                mma_ss(tmem + C::kColQ + b * D, desc_of(d0 + (k * 16 * kItem * 2 >> 4), kHiDs),
                       desc_of(k0 + 2 * D * k, kHi), C::kIdescQ, (!o.fresh || k > 0) ? 1u : 0u);
            if (o.last) {
                mma_commit(afree0 + 8u * ab);
                mma_commit(accdone0 + 8u * ab);
                if (o.seg_end) mma_commit(dqdone);
            }
        };
        // the waits of stream s's turn for the block before: its dS and P are written, and the
        // accumulators its tile starts in (those of two tiles before) are read out
        auto wait_owed = [&](int s) {
            return wait(pready0 + 8u * s, (s == 0 ? is0 : is1) - 1) &&
                   (s == 1 || !o.first || o.tc < 2 ||
                    wait(accfree0 + 8u * (o.tc & 1u), (o.tc >> 1) - 1));
        };
        // the segment before has given dQ back (the fence orders its TMEM reads before the product
        // that starts dQ afresh in the same columns)
        auto wait_dq = [&]() {
            if (!(o.fresh && o.first) || n_fresh++ == 0) return true;
            if (!wait(segfree0 + 8u * ((n_fresh - 2) & 1u), (n_fresh - 2) >> 1)) return false;
            tc_fence_after();
            return true;
        };
        bool ok = true, fresh = true;
        uint32_t tc = 0;
        const uint32_t nb = prm.n_blocks;
        for (TileIt T(prm); T.valid() && ok; T.next(), ++tc) {
            const uint32_t ab = tc & 1u;
            if (!wait((CALL1 ? afull0 : aready0) + 8u * ab, tc >> 1)) break;
            const bool seg_end = T.last_of_segment();
            for (uint32_t b = 0; b < nb; ++b) {
                const bool has1 = 2 * (int)b + 1 < prm.n_items;
                const uint32_t st0 = it % kS, st1 = (it + 1) % kS;
                ok = wait(full0 + 8u * st0, it / kS) && (!o.any || wait_owed(0));
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) turn(0, true, st0, ab, o.any);
                __syncwarp();
                ++is0;
                ok = (!has1 || wait(full0 + 8u * st1, (it + 1) / kS)) &&
                     (!(o.any && o.two) || wait_owed(1));
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) turn(1, has1, st1, ab, o.any && o.two);
                __syncwarp();
                if (has1) ++is1;
                it += has1 ? 2 : 1;
                if (o.any) {
                    ok = wait_dq();
                    if (!ok) break;
                    if (elect_one()) finish_block(b == 0 ? nb - 1 : b - 1);
                    __syncwarp();
                }
                o = Block{true, has1, b == 0, b + 1 == nb, seg_end, fresh, tc, st0, st1};
                ++bg;
            }
            fresh = seg_end;
        }
        if (ok && o.any && wait_owed(0)) {
            tc_fence_after();
            if (elect_one()) turn(0, false, 0, 0, true);
            __syncwarp();
            if (!o.two || wait_owed(1)) {
                tc_fence_after();
                if (o.two && elect_one()) turn(1, false, 0, 0, true);
                __syncwarp();
                if (wait_dq() && elect_one()) finish_block(nb - 1);
                __syncwarp();
            }
        }
        // every product issued has completed before TMEM is released
        if (elect_one()) mma_commit(fin);
        __syncwarp();
        const uint64_t w0 = globaltimer_ns();
        while (!__all_sync(0xffffffffu, mbar_try_wait(fin, 0)) &&
               globaltimer_ns() - w0 < prm.wait_ns) {
        }
    } else if (warp >= kFirstSoftmaxWarp) {
        // ------------------------------------------------------------ softmax warpgroups
        const int w = (warp - kFirstSoftmaxWarp) >> 2;
        const int s = w >> 1, h = w & 1;  // stream, column half
        const int q = warp & 3;
        const int r = 32 * q + lane;
        const uint32_t lane_t = tmem + ((uint32_t)(32 * q) << 16);
        const uint32_t colS = lane_t + s * 2 * kItem + 32 * h;
        const uint32_t colT = colS + kItem;
        const uint64_t c2 = pack_f32x2(prm.c, prm.c);
        uint8_t* ds_row = ds_buf + s * C::kDsTile + r * (kItem * 2);
        uint32_t seg = 0, is = 0, bg = 0, nprep = 0;
        bool ok = true;
        // Calls 3 and 2: this row's statistics of a tile, and (all 512 threads) the pair u V over V
        // in its shared-memory tile and in the one behind dY's: thread (w, r) takes 16-byte chunk w
        // of row r.
        // load_row fetches the row's statistics (L3, c3, R) ahead.
        auto load_row = [&](const TileIt& T) -> RowStats {
            RowStats rs{0.f, 0.f, INFINITY};
            if constexpr (!CALL1) {
                const int64_t row = (int64_t)T.tile * kRows + r;
                if (T.valid() && row < prm.N) {
                    rs.nL = prm.Lrow[(int64_t)T.bh * prm.N + row];
                    rs.nc = prm.crow[(int64_t)T.bh * prm.N + row];
                    rs.u = prm.Rb[T.bh];
                }
            }
            return rs;
        };
        auto prep = [&](RowStats rs) -> RowStats {
            const uint32_t ab = nprep & 1u;
            if constexpr (!CALL1) {
                rs.u = exp2f(rs.nL - rs.u);  // 0 in a row beyond N
                rs.nL = -rs.nL;
                rs.nc = -rs.nc;
                if (!wait(afull0 + 8u * ab, nprep >> 1)) ok = false;
                if (ok && w < D / 8) {
                    const int sw = ((r * D * 2) >> 7) & (D / 8 - 1);
                    uint4* p = reinterpret_cast<uint4*>(abuf + ab * C::kABytes + C::kATile +
                                                        r * D * 2) + (w ^ sw);
                    uint4 v = *p, lo;
                    uint32_t* x = reinterpret_cast<uint32_t*>(&v);
                    uint32_t* y = reinterpret_cast<uint32_t*>(&lo);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f =
                            __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&x[e]));
                        const float a = f.x * rs.u, b = f.y * rs.u;
                        x[e] = pack_bf16(a, b);
                        const float2 g =
                            __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&x[e]));
                        y[e] = pack_bf16(a - g.x, b - g.y);
                    }
                    *p = v;
                    p[2 * C::kATile / 16] = lo;
                    fence_proxy_async();
                }
                if (ok) mbar_arrive(aready0 + 8u * ab);
            }
            ++nprep;
            return rs;
        };
        // The tile whose dK and dV are owed: they leave during the next tile, once its first item
        // is handed over.
        bool owed = false;
        int o_bh = 0, o_tile = 0;
        constexpr int HD = D / 2;  // warpgroup w writes half h of the channels of dK (s 0) or dV
        uint32_t n_epi = 0;
        auto read_acc = [&](uint32_t* a) -> bool {
            const uint32_t par = n_epi & 1u;
            if (!wait(accdone0 + 8u * par, n_epi >> 1)) return false;
            ++n_epi;
            tc_fence_after();
            const uint32_t col = lane_t + C::kColAcc + par * 2 * D + s * D + h * HD;
            if constexpr (HD == 16) {
                tmem_ld16(col, a);
                tmem_wait_ld16(a);
            } else {
                tmem_ld8(col, a);
                tmem_wait_ld8(a);
            }
            tc_fence_before();
            mbar_arrive(accfree0 + 8u * par);
            return true;
        };
        auto write_acc = [&](const uint32_t* a) {
            const int64_t row = (int64_t)o_tile * kRows + r;
            if (row < prm.N) {
                const float sc = s == 0 ? prm.scale : 1.f;
                uint4* dst = reinterpret_cast<uint4*>((s == 0 ? prm.out0 : prm.out1) +
                                                      ((int64_t)o_bh * prm.N + row) * D + h * HD);
#pragma unroll
                for (int k = 0; k < HD / 8; ++k) {
                    const auto f = [&](int e) { return __uint_as_float(a[8 * k + e]) * sc; };
                    uint4 v;
                    v.x = pack_bf16(f(0), f(1));
                    v.y = pack_bf16(f(2), f(3));
                    v.z = pack_bf16(f(4), f(5));
                    v.w = pack_bf16(f(6), f(7));
                    dst[k] = v;
                }
            }
        };
        TileIt T(prm);
        RowStats next{};
        if (T.valid()) next = prep(load_row(T));
        // the next tile is prepared during this one, after its last block but one
        const int prep_at = prm.n_blocks > 1 ? prm.n_blocks - 2 : 0;
        int prev_bh = -1;
        const float* st0 = stats;
        while (T.valid() && ok) {
            if (T.bh != prev_bh) {
                prev_bh = T.bh;
                if (!wait(statfull0 + 8u * (seg & 1u), seg >> 1)) break;
                st0 = stats + (seg & 1u) * 2 * C::kMaxM;
            }
            const RowStats rs = next;
            const uint64_t nL2 = pack_f32x2(rs.nL, rs.nL), nc2 = pack_f32x2(rs.nc, rs.nc);
            const uint64_t u2 = pack_f32x2(rs.u, rs.u);
            const bool valid_row = (int64_t)T.tile * kRows + r < prm.N;
            const int bh = T.bh, tile = T.tile;
            const bool seg_end = T.last_of_segment();
            T.next();  // the next tile from here on
            RowStats ahead = load_row(T);
            auto prep_next = [&](int b) {
                if (b == prep_at && T.valid()) next = prep(ahead);
            };
            for (int b = 0; b < prm.n_blocks; ++b, ++bg) {
                const int item = 2 * b + s;
                if (item >= prm.n_items) {  // no item in this block
                    prep_next(b);
                    if (!ok) break;
                    continue;
                }
                // The issuer commits this item's S after the dK and dQ products of two blocks
                // before, so S being ready also says that this dS buffer is free.
                const uint32_t buf = bg & 1u;
                if (!wait(sready0 + 8u * s, is)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                uint32_t sa[16], ta[16];
                tmem_ld16(colS, sa);
                tmem_ld16(colT, ta);
                tmem_wait_ld16(sa);
                tmem_wait_ld16(ta);
                const int m0 = item * kItem + 32 * h;
                const int nv = (int)prm.M - m0;  // valid columns from this warpgroup's first on
                const float* c0 = st0 + m0;
                const float* c1 = c0 + C::kMaxM;
                uint8_t* dst = ds_row + buf * 2 * C::kDsTile;
                auto put = [&](int half, uint32_t* pp, uint32_t* ds) {
                    if (!valid_row) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) ds[e] = 0u;
                    }
                    tmem_st8(colT + 8 * half, pp);
#pragma unroll
                    for (int g = 0; g < 2; ++g)
                        *reinterpret_cast<uint4*>(dst + (((4 * h + 2 * half + g) ^ (r & 7)) << 4)) =
                            make_uint4(ds[4 * g], ds[4 * g + 1], ds[4 * g + 2], ds[4 * g + 3]);
                };
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t pp[8], ds[8];
                    if (nv >= 32)
                        slice_math<CALL1, true>(sa, ta, pp, ds, 16, c2, nL2, nc2, u2,
                                                c0 + 16 * half, c1 + 16 * half);
                    else
                        slice_math<CALL1, false>(sa, ta, pp, ds, nv - 16 * half, c2, nL2, nc2, u2,
                                                 c0 + 16 * half, c1 + 16 * half);
                    if (half == 0) {
                        tmem_ld16(colS + 16, sa);
                        tmem_ld16(colT + 16, ta);
                    }
                    put(half, pp, ds);
                    if (half == 0) {
                        tmem_wait_ld16(sa);
                        tmem_wait_ld16(ta);
                    }
                }
                tmem_wait_st();
                fence_proxy_async();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(pready0 + 8u * s);
                if (owed) {
                    uint32_t acc[HD];
                    if (!read_acc(acc)) {
                        ok = false;
                        break;
                    }
                    write_acc(acc);
                    owed = false;
                }
                ++is;
                prep_next(b);
                if (!ok) break;
            }
            if (!ok) break;
            if (owed) {  // a stream with no item: the tile before
                uint32_t acc[HD];
                if (!read_acc(acc)) break;
                write_acc(acc);
            }
            owed = true;
            o_bh = bh;
            o_tile = tile;
            if (seg_end) {
                // the segment's dQ: warpgroup w takes the route blocks w, w + 4, ...
                if (!wait(dqdone, seg)) break;
                tc_fence_after();
                const int64_t slot =
                    (int64_t)blockIdx.x - first_cta((int64_t)o_bh * prm.nt, prm.tiles, gridDim.x);
                for (int b = w; b < prm.n_blocks; b += 4) {
                    uint32_t t[D];
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        tmem_ld16(lane_t + C::kColQ + b * D + 16 * k, t + 16 * k);
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) tmem_wait_ld16(t + 16 * k);
                    const int64_t route = b * 128 + r;
                    if (route < prm.M) {
                        float4* dst = reinterpret_cast<float4*>(
                            prm.part + (((int64_t)o_bh * prm.slots + slot) * prm.M + route) * D);
#pragma unroll
                        for (int k = 0; k < D / 4; ++k)
                            dst[k] = make_float4(
                                __uint_as_float(t[4 * k]), __uint_as_float(t[4 * k + 1]),
                                __uint_as_float(t[4 * k + 2]), __uint_as_float(t[4 * k + 3]));
                    }
                }
                tc_fence_before();
                mbar_arrive(segfree0 + 8u * (seg & 1u));
                ++seg;
            }
        }
        if (ok && owed) {
            uint32_t acc[HD];
            if (read_acc(acc)) write_acc(acc);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 2) tmem_dealloc(tmem, kTmemCols);
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

// A bf16 [z][rows][D] tensor, boxes of box_rows x D, swizzled to the row width.
bool make_map(CUtensorMap* m, const void* base, int64_t D, int64_t rows, int64_t z,
              uint32_t box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)z};
    cuuint64_t strides[2] = {(cuuint64_t)(D * 2), (cuuint64_t)(rows * D * 2)};
    cuuint32_t box[3] = {(cuuint32_t)D, box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              D == 16 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

template <int D, bool CALL1, bool LO>
cudaError_t launch(const Plan& p, const TokOperands& o, const TokParams& prm, int64_t ctas,
                   cudaStream_t st) {
    using Cf = TokCfg<D, CALL1, LO>;
    const cudaError_t attr = ensure_smem_limit((const void*)tc_tok_kernel<D, CALL1, LO>, Cf::kSmem);
    if (attr != cudaSuccess) return attr;
    CUtensorMap a[3], it[3], lo;
    for (int k = 0; k < 3; ++k) {
        const bool used = k < Cf::kNT;
        if (!make_map(&a[k], o.a[used ? k : 0], D, p.N, p.BH, kRows) ||
            !make_map(&it[k], o.i[used ? k : 0], D, p.M,
                      CALL1 && (k == 0 || !used) ? p.H : p.BH, kItem))
            return cudaErrorInvalidValue;
    }
    lo = it[0];
    if (LO && !make_map(&lo, o.lo, D, p.M, p.BH, kItem)) return cudaErrorInvalidValue;
    return launch_pdl(tc_tok_kernel<D, CALL1, LO>, dim3((unsigned)ctas), dim3(kThreads), Cf::kSmem,
                      st, a[0], a[1], a[2], it[0], it[1], it[2], lo, prm);
}

}  // namespace

cudaError_t tc_tok_pass(const Plan& p, const BwdPlan& bp, bool call1, const TokOperands& o,
                        float scale, int* status, cudaStream_t st) {
    TokParams prm{};
    prm.H = p.H;
    prm.N = p.N;
    prm.M = p.M;
    prm.nt = bp.tok_nt;
    prm.tiles = bp.tok_nt * p.BH;
    prm.slots = bp.tok_slots;
    prm.n_items = (int)cdiv(p.M, kItem);
    prm.n_blocks = (int)cdiv(p.M, 2 * kItem);
    prm.i0_per_head = call1 ? 1 : 0;
    prm.c = scale * 1.4426950408889634f;
    prm.scale = scale;
    prm.Lrow = o.Lrow;
    prm.crow = o.crow;
    prm.Lcol = o.Lcol;
    prm.ccol = o.ccol;
    prm.Rb = o.Rb;
    prm.flags = o.flags;
    prm.part = o.part;
    prm.out0 = (__nv_bfloat16*)o.out0;
    prm.out1 = (__nv_bfloat16*)o.out1;
    prm.status = status;
    test_fault_for(4 + (call1 ? 4 : 5), &prm.wait_ns, &prm.withhold_it);
    const int64_t ctas = bp.tok_ctas;
    switch (p.D) {
        case 16:
            return call1 ? launch<16, true, false>(p, o, prm, ctas, st)
                         : launch<16, false, true>(p, o, prm, ctas, st);
        case 32:
            return call1 ? launch<32, true, false>(p, o, prm, ctas, st)
                         : launch<32, false, true>(p, o, prm, ctas, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace flarepp

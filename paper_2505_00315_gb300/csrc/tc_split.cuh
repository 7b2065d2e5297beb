// Grouped matrix product on the tensor cores (tcgen05.mma kind::f16, bf16
// planes, fp32 accumulation) for the shapes the TMA kernels do not serve: fp32
// storage, and bf16 storage with a head size other than 64.
//
// Every operand element is a sum of bf16 "planes": one for a bf16 input, two
// for a stored bf16 hi/lo pair, three for an fp32 value: p0 = bf16(v), p1 = bf16(v - p0),
// p2 = v - p0 - p1, each rounded to nearest, an exact cut (with v in [2^e, 2^(e+1)), p1 is at
// most 2^(e-8), and p2 at most 2^(e-17) in steps of 2^(e-23)).  The product of
// two operands is the sum of the plane products that matter: 1 (bf16 x bf16),
// 2 (pair x bf16) or, for fp32 x fp32, the six of order up to 2^-17 (p0 q0,
// p0 q1, p1 q0, p1 q1, p0 q2, p2 q0); what is left out is at most 2^-24 of each
// product and of either sign, under the rounding of an fp32 multiply-add chain.  (Parts
// cut off by truncation all have v's sign: they left out up to 2^-21, always
// towards zero, and results were up to four times as far off as a chain's.)  Each plane product
// of a K step is one MMA into the same accumulator, and the accumulator is
// drained into fp32 registers after every 64-wide K block, so that the tensor
// pipe's accumulation rounding acts on short partial sums only.
//
// Non-finite results are those of plain products (see store_non_finite).
//
// One CTA (544 threads) per SM walks over 128 x bn tiles (bn <= 128) of all groups:
//   warps 0-7    drain: TMEM -> registers (four accumulators in turn), then the
//                fused output step; warp w reads TMEM lanes 32 (w % 4) .. +31
//                and columns 64 (w / 4) .. +63
//   warps 8-15   producers: gathered or plain rows, by 16-byte cp.async
//                (bf16 planes already in memory) or through registers, one K
//                block ahead (fp32, cut into planes), into the 128-byte-
//                swizzled layout; row indices one block further ahead
//   warp 16      TMEM allocation and the MMA issuer (one thread)
// Each role runs on into the next tile, so a tile's output step runs beside the next
// one's loads and MMAs: with one tile to a CTA, products of few K blocks were bound
// by the chain of a tile's index loads, first loads and output step.  Measured alone,
// bf16 at B4 T1024 d1024 H16 h'=128 k128: output product 30 -> 21 us, dX 52 -> 37, dW
// 53 -> 38; fp32 at B4 T1000 d768 H12 k125: 20 -> 14, 33 -> 24 (dW 30 -> 31).
// What bounds it: bf16, the copies into shared memory; fp32, the producers (without
// their loads the projection took 21 of 29 us, without five of the six MMAs 28):
// cutting a K block's 16384 values into planes and storing them.  Neither a unit nor the
// issue slots are full: fp32 projection at B4 T1000 d768 H12 k125, 12 K blocks a CTA in
// 33 us under ncu, issue slots 41% used, ALU 30%, shared memory 22%, tensor pipe 13%; bf16
// h'=128 projection 45%, 30%, 13% and 8%.  A K block takes 2.4 us (fp32), where the multiply-adds
// of the CUDA-core product it replaces needed 8192 cycles (4 us) at the FFMA
// rate and ran at a tenth of that.
#pragma once

#include <cfloat>

#include "launch.h"
#include "profile.h"
#include "simt_gemm.cuh"
#include "tc_common.cuh"

namespace mosa {

// Contract of an Op (besides simt_gemm.cuh's M, N, K, a, b, store):
//   TA, TB                element types in memory (float or bf16)
//   kPA, kPB              planes of the operands (float: 3; bf16: 1 or 2)
//   kAMN / kBMN           the operand is contiguous along M / N in memory (else along K)
//   kTrans                outputs go out one column at a time with the lanes along M
//   A, lda, a_lo          base, row stride and offset of the second plane (elements)
//   a_row(g, r)           source row of A for strided index r (r < M or r < K)
//   b_ptr(g, r, c)        eight contiguous elements of B: strided index r (k if kBMN,
//                         else n), contiguous index c; linear in r with stride ldb; b_lo as a_lo
//   store(g, m, n, v, sp)      one result of reduction split sp (-1: the only one)
//   store4(g, m, n, v4, sp)    four consecutive columns (not kTrans)
struct SplitArgs {
    int bn;        // tile width, a multiple of 16, <= 128
    int nt, mt;    // column and row tiles of a group
    int tiles;     // all tiles: nt x mt x splits x groups
    int nkb;       // 64-wide K blocks in the whole reduction
    int splits;    // reduction splits
    int per;       // K blocks of a split
    uint32_t *status;
    unsigned long long *span;
};

constexpr int kSplitThreads = 544;
constexpr int kSplitPlane = 16384;   // one 128 x 64 bf16 plane tile
constexpr int kSplitOut = 8 * 4096;  // output staging, 4 KB per drain warp

template <class Op>
constexpr bool split_f32() { return sizeof(typename Op::TA) == 4; }
template <class Op>
constexpr int split_stages() { return split_f32<Op>() ? 2 : (Op::kPA + Op::kPB == 2 ? 6 : 4); }
// Accumulators (128 TMEM columns each), one K block (four 16-wide steps) in each: the
// tensor pipe does not round its accumulation to nearest, and with sixteen steps between
// drains bf16 errors against 64 bits were up to 4% (d = 1024) above those of the
// multiply-add chains that these products replace.  With four they are at or below them at
// every size measured (fp32 by 15 to 55%; with two steps by 17 to 58%, for 2% of the fp32
// step at B4 T1000 d768 H12 k125: 208 against 212.6 us).
constexpr int kSplitAcc = 4;
template <class Op>
constexpr int split_smem() {
    return 1024 + split_stages<Op>() * (Op::kPA + Op::kPB) * kSplitPlane + kSplitOut + 256;
}

// Two fp32 values rounded to bf16, x in the low half; beyond the bf16 range, infinities
// included, the largest bf16 value of that sign (NaN stays NaN).
__device__ __forceinline__ uint32_t bf16x2_sat(float x, float y) {
    uint32_t r;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
    return r;
}

// Eight fp32 values as three planes of eight bf16 (16 bytes each).
__device__ __forceinline__ void split3(const float4 &x, const float4 &y, uint4 (&pl)[3]) {
    const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    uint32_t w[3][4];
    auto lo = [](uint32_t u) { return __uint_as_float(u << 16); };
    auto hi = [](uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); };
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float a = v[2 * e], b = v[2 * e + 1];
        w[0][e] = bf16x2_sat(a, b);
        const float ra = a - lo(w[0][e]), rb = b - hi(w[0][e]);
        w[1][e] = bf16x2_sat(ra, rb);
        // what is left has at most eight bits: the upper half of its fp32 form
        w[2][e] = __byte_perm(__float_as_uint(ra - lo(w[1][e])), __float_as_uint(rb - hi(w[1][e])),
                              0x7632);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) pl[i] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// Tile t: column tiles fastest (neighbouring CTAs read the same rows of A).
struct SplitTile {
    int g, m0, n0, kb0, nkb, sp;   // sp: reduction split, -1 where there is only one
    __device__ __forceinline__ SplitTile(const SplitArgs &sa, unsigned t) {
        unsigned n = 0, m = 0;   // (a division by 1 is not worth its instructions)
        if (sa.nt > 1) n = t % (unsigned)sa.nt, t /= (unsigned)sa.nt;
        if (sa.mt > 1) m = t % (unsigned)sa.mt, t /= (unsigned)sa.mt;
        kb0 = 0;
        nkb = sa.nkb;
        sp = -1;
        if (sa.splits > 1) {
            sp = (int)(t % (unsigned)sa.splits), t /= (unsigned)sa.splits;
            kb0 = sp * sa.per;
            nkb = min(sa.nkb, kb0 + sa.per) - kb0;
        }
        g = (int)t;
        n0 = (int)n * sa.bn;
        m0 = (int)m * 128;
    }
};

// Non-finite results of a warp's 32 rows x 64 columns.  Where an operand is not finite they
// are right: an infinity is cut into (largest, largest, infinity), p2 meets q0 only, and
// that product comes first, so that it decides the sign (or NaN, times 0).  Where
// both operands are finite and their product passes the fp32 range 2^8 times over, p1 q0 or p0 q1
// does so before p0 q0, with either sign: such elements (non-finite, no non-finite
// operand) are computed again by plain multiply-adds.  Rows and columns that are NaN throughout
// come from a NaN operand and need no look at the operands.
// The issuer waits meanwhile, with a limit: at most kPlainSteps steps (about 0.2 s) a tile.
// (All results of a warp with a NaN again, each by a chain over all of K: a step of B4 T2048
// d768 H12 k512 with one NaN in X took 44 ms instead of 0.7, and takes 1.0 now.)
constexpr int kPlainSteps = 1 << 22;   // 64 columns of 65536 rows
// Puts v's columns nb .. nb + w - 1 of row m right and stores them (w and the number of rows
// are the same in all lanes).  Out of line, and on a copy of the results, so that the
// output step around it keeps them in registers.
template <class Op>
__device__ __noinline__ void store_non_finite(const Op &op, int g, int sp, int m, int rows, int nb,
                                              int w, int k0, int k1, float *v) {
    constexpr uint32_t kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (rows <= 0) return;
    const bool mine = lane < rows;
    uint32_t todo[2] = {0u, 0u}, nan[2] = {0u, 0u};
    for (int j = 0; j < w; ++j) {
        const float x = mine ? v[j] : 0.f;
        const bool is_nan = x != x;
        const bool column = __popc(__ballot_sync(kAll, is_nan)) == rows;
        if (is_nan) nan[j >> 5] |= 1u << (j & 31);
        if (!column && !(fabsf(x) <= FLT_MAX)) todo[j >> 5] |= 1u << (j & 31);
    }
    if (__popc(nan[0]) + __popc(nan[1]) == w) todo[0] = todo[1] = 0u;
    int steps = kPlainSteps - 3 * min(k1 - k0, kPlainSteps);
    if (steps < 0) todo[0] = todo[1] = 0u;
    constexpr int U = 8;   // steps whose loads are in flight at a time (past the end, the last again)
    const int row = mine ? m : m - lane;
    if (__any_sync(kAll, (todo[0] | todo[1]) != 0u)) {
        const int c0 = nb + min(lane, w - 1), c1 = nb + min(lane + 32, w - 1);
        float za = 0.f, z0 = 0.f, z1 = 0.f;   // 0 times a non-finite value is NaN
        for (int k = k0; k < k1; k += U) {
            float a[U], b0[U], b1[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int kk = min(k + i, k1 - 1);
                a[i] = op.a(g, row, kk);
                b0[i] = op.b(g, kk, c0);
                b1[i] = op.b(g, kk, c1);
            }
#pragma unroll
            for (int i = 0; i < U; ++i) {
                za = fmaf(a[i], 0.f, za);
                z0 = fmaf(b0[i], 0.f, z0);
                z1 = fmaf(b1[i], 0.f, z1);
            }
        }
        const uint32_t bad0 = __ballot_sync(kAll, z0 != 0.f), bad1 = __ballot_sync(kAll, z1 != 0.f);
        todo[0] = za != 0.f ? 0u : todo[0] & ~bad0;
        todo[1] = za != 0.f ? 0u : todo[1] & ~bad1;
    }
    for (int j = 0; j < w; ++j) {
        float x = v[j];
        const bool on = todo[j >> 5] >> (j & 31) & 1u;
        if (__any_sync(kAll, on) && (steps -= k1 - k0) >= 0) {
            float acc = 0.f;
            for (int k = k0; k < k1; k += U) {
                float a[U], b[U];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const int kk = min(k + i, k1 - 1);
                    a[i] = op.a(g, row, kk);
                    b[i] = k + i < k1 ? op.b(g, kk, nb + j) : 0.f;   // (a is finite)
                }
#pragma unroll
                for (int i = 0; i < U; ++i) acc = fmaf(a[i], b[i], acc);
            }
            if (on) x = acc;
        }
        if (mine) op.store(g, m, nb + j, x, sp);
    }
}

template <class Op>
__global__ void __launch_bounds__(kSplitThreads, 1)
    split_gemm_kernel(const __grid_constant__ Op op, const SplitArgs sa) {
    using namespace tc;
    using TA = typename Op::TA;
    using TB = typename Op::TB;
    constexpr bool kF32 = split_f32<Op>();
    constexpr int S = split_stages<Op>();
    constexpr int kStage = (Op::kPA + Op::kPB) * kSplitPlane;
    constexpr int NA = kSplitAcc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *outs = ring + S * kStage;
    uint64_t *bars = reinterpret_cast<uint64_t *>(outs + kSplitOut);
    uint64_t *full = bars, *empty = bars + 8, *accf = bars + 16, *acce = bars + 20,
             *mdone = bars + 24;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 25);
    int *s_abort = reinterpret_cast<int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int step = gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&full[s]), 256);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < kSplitAcc; ++b) {
            mbar_init(smem_u32(&accf[b]), 1);
            mbar_init(smem_u32(&acce[b]), 256);
        }
        mbar_init(smem_u32(mdone), 1);
        *s_abort = 0;
        fence_barrier_init();
    }
    if (warp == 16) {
        tmem_alloc(smem_u32(tmem_slot), 128 * kSplitAcc);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();  // everything below may read what the previous kernel wrote
    span_begin(sa.span);
    const uint32_t tmem = *tmem_slot;
    auto give_up = [&]() {
        atomicOr(sa.status, kStatusTimeout);
        *(volatile int *)s_abort = 1;
    };

    if (warp >= 8 && warp < 16) {
        // ------------------------------------------------------ producers
        const int t = threadIdx.x - 256;
        // chunk p of this thread: strided row and 16-byte unit of the tile
        const int arow = Op::kAMN ? t >> 4 : t >> 3, ach = Op::kAMN ? t & 15 : t & 7;
        const int brow = Op::kBMN ? t >> 4 : t >> 3, bch = Op::kBMN ? t & 15 : t & 7;
        constexpr int kAStep = Op::kAMN ? 16 : 32, kBStep = Op::kBMN ? 16 : 32;
        auto place = [](bool mn, int row, int ch) -> uint32_t {
            return (mn ? (uint32_t)(ch >> 3) * 8192u : 0u) + row * 128 + (((ch & 7) ^ (row & 7)) << 4);
        };
        // The K blocks of all tiles in order: (tl, it).
        struct Walk {
            SplitTile tl;
            int tile, it;
        };
        auto advance = [&](Walk &w) {
            if (++w.it < w.tl.nkb) return;
            w.tile += step;
            w.it = 0;
            if (w.tile < sa.tiles) w.tl = SplitTile(sa, w.tile);
        };
        // source rows of block w (-1: zeros), one per lane: a warp's chunks lie in
        // 2 (kAMN) or 4 rows of each step p, lane 2 p + i or 4 p + i holding row i's;
        // K-major rows are the same for all blocks of a tile
        constexpr int kPer = Op::kAMN ? 2 : 4;
        const int my_row = (warp - 8) * kPer + lane % kPer + kAStep * (lane / kPer);
        auto rows_of = [&](const Walk &w, int &idx) {
            if (w.tile >= sa.tiles || (!Op::kAMN && w.it > 0)) return;
            const int i = (Op::kAMN ? (w.tl.kb0 + w.it) * 64 : w.tl.m0) + my_row;
            idx = lane < 4 * kPer && i < (Op::kAMN ? op.K : op.M) ? op.a_row(w.tl.g, i) : -1;
        };
        auto row_at = [&](int idx, int p) {
            return __shfl_sync(0xffffffffu, idx, kPer * p + lane / (32 / kPer));
        };
        auto a_src = [&](const Walk &w, int r) -> const TA * {   // nullptr: zeros
            const int col = Op::kAMN ? w.tl.m0 + ach * 8 : (w.tl.kb0 + w.it) * 64 + ach * 8;
            if (r < 0 || col >= (Op::kAMN ? op.M : op.K)) return nullptr;
            return op.A + (size_t)r * op.lda + col;
        };
        // this thread's first B chunk of a block; the others are kBStep rows apart
        auto b_used = [&](int p) {   // inside the tile's bn columns
            return (Op::kBMN ? bch * 8 : brow + kBStep * p) < sa.bn;
        };
        auto b_first = [&](const Walk &w) -> const TB * {
            const int kk = (w.tl.kb0 + w.it) * 64 + (Op::kBMN ? brow : bch * 8);
            const int n = w.tl.n0 + (Op::kBMN ? bch * 8 : brow);
            if (n >= op.N || kk >= op.K) return nullptr;
            return Op::kBMN ? op.b_ptr(w.tl.g, kk, n) : op.b_ptr(w.tl.g, n, kk);
        };
        auto b_src = [&](const Walk &w, const TB *first, int p) -> const TB * {
            if (first == nullptr || !b_used(p)) return nullptr;
            if (Op::kBMN ? (w.tl.kb0 + w.it) * 64 + brow + kBStep * p >= op.K
                         : w.tl.n0 + brow + kBStep * p >= op.N)
                return nullptr;
            return first + (size_t)(kBStep * p) * op.ldb;
        };
        Walk w{SplitTile(sa, blockIdx.x), (int)blockIdx.x, 0};
        int idx = -1;
        rows_of(w, idx);
        if constexpr (kF32) {
            float4 av[4][2], bv[4][2];
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            auto load_a = [&](const Walk &x) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const TA *s = a_src(x, row_at(idx, p));
                    av[p][0] = s ? *reinterpret_cast<const float4 *>(s) : zero;
                    av[p][1] = s ? *reinterpret_cast<const float4 *>(s + 4) : zero;
                }
            };
            auto load_b = [&](const Walk &x) {
                const TB *first = b_first(x);
                const int n = x.tl.n0 + bch * 8;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const TB *s = b_src(x, first, p);
                    bv[p][0] = s ? *reinterpret_cast<const float4 *>(s) : zero;
                    bv[p][1] = s ? *reinterpret_cast<const float4 *>(s + 4) : zero;
                    if (Op::kBMN && n + 8 > op.N && s != nullptr) {   // past the last column
                        float e[8] = {bv[p][0].x, bv[p][0].y, bv[p][0].z, bv[p][0].w,
                                      bv[p][1].x, bv[p][1].y, bv[p][1].z, bv[p][1].w};
#pragma unroll
                        for (int j = 0; j < 8; ++j) e[j] = n + j < op.N ? e[j] : 0.f;
                        bv[p][0] = make_float4(e[0], e[1], e[2], e[3]);
                        bv[p][1] = make_float4(e[4], e[5], e[6], e[7]);
                    }
                }
            };
            // w runs one block ahead of the one in registers; idx holds its rows
            bool have = w.tile < sa.tiles;
            if (have) {
                load_a(w);
                load_b(w);
                advance(w);
                rows_of(w, idx);
            }
            for (int n = 0; have; ++n) {
                const int s = n % S;
                // (warp-uniform: the row shuffles are warp-collective)
                if (__any_sync(0xffffffffu, !mbar_wait(smem_u32(&empty[s]), ((n / S) & 1) ^ 1) ||
                                                *(volatile int *)s_abort)) {
                    give_up();
                    break;
                }
                have = w.tile < sa.tiles;
                uint8_t *sA = ring + s * kStage, *sB = sA + Op::kPA * kSplitPlane;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    uint4 pl[3];
                    split3(av[p][0], av[p][1], pl);
                    const uint32_t o = place(Op::kAMN, arow + kAStep * p, ach);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        *reinterpret_cast<uint4 *>(sA + i * kSplitPlane + o) = pl[i];
                }
                if (have) load_a(w);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    if (!b_used(p)) continue;
                    uint4 pl[3];
                    split3(bv[p][0], bv[p][1], pl);
                    const uint32_t o = place(Op::kBMN, brow + kBStep * p, bch);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        *reinterpret_cast<uint4 *>(sB + i * kSplitPlane + o) = pl[i];
                }
                if (have) load_b(w);
                fence_proxy_async();
                mbar_arrive(smem_u32(&full[s]));
                if (have) {
                    advance(w);
                    rows_of(w, idx);
                }
            }
        } else {
            constexpr int LAG = S - 2;
            int landed = 0, issued = 0;
            for (int n = 0; w.tile < sa.tiles; ++n) {
                const int s = n % S;
                // (warp-uniform: the row shuffles are warp-collective)
                if (__any_sync(0xffffffffu, !mbar_wait(smem_u32(&empty[s]), ((n / S) & 1) ^ 1) ||
                                                *(volatile int *)s_abort)) {
                    give_up();
                    break;
                }
                uint8_t *sA = ring + s * kStage, *sB = sA + Op::kPA * kSplitPlane;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const TA *src = a_src(w, row_at(idx, p));
                    const uint32_t dst = smem_u32(sA) + place(Op::kAMN, arow + kAStep * p, ach);
#pragma unroll
                    for (int i = 0; i < Op::kPA; ++i)
                        cp_async16(dst + i * kSplitPlane, src ? src + i * op.a_lo : op.A, src ? 16u : 0u);
                }
                const TB *first = b_first(w);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    if (!b_used(p)) continue;
                    const TB *src = b_src(w, first, p);
                    const uint32_t dst = smem_u32(sB) + place(Op::kBMN, brow + kBStep * p, bch);
#pragma unroll
                    for (int i = 0; i < Op::kPB; ++i)
                        cp_async16(dst + i * kSplitPlane,
                                   src ? src + i * op.b_lo : reinterpret_cast<const TB *>(op.A),
                                   src ? 16u : 0u);
                }
                cp_async_commit();
                issued = n + 1;
                advance(w);
                rows_of(w, idx);
                // a stage is confirmed LAG stages after its copies were issued
                if (n >= LAG) {
                    cp_async_wait<LAG>();
                    fence_proxy_async();
                    mbar_arrive(smem_u32(&full[(n - LAG) % S]));
                    ++landed;
                }
            }
            cp_async_wait<0>();
            fence_proxy_async();
            for (int n = landed; n < issued; ++n) mbar_arrive(smem_u32(&full[n % S]));
        }
    } else if (warp == 16) {
        // ----------------------------------------------------- MMA issuer
        if (elect_one()) {
            const uint32_t idesc = idesc_bf16(128, sa.bn, Op::kAMN, Op::kBMN);
            int n = 0;   // K blocks so far
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < sa.tiles; tile += step) {
                const SplitTile tl(sa, tile);
                for (int it = 0; it < tl.nkb; ++it, ++n) {
                    const int s = n % S;
                    ok = mbar_wait(smem_u32(&full[s]), (n / S) & 1) &&
                         mbar_wait(smem_u32(&acce[n % NA]), ((n / NA) & 1) ^ 1);
                    if (!ok || *(volatile int *)s_abort) {
                        give_up();
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = smem_u32(ring + s * kStage), b = a + Op::kPA * kSplitPlane;
                    const int left = op.K - (tl.kb0 + it) * 64;
                    const int steps = left >= 64 ? 4 : (left + 15) / 16;
                    uint32_t acc = 0u;
                    auto product = [&](int i, int j) {
#pragma unroll   // (left rolled, that fp32 step takes 211 us)
                        for (int st = 0; st < 4; ++st) {
                            if (st >= steps) break;
                            const uint32_t ai = a + i * kSplitPlane, bj = b + j * kSplitPlane;
                            const uint64_t ad = Op::kAMN ? smem_desc_sw128(ai + st * 2048, 8192, 1024)
                                                         : smem_desc_sw128(ai + st * 32, 16, 1024);
                            const uint64_t bd = Op::kBMN ? smem_desc_sw128(bj + st * 2048, 8192, 1024)
                                                         : smem_desc_sw128(bj + st * 32, 16, 1024);
                            mma_bf16(tmem + 128 * (n % NA), ad, bd, idesc, acc);
                            acc = 1u;
                        }
                    };
                    // small products first
                    if constexpr (kF32) {
                        product(2, 0);
                        product(0, 2);
                        product(1, 1);
                    }
                    if constexpr (Op::kPA > 1) product(1, 0);
                    if constexpr (Op::kPB > 1) product(0, 1);
                    product(0, 0);
                    mma_commit(smem_u32(&accf[n % NA]));
                    mma_commit(smem_u32(&empty[s]));
                }
            }
            drain_mmas(smem_u32(mdone));
        }
    } else {
        // ------------------------------------------- drain and output step
        const int q = warp & 3, hf = warp >> 2;
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + 64 * hf;
        uint8_t *xb = outs + warp * 4096;
        int c = 0;   // K blocks so far
        bool ok = true;
        for (int tile = blockIdx.x; ok && tile < sa.tiles; tile += step) {
            const SplitTile tl(sa, tile);
            float v[64];
#pragma unroll
            for (int j = 0; j < 64; ++j) v[j] = 0.f;
            for (int u = 0; u < tl.nkb; ++u, ++c) {
                ok = mbar_wait(smem_u32(&accf[c % NA]), (c / NA) & 1);
                // warp-uniform: the TMEM loads below are warp-collective
                if (__any_sync(0xffffffffu, !ok || *(volatile int *)s_abort)) {
                    give_up();
                    ok = false;
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 16) {
                    if (64 * hf + c0 >= sa.bn) continue;   // bn is a multiple of 16
                    float t[16];
                    tmem_ld16(tb + 128 * (c % NA) + c0, t);
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[c0 + j] += t[j];
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&acce[c % NA]));
            }
            if (!ok) break;
            // last tile drained: the next kernel may start its prologue
            if (tile + step >= sa.tiles) pdl_trigger();
            const int nb = tl.n0 + 64 * hf, n_end = min(op.N, tl.n0 + sa.bn);
            const int m = tl.m0 + q * 32 + lane;
            if constexpr (Op::kPA + Op::kPB > 2) {
                bool bad = false;
#pragma unroll
                for (int j = 0; j < 64; ++j) bad = bad || !(fabsf(v[j]) <= FLT_MAX);
                if (__any_sync(0xffffffffu, bad)) {
                    float x[64];
#pragma unroll
                    for (int j = 0; j < 64; ++j) x[j] = v[j];
                    store_non_finite(op, tl.g, tl.sp, m, min(32, op.M - (tl.m0 + q * 32)), nb,
                                     min(64, n_end - nb), tl.kb0 * 64,
                                     min(op.K, (tl.kb0 + tl.nkb) * 64), x);
                    continue;
                }
            }
            if constexpr (Op::kTrans) {
                if (m < op.M) {
#pragma unroll
                    for (int j = 0; j < 64; ++j)
                        if (nb + j < n_end) op.store(tl.g, m, nb + j, v[j], tl.sp);
                }
            } else {
                // through a 4 KB per-warp buffer, so that every store or reduction
                // instruction covers whole 128-byte row pieces
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    if (nb + c0 >= n_end) continue;
                    stage_f32x32(xb, v + c0, 1.f, lane);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rl = (lane >> 3) + 4 * i, mr = tl.m0 + q * 32 + rl;
                        const int n = nb + c0 + 4 * (lane & 7);
                        const float4 x = *reinterpret_cast<const float4 *>(xb + xoff128(rl, lane & 7));
                        if (mr < op.M && n < n_end) op.store4(tl.g, mr, n, x, tl.sp);
                    }
                    __syncwarp();
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    span_end(sa.span);
    if (warp == 16) {
        tc_fence_after();
        tmem_dealloc(tmem, 128 * kSplitAcc);
    }
}

// Launches op over `groups` groups in `splits` reduction splits, none of them empty.
template <class Op>
inline cudaError_t launch_split_gemm(const Op &op, int groups, int splits, uint32_t *status,
                                     cudaStream_t stream) {
    if (op.M <= 0 || op.N <= 0 || groups <= 0) return cudaSuccess;
    constexpr int smem = split_smem<Op>();
    cudaError_t e = allow_smem((const void *)split_gemm_kernel<Op>, smem);
    if (e != cudaSuccess) return e;
    SplitArgs sa;
    sa.nt = (op.N + 127) / 128;
    sa.mt = (op.M + 127) / 128;
    sa.bn = ((op.N + sa.nt - 1) / sa.nt + 15) / 16 * 16;
    sa.nkb = (op.K + 63) / 64;
    sa.splits = splits;
    sa.per = (sa.nkb + splits - 1) / splits;
    const long long tiles = (long long)sa.nt * sa.mt * groups * splits;
    if (tiles > 0x7fffffff - 152) return cudaErrorInvalidValue;
    sa.tiles = (int)tiles;
    sa.status = status;
    sa.span = active_span();
    const dim3 grid(sa.tiles < 152 ? sa.tiles : 152);   // one CTA per SM
    e = launch_pdl(split_gemm_kernel<Op>, grid, dim3(kSplitThreads), smem, stream, op, sa);
    note_launches(1);
    return e;
}

// Reduction splits of a product with M x N outputs in `groups` groups over K:
// enough tiles for the 152 SMs while each takes at least four K blocks, of which the last
// split may find fewer left; none is empty.
inline int split_count(int M, int N, int K, int groups) {
    const long long tiles = (long long)((M + 127) / 128) * ((N + 127) / 128) * groups;
    const int nkb = (K + 63) / 64;
    int sp = 1;
    while (tiles * sp * 2 <= 152 && nkb / (sp * 2) >= 4) sp *= 2;
    const int per = (nkb + sp - 1) / sp;
    return (nkb + per - 1) / per;
}

}  // namespace mosa
